"""The factored product on grids past the line below which the stored blocks
serve (40,000 nodes in 2D, 8,000 in 3D): y = A x on operands of both
alignments with a remainder in every tile (warps of 32 columns and seg rows in
2D, 30 columns and 4 rows in 3D), and the fused forms through solves: plain CG
(f - A x, A d with d.q), deflated CG (A d with V^T, f - A V z, V^T A x) and the
matrix-free A (d - V z). The right-hand side of a time step may be written over
either load or the older stress.

Tolerances: an entry adds fewer than 300 terms, each rounded to 1.1e-16 of sums
bounded by |A| |x|: 1e-13 of the largest entry of |A| |x|. The residual norm a
solve reports and the one formed with the oracle's matrix differ by that
rounding of |A| |x| + |f|, in the 2-norm.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem
from paper_2606_13429_gb300 import dcg, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2606_13429_gb300 import build
    build.build()
    dcg.load()
    torch.cuda.set_device(0)


def _nu(lognormal, d, n):
    return inputs.nu_elements(7, n ** d) if lognormal else None


@pytest.mark.parametrize("d,n", [(2, 202), (2, 203), (2, 226), (3, 22), (3, 24)])
@pytest.mark.parametrize("lognormal", [False, True])
def test_product(d, n, lognormal):
    nu = _nu(lognormal, d, n)
    A = fem.assemble(d, n, 1e-5, nu_elem=nu).matrix().tocsr()
    prob = dcg.dcg_assemble(d, n, 1e-5, nu_elem=nu)
    assert prob.n_nodes > (40000 if d == 2 else 8000)
    x = inputs.rhs(61, prob.N)
    bound = (abs(A) @ np.abs(x)).max()
    buf = torch.zeros(2 * prob.N + 4, dtype=torch.float64, device="cuda")
    for shift in (0, 1):
        xt, yt = buf[shift:shift + prob.N], buf[prob.N + 2 + shift:2 * prob.N + 2 + shift]
        assert xt.data_ptr() % 16 == 8 * shift
        xt.copy_(torch.from_numpy(x))
        dcg.dcg_spmv(prob, xt, yt)
        assert np.abs(yt.cpu().numpy() - A @ x).max() <= 1e-13 * bound


@pytest.mark.parametrize("d,n,matrix_free", [(2, 204, False), (3, 22, False), (3, 22, True)])
@pytest.mark.parametrize("lognormal", [False, True])
@pytest.mark.parametrize("deflate,device_loop", [(0, 0), (1, 0), (1, 1)])
def test_fused_forms(d, n, matrix_free, lognormal, deflate, device_loop):
    nu, dt = _nu(lognormal, d, n), 1e-6
    A = fem.assemble(d, n, dt, nu_elem=nu).matrix().tocsr()
    prob = dcg.dcg_assemble(d, n, dt, nu_elem=nu, matrix_free=matrix_free)
    dcg.dcg_setup(prob, dcg.options(max_levels=2, deflate=deflate, device_loop=device_loop))
    f = inputs.rhs(62, prob.N)
    x = torch.zeros(prob.N, dtype=torch.float64, device="cuda")
    # the residual of an early stop is far above rounding, that of a converged solve at the tolerance
    for max_it in (3, 5000):
        st = dcg.dcg_solve(prob, torch.from_numpy(f).cuda(), x.zero_(), tol=1e-8, max_it=max_it)
        xh = x.cpu().numpy()
        rel = np.linalg.norm(f - A @ xh) / np.linalg.norm(f)
        bound = np.linalg.norm(abs(A) @ np.abs(xh) + np.abs(f)) / np.linalg.norm(f)
        assert abs(st["true_relres"] - rel) <= 1e-13 * bound
        if max_it > 3 and deflate:
            assert st["status"] == dcg.DCG_OK and rel <= 1.01e-8


@pytest.mark.parametrize("d,n", [(2, 203), (2, 30), (3, 23)])
@pytest.mark.parametrize("scheme", [dcg.DCG_IMPLICIT_EULER, dcg.DCG_CRANK_NICOLSON, dcg.DCG_BDF2])
def test_time_rhs_over_an_operand(d, n, scheme):
    prob = dcg.dcg_assemble(d, n, dcg.dcg_scheme_alpha(scheme, 1e-3), nu_elem=_nu(True, d, n))
    v = [torch.from_numpy(inputs.rhs(63 + k, prob.N)).cuda() for k in range(4)]

    def run(over):
        s1, s2, f1, f0 = [t.clone() for t in v]
        out = {"f1": f1, "f0": f0, "s1": s1, "s2": s2}.get(over, torch.zeros_like(s1))
        dcg.dcg_time_rhs(prob, scheme, s1, f1, out, s2=s2 if scheme == dcg.DCG_BDF2 else None,
                         F0=f0 if scheme == dcg.DCG_CRANK_NICOLSON else None)
        return out

    want = run(None)
    for over in ["f1", "s1"] + (["f0"] if scheme == dcg.DCG_CRANK_NICOLSON else []) + \
            (["s2"] if scheme == dcg.DCG_BDF2 else []):
        assert torch.equal(run(over), want), over
