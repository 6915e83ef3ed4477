"""The one-pass right-hand side of a time step and K_div alone against the
oracle's matrices: tile edges in 2D and 3D, a viscosity per element, operands
that are only 8-byte aligned, and a right-hand side written over the previous
stress.

Tolerance: fewer than 300 terms per entry, each rounded to 1.1e-16 of sums
bounded by |M/alpha| |w| + |K| |w| + |F|: 1e-13 of that bound's largest entry.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem
from paper_2606_13429_gb300 import dcg, inputs

pytestmark = pytest.mark.gpu

SCHEMES = [dcg.DCG_IMPLICIT_EULER, dcg.DCG_CRANK_NICOLSON, dcg.DCG_BDF2]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2606_13429_gb300 import build
    build.build()
    dcg.load()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("d,n", [(2, 2), (2, 33), (2, 130), (3, 2), (3, 5), (3, 31)])
@pytest.mark.parametrize("lognormal", [False, True])
@pytest.mark.parametrize("scheme", SCHEMES)
def test_rhs(d, n, lognormal, scheme):
    dt = 1e-3
    alpha = dcg.dcg_scheme_alpha(scheme, dt)
    nu = inputs.nu_elements(6, n ** d) if lognormal else None
    # K_div is what is left of A where the mass part is negligible: two steps
    # sizes separate the parts exactly enough (A_a - A_b = M (1/a - 1/b))
    Aa = fem.assemble(d, n, alpha, nu_elem=nu).matrix().tocsr()
    K = fem.assemble(d, n, 1e30, nu_elem=nu).matrix().tocsr()
    M = Aa - K
    prob = dcg.dcg_assemble(d, n, alpha, nu_elem=nu)
    N = prob.N
    s1, s2, f1, f0 = (inputs.rhs(20 + k, N) for k in range(4))
    w = 4.0 / 3.0 * s1 - 1.0 / 3.0 * s2 if scheme == dcg.DCG_BDF2 else s1
    want = M @ w + f1
    if scheme == dcg.DCG_CRANK_NICOLSON:
        want = want - K @ w + f0
    bound = (abs(M) @ np.abs(w) + abs(K) @ np.abs(w)).max() + 2.0
    for shift in (0, 1):
        def put(a):
            t = torch.empty(N + 1, dtype=torch.float64, device="cuda")[shift:shift + N]
            return t.copy_(torch.from_numpy(a))
        t1, t2, g1, g0 = put(s1), put(s2), put(f1), put(f0)
        out = put(np.zeros(N))
        kw = dict(s2=t2 if scheme == dcg.DCG_BDF2 else None, F0=g0 if scheme == dcg.DCG_CRANK_NICOLSON else None)
        dcg.dcg_time_rhs(prob, scheme, t1, g1, out, **kw)
        torch.cuda.synchronize()
        assert np.abs(out.cpu().numpy() - want).max() <= 1e-13 * bound
        y = put(np.zeros(N))
        dcg.dcg_apply_div(prob, t1, y)
        torch.cuda.synchronize()
        assert np.abs(y.cpu().numpy() - K @ s1).max() <= 1e-13 * (abs(K) @ np.abs(s1)).max()
        dcg.dcg_time_rhs(prob, scheme, t1, g1, t1, **kw)  # over the previous stress
        torch.cuda.synchronize()
        assert torch.equal(t1, out)
