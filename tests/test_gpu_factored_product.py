"""The factored FP64 product against the oracle's assembled matrix: grids at
the edges of its tiles (128 columns in 2D, 30 columns and 4 rows in 3D), the
shortest ones, uniform and per-element viscosity, pointers that are only
8-byte aligned, and the product of a multiple of V (its mass part vanishes).

Tolerance: an entry adds fewer than 300 terms, each rounded to 1.1e-16 of
sums bounded by |A| |x|, so 1e-13 of the largest entry of |A| |x| holds.
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


@pytest.mark.parametrize("d,n", [(2, 2), (2, 3), (2, 18), (2, 129), (2, 130), (2, 161), (3, 2), (3, 3), (3, 6), (3, 31),
                                 (3, 32)])
@pytest.mark.parametrize("lognormal", [False, True])
@pytest.mark.parametrize("dt", [1e-6, 1e-1])
def test_product(d, n, lognormal, dt):
    nu = inputs.nu_elements(5, n ** d) if lognormal else None
    A = fem.assemble(d, n, dt, nu=0.7, nu_elem=nu).matrix().tocsr()
    prob = dcg.dcg_assemble(d, n, dt, nu=0.7, nu_elem=nu)
    x = inputs.rhs(3, prob.N)
    buf = torch.zeros(2 * prob.N + 4, dtype=torch.float64, device="cuda")
    bound = (abs(A) @ np.abs(x)).max()
    for shift in (0, 1):  # the second round: 8-byte aligned only
        xt, yt = buf[shift:shift + prob.N], buf[prob.N + 2 + shift:2 * prob.N + 2 + shift]
        xt.copy_(torch.from_numpy(x))
        dcg.dcg_spmv(prob, xt, yt)
        torch.cuda.synchronize()
        assert np.abs(yt.cpu().numpy() - A @ x).max() <= 1e-13 * bound
    # V z: the factored product's mass part is exactly zero, so the product is
    # that of K_div. (Small aligned 2D and small 3D operands take the stored
    # blocks, which cancel the mass part to rounding only.)
    if d == 3 and prob.n_nodes <= 8000:
        return
    q = torch.from_numpy(inputs.rhs(4, prob.n_nodes)).cuda()
    v = torch.empty(prob.N + 1, dtype=torch.float64, device="cuda")[1:]
    y, k = (torch.empty(prob.N, dtype=torch.float64, device="cuda") for _ in range(2))
    dcg.dcg_embed(prob, q, v)
    dcg.dcg_spmv(prob, v, y)
    dcg.dcg_apply_div(prob, v, k)
    torch.cuda.synchronize()
    assert (y - k).abs().max().item() <= 1e-13 * max(k.abs().max().item(), 1e-300)
