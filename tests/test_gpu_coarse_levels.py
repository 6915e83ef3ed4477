"""Dense coarsest solves on few tiles and the residual forms of the Q1
Laplacian, at the edges of their tiles: panels of 16 x 32 outputs, line sweeps
in batches of 8 rows, row walks of 2 and 8, 3D walks over pairs of rows and 2
or 8 planes.

Tolerances: a coarsest solve is a chain of three stable transforms in FP64
(1e-11 of the largest entry, as for the other coarse solves). A W-cycle
amplifies rounding by less than 10^3 (1e-10). The norm that stops Algorithm 3
comes from the residual kernel: the norm formed by the oracle's matrix agrees
to the rounding of Z z against g, below 1e-10 ||g||.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, mg
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


# coarsest extents m: 2D 9, 16 (one tile), 17, 33, 48, 49, 389 (the last panel) and 399 (tiles); 3D 5, 9, 13
@pytest.mark.parametrize("d,n,levels", [(2, 20, 2), (2, 34, 2), (2, 36, 2), (2, 68, 2), (2, 98, 2), (2, 100, 2),
                                        (2, 780, 2), (2, 800, 2), (3, 12, 2), (3, 20, 2), (3, 28, 2)])
@pytest.mark.parametrize("precision", [dcg.DCG_FP64, dcg.DCG_MIXED])
def test_dense_coarse_solve(d, n, levels, precision):
    prob = dcg.dcg_assemble(d, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(max_levels=levels, precision=precision))
    m = n // 2 - 1
    j = np.arange(1, m + 1)
    # smooth and rough sine modes: eigenvectors of the coarsest matrix
    h, f, want = 2.0 / n, 0.0, 0.0
    for k in (1, 2, m // 2 + 1, m):
        s = np.sin(np.pi * k * j / (m + 1))
        kap, mu = (2 - 2 * np.cos(np.pi * k * h)) / h, h * (4 + 2 * np.cos(np.pi * k * h)) / 6
        v = s
        for _ in range(d - 1):
            v = np.multiply.outer(s, v)
        lam = kap * mu ** (d - 1)  # (1/d) sum over d equal terms
        f, want = f + lam * v.ravel(), want + v.ravel()
    z = torch.zeros(m ** d, dtype=torch.float64, device="cuda")
    dcg.dcg_coarse_solve(prob, torch.from_numpy(f).cuda(), z)
    # FP32: m-term sums of rounding 2^-24 and the solve's conditioning (4 (m + 1)^2 / pi^2, smooth modes) on rough data
    tol = 1e-11 if precision == dcg.DCG_FP64 else 2.0 ** -24 * (m + 1) ** 2
    assert np.abs(z.cpu().numpy() - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("d,n", [(3, 8), (3, 10), (3, 16), (3, 18), (3, 24), (2, 164), (2, 256)])
def test_residual_forms(d, n):
    o = mg.MGOptions(patch=4, overlap=1, m1=2, m2=2, max_levels=2)
    asm = fem.assemble(d, n, 1e-3)
    Z = mg.inner_matrix(fem.V_matrix(asm.mesh), asm.matrix())
    prob = dcg.dcg_assemble(d, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(patch=4, overlap=1, max_levels=2))
    g = inputs.rhs(21, prob.n_nodes)
    gt, z = torch.from_numpy(g).cuda(), torch.zeros(prob.n_nodes, dtype=torch.float64, device="cuda")
    dcg.dcg_mg_cycles(prob, gt, z, 1)
    want = mg.Hierarchy(d, n, Z, o).wcycle(g, np.zeros_like(g))
    assert np.abs(z.cpu().numpy() - want).max() <= 1e-10 * np.abs(want).max()
    # one cycle too few or too many for a tolerance just above / below the true residual
    r = np.linalg.norm(g - Z @ z.cpu().numpy()) / np.linalg.norm(g)
    for tol, cycles in ((r + 1e-10, 1), (r - 1e-10, 2)):
        assert dcg.dcg_mg_solve(prob, gt, torch.zeros_like(gt), tol, 5) == cycles
