"""The FP64 smoother's fixed-point local solves against the oracle: every
compile-time extent, odd and ragged box extents (the general path beside the
interior class), scales near the ends of the FP64 range, and non-finite input.

Tolerance: the kernel keeps at least 52 bits below the largest entry of a box
and amplifies its rounding by at most the norm of the local inverse (below
2^6 for the extents used), so 1e-12 of the largest result holds with room.
"""
import itertools

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


def _setup(d, n, P, o):
    asm = fem.assemble(d, n, 1e-3)
    H = mg.Hierarchy(d, n, mg.inner_matrix(fem.V_matrix(asm.mesh), asm.matrix()),
                     mg.MGOptions(patch=P, overlap=o, m1=2, m2=2, max_levels=2))
    prob = dcg.dcg_assemble(d, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(patch=P, overlap=o, max_levels=2))
    return H, prob


def _step(prob, f, z):
    ft, zt = torch.from_numpy(f).cuda(), torch.from_numpy(z.copy()).cuda()
    dcg.dcg_ras_step(prob, 2, ft, zt)
    torch.cuda.synchronize()
    return zt.cpu().numpy()


# extents: 4, 5 (odd), 6, 7 (odd), 8, 10, 12, 16 in 2D; 4, 5, 6 in 3D
@pytest.mark.parametrize("d,n,P,o", [(2, 22, 2, 1), (2, 30, 3, 1), (2, 34, 4, 1), (2, 36, 5, 1), (2, 38, 6, 1),
                                     (2, 46, 8, 1), (2, 52, 8, 2), (2, 62, 12, 2), (3, 10, 2, 1), (3, 12, 3, 1),
                                     (3, 16, 4, 1)])
def test_every_extent(d, n, P, o):
    H, prob = _setup(d, n, P, o)
    nn = prob.n_nodes
    f, z = inputs.rhs(7, nn), inputs.rhs(8, nn)
    for scale in (1.0, 1e-200, 1e200):
        want = H.ras_step(2, f, z) * scale
        got = _step(prob, f * scale, z * scale)
        assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max(), scale
    # one nonzero entry: boxes that hold nothing stay exactly zero
    g = np.zeros(nn)
    g[nn // 2] = 1.0
    want = H.ras_step(2, g, np.zeros(nn))
    got = _step(prob, g, np.zeros(nn))
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
    assert got[0] == 0.0 and got[-1] == 0.0


@pytest.mark.parametrize("d,n", [(2, 24), (3, 10)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_entries_stay_visible(d, n, bad):
    _, prob = _setup(d, n, 4, 1)
    nn = prob.n_nodes
    f = inputs.rhs(9, nn)
    f[nn // 2] = bad
    got = _step(prob, f, np.zeros(nn))
    # non-finite exactly on the boxes that contain the entry
    m, mask = n - 1, np.zeros((n - 1,) * d, dtype=bool)
    c = np.unravel_index(nn // 2, mask.shape)
    rng = [(max(0, t - 1), min(m, t + 5)) for t in range(0, m, 4)]
    for box in itertools.product(rng, repeat=d):
        if all(lo <= c[k] < hi for k, (lo, hi) in enumerate(box)):
            mask[tuple(slice(lo, hi) for lo, hi in box)] = True
    assert np.array_equal(np.isfinite(got), ~mask.reshape(-1))
