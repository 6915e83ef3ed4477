"""The one-kernel inner solve of small 2D hierarchies against the
level-by-level kernels of the same library (which timing of a kernel class
selects) and, for one hierarchy, the oracle's W-cycle: one CTA for all levels,
solo levels under a cluster, groups of boxes on the finest level, dense
coarsest levels, no and odd numbers of smoothing steps, restricted weights.

Tolerance: both paths run the same smoothing steps and transfers; the coarsest
solves differ by rounding, which a cycle amplifies by less than 10^3, so 1e-12
of the largest entry holds.
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


def _cycles(prob, g, n):
    z = torch.zeros_like(g)
    dcg.dcg_mg_cycles(prob, g, z, n)
    torch.cuda.synchronize()
    return z


@pytest.mark.parametrize("n,levels,P,o,m1,m2", [(8, 2, 4, 1, 2, 2), (16, 4, 4, 1, 2, 2), (26, 2, 4, 1, 2, 2),
                                                (32, 4, 4, 1, 1, 3), (40, 3, 2, 1, 2, 2), (64, 4, 8, 2, 2, 2),
                                                (72, 3, 6, 1, 0, 1), (96, 4, 4, 1, 2, 2), (96, 2, 12, 2, 2, 2),
                                                (130, 2, 5, 1, 2, 2), (160, 3, 8, 1, 1, 1), (162, 2, 4, 1, 2, 0)])
@pytest.mark.parametrize("weights", [0, 1])
def test_matches_level_kernels(n, levels, P, o, m1, m2, weights):
    prob = dcg.dcg_assemble(2, n, 1e-4)
    dcg.dcg_setup(prob, dcg.options(max_levels=levels, patch=P, overlap=o, m1=m1, m2=m2, ras_weights=weights))
    g = torch.from_numpy(inputs.rhs(11, prob.n_nodes)).cuda()
    k0 = dcg.dcg_kernel_launches()
    one = _cycles(prob, g, 2)
    # the one-kernel path ran, up to its sizes: 26,000 nodes, 13,000 with two levels
    assert (dcg.dcg_kernel_launches() - k0 == 1) == (prob.n_nodes <= (26000 if prob.levels > 2 else 13000))
    dcg.dcg_profile_enable(prob, ["coarse"])
    many = _cycles(prob, g, 2)
    dcg.dcg_profile_enable(prob, [])
    assert (one - many).abs().max().item() <= 1e-12 * many.abs().max().item()
    # Algorithm 3 stops at the tolerance with the same cycle count
    z1, z2 = torch.zeros_like(g), torch.zeros_like(g)
    n1 = dcg.dcg_mg_solve(prob, g, z1, 1e-6, 60)
    dcg.dcg_profile_enable(prob, ["coarse"])
    n2 = dcg.dcg_mg_solve(prob, g, z2, 1e-6, 60)
    assert n1 == n2 and (z1 - z2).abs().max().item() <= 1e-10 * z2.abs().max().item()


def test_matches_oracle():
    n, o = 48, mg.MGOptions(patch=4, overlap=1, m1=2, m2=2, max_levels=4)
    asm = fem.assemble(2, n, 1e-3)
    H = mg.Hierarchy(2, n, mg.inner_matrix(fem.V_matrix(asm.mesh), asm.matrix()), o)
    prob = dcg.dcg_assemble(2, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(patch=4, overlap=1, max_levels=4))
    g = inputs.rhs(12, prob.n_nodes)
    z = _cycles(prob, torch.from_numpy(g).cuda(), 1).cpu().numpy()
    want = H.wcycle(g, np.zeros_like(g))
    assert np.abs(z - want).max() <= 1e-10 * np.abs(want).max()


def test_zero_right_hand_side_and_cycle_cap():
    prob = dcg.dcg_assemble(2, 32, 1e-4)
    dcg.dcg_setup(prob, dcg.options())
    g = torch.zeros(prob.n_nodes, dtype=torch.float64, device="cuda")
    z = torch.zeros_like(g)
    assert dcg.dcg_mg_solve(prob, g, z, 1e-10) == 0 and z.abs().max().item() == 0.0
    g = torch.from_numpy(inputs.rhs(13, prob.n_nodes)).cuda()
    assert dcg.dcg_mg_solve(prob, g, z, 1e-14, 1) == 1
