"""FP64 smoothing steps and W-cycles are linear: data scaled by a power of two
gives the scaled result, up to the ends of the FP64 range, in the one-kernel
inner solve, the level kernels and single steps, with boxes that hold only
zeros among the others.

Tolerance: a power of two changes no rounding except where a value becomes
subnormal: half a unit of 2^-1074 on each of fewer than 2^12 values a result
combines, with factors below 2^8 (norms of the local and coarse inverses).
"""
import pytest

torch = pytest.importorskip("torch")

from paper_2606_13429_gb300 import dcg, inputs

pytestmark = pytest.mark.gpu

SCALES = [-960, -1010, -1040, 990]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2606_13429_gb300 import build
    build.build()
    dcg.load()
    torch.cuda.set_device(0)


def _scaled(v, k):
    return v * 2.0 ** (k // 2) * 2.0 ** (k - k // 2)  # either factor is a number


def _compare(run, v):
    want = run(v)
    size = want.abs().max().item()
    for k in SCALES:
        got = run([_scaled(t, k) for t in v] if isinstance(v, list) else _scaled(v, k))
        got = _scaled(got, -k)
        tol = 2.0 ** (-1074 + 20 - k) if k < 0 else 0.0
        assert (got - want).abs().max().item() <= tol + 2.0 ** -52 * size, k


@pytest.mark.parametrize("d,n,P,o", [(2, 22, 2, 1), (2, 34, 4, 1), (2, 46, 8, 2), (2, 62, 12, 2), (3, 10, 2, 1),
                                     (3, 16, 4, 1)])
@pytest.mark.parametrize("zero_z", [False, True])
def test_step(d, n, P, o, zero_z):
    prob = dcg.dcg_assemble(d, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(patch=P, overlap=o, max_levels=2))
    f = torch.from_numpy(inputs.rhs(41, prob.n_nodes)).cuda()
    z = torch.from_numpy(inputs.rhs(42, prob.n_nodes)).cuda()
    if zero_z:
        z.zero_()
        f[: prob.n_nodes // 2] = 0.0

    def run(v):
        y = v[1].clone()
        dcg.dcg_ras_step(prob, 2, v[0], y)
        return y

    _compare(run, [f, z])


@pytest.mark.parametrize("d,n,levels,P,o", [(2, 24, 4, 4, 1), (2, 64, 3, 4, 1), (2, 96, 4, 2, 1), (2, 256, 2, 8, 2),
                                            (3, 16, 2, 4, 1)])
def test_cycle(d, n, levels, P, o):
    prob = dcg.dcg_assemble(d, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(patch=P, overlap=o, max_levels=levels))
    g = torch.from_numpy(inputs.rhs(43, prob.n_nodes)).cuda()

    def run(v):
        z = torch.zeros_like(v)
        dcg.dcg_mg_cycles(prob, v, z, 1)
        return z

    _compare(run, g)
