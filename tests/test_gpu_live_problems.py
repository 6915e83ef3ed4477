"""Several live problems of different sizes: a kernel's launch limits must not
depend on which problem was set up last. Every size is set up first, then each
problem is used, one by one and as one batch in both orders.

Tolerance: a solve ends at a true relative residual of 1e-8; an inner solve
reaches its relative tolerance, checked against the library's own Z_J product.
"""
import pytest

torch = pytest.importorskip("torch")

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


def _problems(d, sizes, **kw):
    ps = [dcg.dcg_assemble(d, n, 1e-5) for n in sizes]
    for p in ps:
        dcg.dcg_setup(p, dcg.options(**kw))
    return ps


def _inner_solves(ps, tol):
    for p in ps:
        g = torch.from_numpy(inputs.rhs(31, p.n_nodes)).cuda()
        z, y = torch.zeros_like(g), torch.empty_like(g)
        dcg.dcg_mg_solve(p, g, z, tol)
        dcg.dcg_inner_apply(p, z, y)
        assert (torch.linalg.norm(g - y) / torch.linalg.norm(g)).item() <= 1.01 * tol


# one CTA or a cluster, four levels and two: the shared memory of the small
# inner solve differs from size to size, and is largest at 32
@pytest.mark.parametrize("levels", [4, 2])
def test_small_inner_solves(levels):
    sizes = [32, 24, 40, 96, 16]
    for order in (sizes, sizes[::-1]):
        ps = _problems(2, order, max_levels=levels)
        _inner_solves(ps, 1e-8)
        fs = [torch.from_numpy(inputs.rhs(32 + i, p.N)).cuda() for i, p in enumerate(ps)]
        for batch in (ps, ps[::-1]):
            f = [fs[ps.index(p)] for p in batch]
            xs = [torch.zeros_like(v) for v in f]
            for st in dcg.dcg_solve_batched(batch, 1, f, xs, tol=1e-8, max_it=2000)[1]:
                assert st["status"] == dcg.DCG_OK and st["true_relres"] <= 1e-8
        for p, f in zip(ps, fs):
            st = dcg.dcg_solve(p, f, torch.zeros_like(f), tol=1e-8, max_it=2000)
            assert st["status"] == dcg.DCG_OK and st["true_relres"] <= 1e-8


# box solves: 3D problems whose boxes are smaller than the compile-time extent
# (6 per axis) need less shared memory, as do 2D levels with smaller boxes
@pytest.mark.parametrize("d,first,then", [(3, (16, 4, 1), (8, 4, 1)), (3, (16, 4, 1), (12, 3, 1)),
                                          (2, (22, 4, 1), (12, 3, 1)), (2, (46, 8, 2), (22, 7, 2))])
def test_smoothing_steps(d, first, then):
    ps, want = [], []
    for n, P, o in (first, then):
        p = dcg.dcg_assemble(d, n, 1e-4)
        dcg.dcg_setup(p, dcg.options(max_levels=2, patch=P, overlap=o))
        f = torch.from_numpy(inputs.rhs(33, p.n_nodes)).cuda()
        z = torch.zeros_like(f)
        dcg.dcg_ras_step(p, 2, f, z)
        ps.append((p, f))
        want.append(z)
    for (p, f), w in zip(ps, want):  # the first again, after the second was set up
        z = torch.zeros_like(f)
        dcg.dcg_ras_step(p, 2, f, z)
        assert torch.equal(z, w)
    if d == 3:
        _inner_solves([p for p, _ in ps], 1e-8)
