"""Error of one FP64 smoothing step against extended precision on iterates as
they occur near convergence: smooth, steep inside a box, one large entry over
small noise, each with f = Z z rounded to FP64, and random data.

Tolerance: the same step in plain FP64 arithmetic (numpy: residual, sine
transforms, division by the eigenvalues) has some error, the largest of four
forms of the residual: by the 1D factors, by the stencil, by the sums over
neighbours with equal coefficients, and in 3D this with the centre coefficient
one unit (2^-52) off, since that residual takes its coefficients from the
assembled operator. The kernel may have twice that (its solves round in yet another
order) and at least twice 2^-53 of the largest entry, the rounding of the
result itself and of its last addition.
"""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2606_13429_gb300 import dcg

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2606_13429_gb300 import build
    build.build()
    dcg.load()
    torch.cuda.set_device(0)


def _along(v, ax, off, dia):
    r = dia * v
    up, dn = [slice(None)] * v.ndim, [slice(None)] * v.ndim
    up[ax], dn[ax] = slice(1, None), slice(None, -1)
    r[tuple(up)] += off * v[tuple(dn)]
    r[tuple(dn)] += off * v[tuple(up)]
    return r


def _inner(z, n):
    """Z z in z's arithmetic: (1/d) sum over i of K along axis i, M along the others."""
    d, h, out = z.ndim, z.dtype.type(1) / n, 0
    for i in range(d):
        v = z
        for ax in range(d):
            v = _along(v, ax, -1 / h, 2 / h) if ax == i else _along(v, ax, h / 6, 4 * h / 6)
        out = out + v
    return out / d


def _stencil(z, n):
    """Z z as the sum over the 3^d neighbours, coefficients rounded to z's type."""
    d, m, out = z.ndim, n - 1, np.zeros_like(z)
    K, M = np.array([-n, 2 * n, -n], dtype=LD), np.array([1, 4, 1], dtype=LD) / (6 * LD(n))
    g = np.zeros((m + 2,) * d, dtype=z.dtype)
    g[(slice(1, -1),) * d] = z
    for off in itertools.product(range(3), repeat=d):
        c = sum(np.prod([K[off[ax]] if ax == i else M[off[ax]] for ax in range(d)]) for i in range(d)) / d
        out += z.dtype.type(c) * g[tuple(slice(q, q + m) for q in off)]
    return out


def _equal(z, n, unit=0.0):
    """Z z by neighbours at equal distance: 2D c1 (3 x 3 sum) + c0 z, 3D c3 (8
    corners + 2 (12 edges)) + c0 z."""
    d, m, T, sums = z.ndim, n - 1, z.dtype.type, {}
    g = np.zeros((m + 2,) * d, dtype=z.dtype)
    g[(slice(1, -1),) * d] = z
    for off in itertools.product(range(3), repeat=d):
        k = sum(q != 1 for q in off)
        sums[k] = sums.get(k, 0) + g[tuple(slice(q, q + m) for q in off)]
    if d == 2:
        return T(-1 / LD(6)) * (sums[1] + sums[2] + z) + T(9 / LD(6) * (1 + LD(unit))) * z
    return T(-1 / (36 * LD(n))) * (sums[3] + 2 * sums[2]) + T(32 / (36 * LD(n)) * (1 + LD(unit))) * z


def _step(f, z, n, P, o, inner=_inner):
    """One step with weights 1/multiplicity, in the arithmetic of f and z."""
    T, d, m = z.dtype.type, z.ndim, n - 1
    h, r = T(1) / n, f - inner(z, n)
    acc, mult = np.zeros_like(r), np.zeros_like(r)
    rng = [(max(0, t - o), min(m, t + P + o)) for t in range(0, m, P)]
    for box in itertools.product(rng, repeat=d):
        sl, v, D = tuple(slice(*b) for b in box), None, 0
        j = [np.arange(1, b[1] - b[0] + 1) for b in box]
        S = [(np.sqrt(LD(2) / (k.size + 1)) * np.sin(PI * (np.outer(k, k) % (2 * k.size + 2)) / (k.size + 1))).astype(T)
             for k in j]
        v = r[sl]
        for ax in range(d):
            v = np.moveaxis(np.tensordot(S[ax], v, axes=([1], [ax])), 0, ax)
        for i in range(d):
            t = T(1)
            for ax in range(d):
                c = np.cos(PI * j[ax] / (j[ax].size + 1))
                e = ((2 / h) * (1 - c) if ax == i else (h / 3) * (2 + c)).astype(T)
                t = t * e.reshape([-1 if q == ax else 1 for q in range(d)])
            D = D + t / d
        v = v / D
        for ax in range(d):
            v = np.moveaxis(np.tensordot(S[ax], v, axes=([1], [ax])), 0, ax)
        acc[sl] += v
        mult[sl] += 1
    return z + acc / mult


def _data(kind, d, n):
    m, rs = n - 1, np.random.RandomState(5)

    def product(v):
        r = v
        for _ in range(d - 1):
            r = np.multiply.outer(r, v)
        return r

    if kind == "random":
        return rs.uniform(-1, 1, (m,) * d), rs.uniform(-1, 1, (m,) * d)
    if kind == "smooth":
        z = product(np.sin(np.pi * np.arange(1, n) / n))
    elif kind == "steep":
        z = product(np.exp(-0.5 * np.arange(m)))
    else:
        z = 1e-8 * rs.uniform(-1, 1, (m,) * d)
        z[(m // 2,) * d] += 1.0
    return np.asarray(_inner(z.astype(LD), n), dtype=np.float64), z


@pytest.mark.parametrize("d,n,P,o", [(2, 48, 4, 1), (2, 48, 8, 2), (2, 52, 12, 2), (3, 16, 4, 1), (3, 16, 2, 1)])
@pytest.mark.parametrize("kind", ["random", "smooth", "steep", "peak"])
def test_step(d, n, P, o, kind):
    f, z = _data(kind, d, n)
    want = _step(f.astype(LD), z.astype(LD), n, P, o)
    size = np.abs(want).max()
    forms = (_inner, _stencil, _equal) + ((lambda v, k: _equal(v, k, 2.0 ** -52),) if d == 3 else ())
    plain = max(np.abs(_step(f, z, n, P, o, form) - want).max() for form in forms) / size
    prob = dcg.dcg_assemble(d, n, 1e-3)
    dcg.dcg_setup(prob, dcg.options(patch=P, overlap=o, max_levels=2))
    zt = torch.from_numpy(z.reshape(-1).copy()).cuda()
    dcg.dcg_ras_step(prob, 2, torch.from_numpy(f.reshape(-1).copy()).cuda(), zt)
    err = np.abs(zt.cpu().numpy().reshape(z.shape) - want).max() / size
    print("error %.2e, plain FP64 %.2e" % (err, plain))
    assert err <= 2 * max(plain, 2.0 ** -53)
