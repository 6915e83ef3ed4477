"""Performance cases of the deflated-CG library: the calls its users make.

Each case is one call of a public entry point on device arrays: the operator
products an outer iteration spends (assembled 2D and 3D, matrix-free in both
precisions), the inner multigrid solves (Algorithm 3 to the relative tolerance
1e-10 that an outer tolerance of 1e-8 with c_F = 0.01 asks for), the right-hand
side of a time step, and whole solves (a small one, the 1024^2 headline
workload, and a batch in mixed precision). Sizes are those of the benchmark's
workloads and of the tests, with odd and ragged ones between.
"""
import math

import numpy as np
import torch

from paper_2606_13429_gb300 import dcg


def listed():
    return [
        # the assembled product: once per outer iteration and per plain-CG
        # iteration; at the headline size and at the tests' 3D scale
        {"name": "spmv_2d_1024", "kind": "spmv", "d": 2, "n": 1024, "dt": 1e-4, "nu": "one"},
        {"name": "spmv_3d_80", "kind": "spmv", "d": 3, "n": 80, "dt": 1e-4, "nu": "one"},
        # matrix-free products with a viscosity per element: FP64 for the true
        # residual and the reconstruction (odd extent), FP32 arithmetic for the
        # outer iterations of the mixed mode at the 256^3 workload
        {"name": "mf_fp64_129", "kind": "mf", "n": 129, "dt": 1e-5, "nu": "lognormal", "prec": "fp64"},
        {"name": "mf_fp32_256", "kind": "mf", "n": 256, "dt": 1e-5, "nu": "lognormal", "prec": "mixed"},
        # inner solves: smallest levels (launches count), the headline
        # hierarchy, the batch's autotuned mixed hierarchy at a size whose
        # coarsest level is no power of two, and 3D
        {"name": "mg_2d_96", "kind": "mg", "d": 2, "n": 96, "levels": 4, "P": 4, "o": 1, "prec": "fp64"},
        {"name": "mg_2d_1024", "kind": "mg", "d": 2, "n": 1024, "levels": 2, "P": 8, "o": 2, "prec": "fp64"},
        {"name": "mg_2d_496_bf16", "kind": "mg", "d": 2, "n": 496, "levels": 2, "P": 4, "o": 1, "prec": "bf16"},
        {"name": "mg_3d_128", "kind": "mg", "d": 3, "n": 128, "levels": 4, "P": 4, "o": 1, "prec": "fp64"},
        # right-hand side of a Crank-Nicolson step (time stepping)
        {"name": "rhs_cn_2d_700", "kind": "rhs", "d": 2, "n": 700, "dt": 1e-4, "scheme": 1, "nu": "lognormal"},
        # whole solves: a small one, one of the headline's six, and a batch of
        # mixed-precision problems with two right-hand sides each
        {"name": "solve_2d_32", "kind": "solve", "n": 32, "dt": 1e-4, "levels": 4, "P": 4, "o": 1},
        {"name": "solve_2d_1024", "kind": "solve", "n": 1024, "dt": 1e-6, "levels": 2, "P": 8, "o": 2},
        {"name": "batch_mixed", "kind": "batch", "n0": 64, "count": 6, "nrhs": 2, "dt": 1e-5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmv2", "spmv3", "mf", "mg2", "mg2", "mg3", "rhs", "solve", "batch"])
    dt = 10.0 ** rng.uniform(-6.0, -2.0)
    nu = rng.choice(["one", "lognormal"])
    if kind == "spmv2":
        return {"kind": "spmv", "d": 2, "n": _log(rng, 24, 1024), "dt": dt, "nu": nu}
    if kind == "spmv3":
        return {"kind": "spmv", "d": 3, "n": _log(rng, 6, 80), "dt": dt, "nu": nu}
    if kind == "mf":
        return {"kind": "mf", "n": _log(rng, 8, 200), "dt": dt, "nu": nu, "prec": rng.choice(["fp64", "mixed"])}
    if kind == "mg2":
        P, o = rng.choice([(4, 1), (8, 1), (8, 2), (12, 2)])
        return {"kind": "mg", "d": 2, "n": _log(rng, 24, 1024), "levels": rng.choice([2, 3, 4]), "P": P, "o": o,
                "prec": rng.choice(["fp64", "fp64", "fp32", "bf16"])}
    if kind == "mg3":
        return {"kind": "mg", "d": 3, "n": _log(rng, 8, 128), "levels": rng.choice([2, 3, 4]), "P": 4, "o": 1,
                "prec": rng.choice(["fp64", "fp64", "fp32", "bf16"])}
    if kind == "rhs":
        return {"kind": "rhs", "d": 2, "n": _log(rng, 24, 1000), "dt": dt, "scheme": rng.choice([0, 1, 2]), "nu": nu}
    if kind == "solve":
        P, o = rng.choice([(4, 1), (8, 2)])
        return {"kind": "solve", "n": 2 * _log(rng, 8, 128), "dt": 10.0 ** rng.uniform(-6.0, -4.0),
                "levels": rng.choice([2, 3, 4]), "P": P, "o": o}
    return {"kind": "batch", "n0": 16 * rng.randint(2, 6), "count": rng.randint(2, 6), "nrhs": rng.randint(1, 3),
            "dt": 10.0 ** rng.uniform(-6.0, -4.5)}


# ---------------------------------------------------------------------------


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _uniform(seed, stream, n):
    """i.i.d. uniform on [-1, 1), the right-hand sides of every workload."""
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=_gen(seed, stream)).mul_(2.0).sub_(1.0)


def _nu(case, seed):
    """Per-element viscosity lognormal(0, 1) on the host, or None for 1."""
    if case.get("nu") != "lognormal":
        return None
    d = case.get("d", 3)
    g = torch.randn(case["n"] ** d, dtype=torch.float64, device="cuda", generator=_gen(seed, 77))
    return g.exp_().cpu().numpy()


_PREC = {"fp64": {}, "fp32": {"precision": dcg.DCG_MIXED, "ras_inverse": dcg.DCG_INV_FP32},
         "bf16": {"precision": dcg.DCG_MIXED, "ras_inverse": dcg.DCG_INV_BF16}}


def _batch_sizes(case):
    return [(case["n0"] + 16 * i, case["dt"] * 2.0 ** i) for i in range(case["count"])]


def prepare(case, seed):
    k = case["kind"]
    if k in ("spmv", "mf"):
        d = case.get("d", 3)
        p = dcg.dcg_assemble(d, case["n"], case["dt"], nu_elem=_nu(case, seed), matrix_free=k == "mf")
        x = _uniform(seed, 1, p.N)
        return {"case": case, "p": p, "x": x, "y": torch.empty_like(x)}
    if k == "mg":
        # the inner system does not depend on dt or the viscosity; in 3D the
        # matrix-free operator provides it without the assembled matrix
        p = dcg.dcg_assemble(case["d"], case["n"], 1e-4, matrix_free=case["d"] == 3)
        dcg.dcg_setup(p, dcg.options(max_levels=case["levels"], patch=case["P"], overlap=case["o"],
                                     **_PREC[case["prec"]]))
        g = _uniform(seed, 2, p.n_nodes)
        return {"case": case, "p": p, "g": g, "z": torch.zeros_like(g)}
    if k == "rhs":
        alpha = dcg.dcg_scheme_alpha(case["scheme"], case["dt"])
        p = dcg.dcg_assemble(case["d"], case["n"], alpha, nu_elem=_nu(case, seed))
        v = [_uniform(seed, 3 + i, p.N) for i in range(4)]
        return {"case": case, "p": p, "v": v, "b": torch.empty_like(v[0])}
    if k == "solve":
        p = dcg.dcg_assemble(2, case["n"], case["dt"])
        dcg.dcg_setup(p, dcg.options(max_levels=case["levels"], patch=case["P"], overlap=case["o"]))
        f = _uniform(seed, 8, p.N)
        return {"case": case, "p": p, "f": f, "x": torch.zeros_like(f)}
    ps, fs, xs = [], [], []
    for i, (n, dt) in enumerate(_batch_sizes(case)):
        p = dcg.dcg_assemble(2, n, dt)
        dcg.dcg_setup(p, dcg.options(max_levels=2, patch=4, overlap=1, **_PREC["bf16"]))
        ps.append(p)
        for r in range(case["nrhs"]):
            fs.append(_uniform(seed, 100 + 10 * i + r, p.N))
            xs.append(torch.zeros_like(fs[-1]))
    return {"case": case, "ps": ps, "fs": fs, "xs": xs}


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "spmv":
        dcg.dcg_spmv(s["p"], s["x"], s["y"])
        return s["y"]
    if k == "mf":
        dcg.dcg_spmv_prec(s["p"], s["x"], s["y"], dcg.DCG_FP64 if c["prec"] == "fp64" else dcg.DCG_MIXED)
        return s["y"]
    if k == "mg":
        s["z"].zero_()
        dcg.dcg_mg_solve(s["p"], s["g"], s["z"], 1e-10)
        return s["z"]
    if k == "rhs":
        s1, s2, f1, f0 = s["v"]
        dcg.dcg_time_rhs(s["p"], c["scheme"], s1, f1, s["b"], s2=s2 if c["scheme"] == dcg.DCG_BDF2 else None,
                         F0=f0 if c["scheme"] == dcg.DCG_CRANK_NICOLSON else None)
        return s["b"]
    if k == "solve":
        s["x"].zero_()
        dcg.dcg_solve(s["p"], s["f"], s["x"], tol=1e-8, max_it=2000)
        return s["x"]
    for x in s["xs"]:
        x.zero_()
    dcg.dcg_solve_batched(s["ps"], c["nrhs"], s["fs"], s["xs"], tol=1e-8, max_it=2000)
    return list(s["xs"])


# ---------------------------------------------------------------------------


def work(case):
    """Bytes and operations the call cannot do without: inputs (the stored
    operator's structural entries among them) read once, outputs written once;
    for the iterative calls the vectors alone and one pass of the method's
    arithmetic (one W-cycle with two smoothing steps each way, or one outer
    iteration), since the number of passes depends on the data."""
    k = case["kind"]
    if k in ("spmv", "mf", "rhs"):
        d, n = case.get("d", 3), case["n"]
        nn, b = float(n - 1) ** d, d * d
        nz = 10.0 if d == 2 else 33.0
        blocks = float(3 * (n - 1) - 2) ** d
        if k == "mf":
            return {"bytes": nn * b * 16.0 + (8.0 * n ** 3 if case["nu"] != "one" else 0.0), "flops": 2.0 * 702.0 * nn}
        extra = 0.0 if k == "spmv" else (16.0 if case["scheme"] else 8.0) * nn * b
        return {"bytes": blocks * nz * 8.0 + nn * b * 16.0 + extra, "flops": 2.0 * nz * blocks}
    if k == "mg":
        nn = float(case["n"] - 1) ** case["d"]
        return {"bytes": 16.0 * nn, "flops": 400.0 * nn}
    if k == "solve":
        nn = float(case["n"] - 1) ** 2
        return {"bytes": nn * (64.0 + 9.0 * 80.0), "flops": 1000.0 * nn}
    nn = sum(float(n - 1) ** 2 for n, _ in _batch_sizes(case))
    return {"bytes": nn * (64.0 * case["nrhs"] + 9.0 * 80.0), "flops": 1000.0 * nn * case["nrhs"]}


# --- plain 64-bit values ----------------------------------------------------


def _element_1d(n):
    h = 1.0 / n
    mass = [[h / 3.0, h / 6.0], [h / 6.0, h / 3.0]]
    stiff = [[1.0 / h, -1.0 / h], [-1.0 / h, 1.0 / h]]
    mixed = [[-0.5, -0.5], [0.5, 0.5]]  # int phi_a' phi_b
    return mass, stiff, mixed


def _apply(d, n, w, x):
    """(M_dev x with the weights w = 1/(nu dt), K_div x) for x of shape
    [..., m^d nodes (x fastest), d, d], summed element corner by corner."""
    mass, stiff, mixed = _element_1d(n)
    lead = x.dim() - d - 2
    grid = x.new_zeros(list(x.shape[:lead]) + [n + 1] * d + [d, d])
    inner = (slice(None),) * lead + (slice(1, n),) * d
    grid[inner] = x
    tr = grid.diagonal(dim1=-2, dim2=-1).sum(-1)
    dev = grid - tr[..., None, None] * torch.eye(d, dtype=x.dtype, device=x.device) / d
    ym, yk = torch.zeros_like(grid), torch.zeros_like(grid)

    def corner(bits):
        # axes of the array run from the last coordinate to x
        return (slice(None),) * lead + tuple(slice((bits >> (d - 1 - ax)) & 1, n + ((bits >> (d - 1 - ax)) & 1))
                                             for ax in range(d))

    wt = w if not torch.is_tensor(w) else w.reshape([n] * d)[..., None, None]
    for a in range(1 << d):
        ca = corner(a)
        for b in range(1 << d):
            cb = corner(b)
            mab = 1.0
            G = torch.empty(d, d, dtype=x.dtype)
            for k in range(d):
                mab *= mass[(a >> k) & 1][(b >> k) & 1]
            for p in range(d):
                for q in range(d):
                    v = 1.0
                    for k in range(d):
                        i, j = (a >> k) & 1, (b >> k) & 1
                        v *= stiff[i][j] if k == p and k == q else mixed[i][j] if k == p else mixed[j][i] if k == q \
                            else mass[i][j]
                    G[p, q] = v
            ym[ca] += wt * mab * dev[cb]
            yk[ca] += torch.matmul(grid[cb], G.to(x.device).t())
    return ym[inner].contiguous(), yk[inner].contiguous()


def _weights(case, seed, dt):
    nu = _nu(case, seed)
    return 1.0 / dt if nu is None else (1.0 / torch.from_numpy(nu).cuda()) / dt


def exact(case, seed):
    k = case["kind"]
    if k in ("spmv", "mf"):
        d, n = case.get("d", 3), case["n"]
        m = n - 1
        x = _uniform(seed, 1, m ** d * d * d).reshape([m] * d + [d, d])
        ym, yk = _apply(d, n, _weights(case, seed, case["dt"]), x)
        return (ym + yk).reshape(-1)
    if k == "rhs":
        d, n, sch = case["d"], case["n"], case["scheme"]
        m = n - 1
        s1, s2, f1, f0 = [_uniform(seed, 3 + i, m ** d * d * d) for i in range(4)]
        alpha = (1.0, 0.5, 2.0 / 3.0)[sch] * case["dt"]
        v = 4.0 / 3.0 * s1 - 1.0 / 3.0 * s2 if sch == 2 else s1
        ym, yk = _apply(d, n, _weights(case, seed, alpha), v.reshape([m] * d + [d, d]))
        b = ym.reshape(-1) + f1
        return b - yk.reshape(-1) + f0 if sch == 1 else b
    if k == "mg":
        # Z_J = (1/d) sum_i (stiffness along axis i, mass along the others),
        # diagonal in the sine basis
        d, n = case["d"], case["n"]
        m, h = n - 1, 1.0 / n
        g = _uniform(seed, 2, m ** d).reshape([m] * d)
        j = torch.arange(1, n, dtype=torch.float64, device="cuda")
        S = math.sqrt(2.0 / n) * torch.sin(math.pi / n * torch.remainder(j[:, None] * j[None, :], 2 * n))
        th = math.pi * j / n
        kap, mu = (2.0 / h) * (1.0 - torch.cos(th)), (h / 3.0) * (2.0 + torch.cos(th))
        lam = torch.zeros([m] * d, dtype=torch.float64, device="cuda")
        for i in range(d):
            t = torch.ones([m] * d, dtype=torch.float64, device="cuda")
            for ax in range(d):
                t = t * (kap if ax == i else mu).reshape([-1 if q == ax else 1 for q in range(d)])
            lam += t / d
        for ax in range(d):
            g = torch.tensordot(S, g, dims=([1], [ax])).movedim(0, ax)
        g = g / lam
        for ax in range(d):
            g = torch.tensordot(S, g, dims=([1], [ax])).movedim(0, ax)
        return g.contiguous().reshape(-1)
    if k == "solve":
        n = case["n"]
        N = 4 * (n - 1) ** 2
        if n > 48:
            return None  # a direct solve takes too long
        m = n - 1
        A = torch.empty(N, N, dtype=torch.float64, device="cuda")
        for c0 in range(0, N, 512):
            c1 = min(N, c0 + 512)
            e = torch.zeros(c1 - c0, N, dtype=torch.float64, device="cuda")
            e[torch.arange(c1 - c0), torch.arange(c0, c1)] = 1.0
            ym, yk = _apply(2, n, 1.0 / case["dt"], e.reshape(-1, m, m, 2, 2))
            A[c0:c1] = (ym + yk).reshape(c1 - c0, N)
        f = torch.from_numpy(_uniform(seed, 8, N).cpu().numpy())
        return torch.from_numpy(np.linalg.solve(A.cpu().numpy(), f.numpy())).cuda()
    return None
