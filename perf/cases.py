"""Performance cases of the Helmholtz solver: what its users run, over the sizes they run it at.

Every case goes through the public binding ``paper_1312_2880_gb300.hz``. Solves run a fixed number
of Bi-CGSTAB iterations (an iteration budget, ``maxit``) instead of running to a tolerance: on these
indefinite systems Bi-CGSTAB amplifies rounding, while an iteration costs the same from the first to
the last. Scaling b by one ulp moves the iterate of the FP32-V-cycle form by 1e-15 up to the third
iteration and by up to 6e-4 at the eighth (an FP32 rounding flips), so longer runs of two correct
programs cannot be compared. ``exact`` is the same mathematics written out on dense 2-D arrays in
complex128, from the paper's definitions.
"""
import math

import numpy as np
import torch

from paper_1312_2880_gb300 import hz

BETA = 0.5
EIGHT = 8  # directions of the ray correction


def listed():
    return [
        # The plain method on its smallest grid, in the binding's default precision: launch latency.
        {"name": "solve_n64_fp64", "kind": "solve", "n": 64, "kh": 0.3125, "medium": "const", "variant": "sl_plain",
         "precision": "fp64", "maxit": 3},
        # One small served medium solved alone in the FP32-V-cycle form.
        {"name": "solve_n128_fp32", "kind": "solve", "n": 128, "kh": 2 * math.pi / 12, "medium": "wedge",
         "variant": "hyb", "precision": "fp32", "maxit": 3},
        # The hybrid hierarchy on the n = 512 wedge, both precisions.
        {"name": "solve_n512_fp32", "kind": "solve", "n": 512, "kh": 100.0 / 512, "medium": "wedge",
         "variant": "hyb", "precision": "fp32", "maxit": 3},
        {"name": "solve_n512_fp64", "kind": "solve", "n": 512, "kh": 100.0 / 512, "medium": "wedge",
         "variant": "hyb", "precision": "fp64", "maxit": 3},
        # The large heterogeneous problem (n = 4096, k = 1000, +-30% random medium), both precisions.
        {"name": "solve_n4096_fp32", "kind": "solve", "n": 4096, "kh": 1000.0 / 4096, "medium": "grf",
         "variant": "hyb", "precision": "fp32", "maxit": 3},
        {"name": "solve_n4096_fp64", "kind": "solve", "n": 4096, "kh": 1000.0 / 4096, "medium": "grf",
         "variant": "hyb", "precision": "fp64", "maxit": 3},
        # 64 right-hand sides over the four grids of the batched workload (n = 96 ... 576), one group solve.
        {"name": "group_n576_fp32", "kind": "group", "n": 576, "kh": 300.0 / 576, "grids": 4, "batch": 16,
         "precision": "fp32", "maxit": 3},
        # Three served requests of n = 256, 512, 1024 in flight at once through the non-blocking calls.
        {"name": "served_n1024_fp32", "kind": "served", "n": 1024, "kh": 2 * math.pi / 12, "medium": "grf",
         "precision": "fp32", "maxit": 3},
        # One V-cycle on its own, as a preconditioner of another iteration: a ragged grid (27 * 32) in
        # FP32, and the FP64 cycle on Table 1's largest grid (15 * 16).
        {"name": "vcycle_n864_fp32", "kind": "vcycle", "n": 864, "kh": 0.3, "medium": "grf", "variant": "hyb",
         "precision": "fp32"},
        {"name": "vcycle_n240_fp64", "kind": "vcycle", "n": 240, "kh": 0.625, "medium": "const", "variant": "hyb",
         "precision": "fp64"},
        # The operator alone (residual checks of a solution) on a ragged grid (31 * 64).
        {"name": "apply_n1984", "kind": "apply", "n": 1984, "kh": 0.25, "medium": "wedge", "op": "L"},
        # V-cycle + ray correction as a solver: Table 7's largest column, to its tolerance of 1e-7
        # (a contraction of ten cycles, which amplifies nothing).
        {"name": "cycle_n512_fp64", "kind": "cycle", "n": 512, "kh": 0.3125, "variant": "hlm", "precision": "fp64"},
    ]


# Grids with at most 1089 unknowns on the coarsest level: odd m <= 31 times a power of two.
_SIZES = sorted({m << p for m in range(1, 32, 2) for p in range(1, 13) if 64 <= m << p <= 4096})


def _size(rng, lo, hi):
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in _SIZES if lo <= n <= hi), key=lambda n: abs(math.log(n / want)))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "group", "served", "vcycle", "vcycle", "apply", "cycle"))
    prec = rng.choice(("fp32", "fp64"))
    medium = rng.choice(("const", "wedge", "grf"))
    kh = round(rng.uniform(0.19, 0.625), 4)
    if kind == "solve":
        n = _size(rng, 64, 3968 if prec == "fp32" else 2048)
        return {"kind": kind, "n": n, "kh": kh, "medium": medium, "variant": rng.choice(("hyb", "hyb", "sl", "sl_plain")),
                "precision": prec, "maxit": rng.choice((2, 3))}
    if kind == "group":
        return {"kind": kind, "n": rng.choice([n for n in _SIZES if 128 <= n <= 576 and n % 16 == 0]), "kh": kh,
                "grids": rng.randint(1, 3), "batch": rng.randint(2, 16), "precision": "fp32", "maxit": rng.choice((2, 3))}
    if kind == "served":
        return {"kind": kind, "n": rng.choice([n for n in _SIZES if 256 <= n <= 1536 and n % 16 == 0]), "kh": kh,
                "medium": medium, "precision": "fp32", "maxit": rng.choice((2, 3))}
    if kind == "vcycle":
        return {"kind": kind, "n": _size(rng, 64, 4096 if prec == "fp32" else 2048), "kh": kh, "medium": medium,
                "variant": rng.choice(("hyb", "sl", "sl_plain")), "precision": prec}
    if kind == "apply":
        return {"kind": kind, "n": _size(rng, 64, 4096), "kh": kh, "medium": medium, "op": rng.choice("LM")}
    # Table 7's constant scale kh = 0.3125: a ray grid of spacing 8h on every grid
    n = rng.choice([n for n in _SIZES if 64 <= n <= 480 and n % 8 == 0])
    return {"kind": kind, "n": n, "kh": 0.3125, "variant": "hlm", "precision": prec}


# ------------------------------------------------------------------ inputs


def _grids(case):
    """Grid sizes of a group (k h constant, sizes as in the batched workload) or of the served requests."""
    n = case["n"]
    if case["kind"] == "served":
        return [n // 4, n // 2, n]
    ratios = (1.0, 2.0 / 3.0, 1.0 / 3.0, 1.0 / 6.0)[: case["grids"]]
    ok = [m << p for m in range(1, 32, 2) for p in range(1, 13)]
    return [min((g for g in ok if g >= 16), key=lambda g: abs(g - n * r)) for r in ratios]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _kfield(n, kh, medium, seed):
    """Wavenumbers on the (n+1)^2 grid: constant; three layers k * {1, 1.5, 0.75} between tilted
    interfaces; or k (1 + 0.3 g) with g a smooth field of correlation length 0.05 and unit variance
    (random cosines), clipped to [-1, 1]."""
    k = kh * n
    x = torch.linspace(0, 1, n + 1, dtype=torch.float64, device="cuda")
    if medium == "const":
        return np.full((n + 1, n + 1), k)
    rs = np.random.RandomState(seed % (1 << 31))
    if medium == "wedge":
        s = rs.uniform(-0.5, 0.5, 2)
        y = x[:, None]
        top = y >= 2.0 / 3.0 + s[0] * (x - 0.5)
        mid = y >= 1.0 / 3.0 + s[1] * (x - 0.5)
        return (k * (0.75 + 0.25 * top.double() + 0.75 * (mid & ~top).double())).cpu().numpy()
    modes = 48
    w = torch.from_numpy(rs.normal(0.0, 20.0, (modes, 2))).cuda()
    ph = torch.from_numpy(rs.uniform(0, 2 * math.pi, modes)).cuda()
    ax, ay = x[:, None] * w[:, 0] + ph, x[:, None] * w[:, 1]
    g = math.sqrt(2.0 / modes) * (torch.cos(ay) @ torch.cos(ax).T - torch.sin(ay) @ torch.sin(ax).T)
    return (k * (1 + 0.3 * g.clamp(-1, 1))).cpu().numpy()


def _sources(n, count, seed):
    """`count` right-hand sides, each one to eight interior point sources of 1/h^2."""
    rs = np.random.RandomState((seed + 7) % (1 << 31))
    b = torch.zeros((count, n + 1, n + 1), dtype=torch.complex128, device="cuda")
    per = 8 if count == 1 else 1
    for c in range(count):
        for i, j in rs.randint(1, n, (per, 2)):
            b[c, j, i] += float(n * n)
    return b


def _waves(n, kh, seed):
    """A field of solution type: plane waves of wavenumber k in eight random directions, a little noise."""
    rs = np.random.RandomState((seed + 11) % (1 << 31))
    x = torch.linspace(0, 1, n + 1, dtype=torch.float64, device="cuda")
    u = torch.zeros((n + 1, n + 1), dtype=torch.complex128, device="cuda")
    for t, a in zip(rs.uniform(0, 2 * math.pi, 8), rs.normal(size=8)):
        ex = torch.polar(torch.ones_like(x), kh * n * math.cos(t) * x)
        ey = torch.polar(torch.ones_like(x), kh * n * math.sin(t) * x)
        u += a * ey[:, None] * ex
    return u + 1e-3 * torch.randn((n + 1, n + 1), dtype=torch.complex128, device="cuda", generator=_gen(seed))


def _inputs(case, seed):
    """(media, right-hand sides or fields) of a case, one entry per grid."""
    kind, n = case["kind"], case["n"]
    if kind == "group":
        gs = _grids(case)
        return [_kfield(g, case["kh"], "const", seed) for g in gs], [_sources(g, case["batch"], seed + q) for q, g in enumerate(gs)]
    if kind == "served":
        gs = _grids(case)
        return ([_kfield(g, case["kh"], case["medium"], seed + q) for q, g in enumerate(gs)],
                [_sources(g, 1, seed + q)[0] for q, g in enumerate(gs)])
    if kind == "cycle":  # Table 7: a unit source (here at a seeded node near the centre)
        rs = np.random.RandomState((seed + 7) % (1 << 31))
        b = torch.zeros((n + 1, n + 1), dtype=torch.complex128, device="cuda")
        i, j = (n // 2 + rs.randint(-n // 8, n // 8 + 1, 2)).tolist()
        b[j, i] = 1.0
        return [_kfield(n, case["kh"], "const", seed)], [b]
    kf = _kfield(n, case["kh"], case["medium"], seed)
    if kind == "solve":
        return [kf], [_sources(n, 1, seed)[0]]
    if kind == "vcycle":  # a residual: no smoothness to speak of
        return [kf], [torch.randn((n + 1, n + 1), dtype=torch.complex128, device="cuda", generator=_gen(seed))]
    return [kf], [_waves(n, case["kh"], seed)]


def prepare(case, seed):
    kfs, fields = _inputs(case, seed)
    opts = {"variant": case.get("variant", "hyb"), "precision": case.get("precision", "fp64")}
    probs = [hz.Problem(kf.shape[0] - 1, kf, BETA, k_ref=case["kh"] * (kf.shape[0] - 1), batch=case.get("batch", 1), **opts)
             for kf in kfs]
    st = {"case": case, "P": probs, "f": fields}
    if case["kind"] == "group":
        st["G"] = hz.Group(probs)
    if case["kind"] == "cycle":
        st["R"] = hz.Ray(probs[0], case["kh"] * case["n"])
    return st


def run(st):
    case, P, f = st["case"], st["P"], st["f"]
    kind = case["kind"]
    if kind == "solve":
        x, _, hist = P[0].solve(f[0], tol=1e-14, maxit=case["maxit"], allow_fail=True)
        return {"x": x, "history": hist}
    if kind == "group":
        xs, _ = st["G"].solve(f, tol=1e-14, maxit=case["maxit"], allow_fail=True)
        return {"x": xs}
    if kind == "served":
        xs = [torch.empty_like(b) for b in f]
        for p, b, x in zip(P, f, xs):
            p.solve_start(b, x, tol=1e-14, maxit=case["maxit"])
        waiting = list(P)
        while waiting:
            for p in list(waiting):
                if p.solve_poll():
                    p.solve_finish(allow_fail=True)
                    waiting.remove(p)
        return {"x": xs}
    if kind == "vcycle":
        return {"z": P[0].vcycle(f[0])}
    if kind == "apply":
        return {"v": P[0].apply(f[0], case["op"])}
    x, info, _ = P[0].cycle_solve(f[0], st["R"], tol=1e-7)
    return {"x": x, "cycles": info["cycles"]}


# ------------------------------------------------------------------ what a pass cannot do without


def _vcycle_work(n, e):
    """Bytes and flops of one V-cycle with e bytes per complex element: every level reads f and k h and
    writes its correction on the way down, and reads both, the correction and the coarser one and
    writes the result on the way up (the geometric sum over levels is 4/3); about 100 flops a node."""
    N = (n + 1) ** 2 * 4.0 / 3.0
    return 6.5 * e * N, 100.0 * N


def _solve_work(n, e, its):
    """Bi-CGSTAB: the five vector stages that its reductions separate (288 bytes a node in complex128,
    and the preconditioned vectors twice each) and two V-cycles per iteration; b in, x out."""
    N = (n + 1) ** 2
    vb, vf = _vcycle_work(n, e)
    return its * ((288.0 + 4 * e) * N + 2 * vb) + 32.0 * N, its * (108.0 * N + 2 * vf)


def work(case):
    kind, n = case["kind"], case["n"]
    e = 8 if case.get("precision") == "fp32" else 16
    if kind == "solve":
        b, f = _solve_work(n, e, case["maxit"])
    elif kind in ("group", "served"):
        w = [_solve_work(g, e, case["maxit"]) for g in _grids(case)]
        b, f = (case.get("batch", 1) * sum(c) for c in zip(*w))
    elif kind == "vcycle":
        b, f = _vcycle_work(n, e)
        b += 32.0 * (n + 1) ** 2 - 2.0 * e * (n + 1) ** 2 if e == 8 else 0.0
    elif kind == "apply":
        b, f = 40.0 * (n + 1) ** 2, 14.0 * (n + 1) ** 2
    else:  # ten cycles: V-cycle, two residuals, ray restriction and prolongation, block substitutions
        vb, vf = _vcycle_work(n, e)
        nr = n // 8 + 1
        blocks = 3.0 * nr * (8 * nr) ** 2  # inverse, lower and upper factor of every block row
        b = 10 * (vb + 128.0 * (n + 1) ** 2 + 16.0 * blocks)
        f = 10 * (vf + (48.0 + 16 * EIGHT) * (n + 1) ** 2 + 8.0 * blocks)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in complex128, written out
#
# Rows are scaled by H^2: (A u)_p = sum of the four neighbours + d_p u_p,
# d = -4 + (kH)^2 (1 + i beta) + 2 i s kH with s the number of sides the node lies on; a neighbour
# outside the square is its mirror node.


def _nb(u):
    u = torch.cat([u[..., 1:2], u, u[..., -2:-1]], -1)
    h = u[..., :-2] + u[..., 2:]
    c = u[..., 1:-1]
    return h + torch.cat([c[..., 1:2, :], c[..., :-1, :]], -2) + torch.cat([c[..., 1:, :], c[..., -2:-1, :]], -2)


def _nb_adjoint(d):
    o = torch.zeros_like(d)
    o[..., 1:] += d[..., :-1]
    o[..., :-1] += d[..., 1:]
    o[..., 1] += d[..., 0]
    o[..., -2] += d[..., -1]
    o[..., 1:, :] += d[..., :-1, :]
    o[..., :-1, :] += d[..., 1:, :]
    o[..., 1, :] += d[..., 0, :]
    o[..., -2, :] += d[..., -1, :]
    return o


def _diag(kH, beta):
    n = kH.shape[-1] - 1
    edge = torch.zeros(n + 1, dtype=torch.float64, device=kH.device)
    edge[0] = edge[n] = 1.0
    s = edge[:, None] + edge
    return torch.complex(kH * kH - 4.0, beta * kH * kH + 2.0 * s * kH)


def _row_norm2(d):
    n = d.shape[-1] - 1
    w = torch.full((n + 1,), 2.0, dtype=torch.float64, device=d.device)
    w[0] = w[n] = 4.0  # the mirror node's coefficient is 2
    return (d.real**2 + d.imag**2) + w[:, None] + w


def _reflect_fw(r):
    r = torch.cat([r[..., 1:2], r, r[..., -2:-1]], -1)
    r = 0.25 * (r[..., :-2:2] + r[..., 2::2]) + 0.5 * r[..., 1:-1:2]
    r = torch.cat([r[..., 1:2, :], r, r[..., -2:-1, :]], -2)
    return 0.25 * (r[..., :-2:2, :] + r[..., 2::2, :]) + 0.5 * r[..., 1:-1:2, :]


def _bilinear(e):
    m = e.shape[-1] - 1
    o = torch.empty(e.shape[:-1] + (2 * m + 1,), dtype=e.dtype, device=e.device)
    o[..., ::2] = e
    o[..., 1::2] = 0.5 * (e[..., :-1] + e[..., 1:])
    q = torch.empty(o.shape[:-2] + (2 * m + 1, 2 * m + 1), dtype=e.dtype, device=e.device)
    q[..., ::2, :] = o
    q[..., 1::2, :] = 0.5 * (o[..., :-1, :] + o[..., 1:, :])
    return q


def _levels(kf, k_ref, variant):
    """Per level: the relaxation and residual diagonals and whether it relaxes by Kaczmarz (Sec. 5)."""
    n = kf.shape[0] - 1
    k = torch.from_numpy(kf).cuda()
    out, r2 = [], math.sqrt(2.0)
    while True:
        kH = k / n
        if n % 2 or n <= 8:
            d = _diag(kH, BETA if variant in ("sl", "sl_plain") else 0.0)
            N = (n + 1) ** 2
            A = _nb(torch.eye(N, dtype=torch.complex128, device="cuda").reshape(N, n + 1, n + 1)).reshape(N, N).T
            out.append({"n": n, "A": A + torch.diag(d.reshape(-1))})
            return out
        c = k_ref / n
        band = bool(((kH >= 0.625 * r2) & (kH < 2 * r2)).any())
        kacz = band and variant != "sl_plain"
        if variant == "sl_plain" or variant == "sl":
            relax, resid = BETA, BETA
        elif variant == "hlm":
            relax, resid = 0.0, 0.0
        else:
            resid = 0.0
            shifted = 0.625 / r2 <= c < 1.25 * r2 or kacz or bool(((kH > 1.0) & (kH < 2 * r2)).any())
            relax = BETA if shifted else 0.0
        dA = _diag(kH, relax)
        j = torch.arange(n + 1, device="cuda")
        out.append({"n": n, "dA": dA, "dB": _diag(kH, resid), "kacz": kacz,
                    "norm2": _row_norm2(dA), "parity": (j[:, None] + j) % 2, "colour": (2 * j[:, None] + j) % 5})
        k, n = k[::2, ::2], n // 2


def _sweeps(L, f, u, post):
    if L["kacz"]:
        for _ in range(4):
            for c in range(5):
                m = L["colour"] == (4 - c if post else c)
                d = torch.where(m, (f - _nb(u) - L["dA"] * u) / L["norm2"], 0)
                u = u + L["dA"].conj() * d + _nb_adjoint(d)
        return u
    for c in (1, 0) if post else (0, 1):
        u = torch.where(L["parity"] == c, (f - _nb(u)) / L["dA"], u)
    return u


def _vcycle(levels, f, l=0):
    """Of the H^2-scaled right-hand side f."""
    L = levels[l]
    if "A" in L:
        N = L["A"].shape[0]
        return torch.linalg.solve(L["A"], f.reshape(-1, N).T).T.reshape(f.shape)
    u = _sweeps(L, f, torch.zeros_like(f), False)
    r = f - _nb(u) - L["dB"] * u
    u = u + _bilinear(_vcycle(levels, 4.0 * _reflect_fw(r), l + 1))
    return _sweeps(L, f, u, True)


def _shadow(N):
    """The fixed shadow residual of the iteration: SplitMix64 uniforms in [-1/2, 1/2)."""
    with np.errstate(over="ignore"):
        z = np.uint64(0x5EED1312) + np.uint64(0x9E3779B97F4A7C15) * np.arange(1, 2 * N + 1, dtype=np.uint64)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = (z >> np.uint64(11)).astype(np.float64) * 2.0**-53 - 0.5
    return torch.from_numpy(u.view(np.complex128)).cuda()


def _bicgstab(kf, k_ref, variant, b, its):
    """`its` right-preconditioned Bi-CGSTAB iterations (van der Vorst) from x = 0 for every b[c]."""
    n = kf.shape[0] - 1
    levels = _levels(kf, k_ref, variant)
    d = _diag(torch.from_numpy(kf).cuda() / n, 0.0)
    rh = _shadow((n + 1) ** 2).reshape(n + 1, n + 1)

    def dot(a, c):
        return (a.conj() * c).sum((-2, -1), keepdim=True)

    b = b.reshape(-1, n + 1, n + 1) / float(n) ** 2
    r, x, p = b, torch.zeros_like(b), b
    rho, hist, bn = dot(rh, b), [], dot(b, b).real.sqrt()
    for it in range(its):
        y = _vcycle(levels, p)
        v = _nb(y) + d * y
        alpha = rho / dot(rh, v)
        s = r - alpha * v
        hist.append(dot(s, s).real.sqrt() / bn)
        z = _vcycle(levels, s)
        t = _nb(z) + d * z
        omega = dot(t, s) / dot(t, t).real
        x = x + alpha * y + omega * z
        r = s - omega * t
        hist.append(dot(r, r).real.sqrt() / bn)
        new = dot(rh, r)
        p = r + (new / rho) * (alpha / omega) * (p - omega * v)
        rho = new
    return x, torch.stack(hist).reshape(2 * its, -1)


def _direct(kf, b):
    """L x = b by block elimination over grid rows with two steps of refinement (constant-k grids of
    a few hundred rows)."""
    n = kf.shape[0] - 1
    d = _diag(torch.from_numpy(kf).cuda() / n, 0.0)
    shift = torch.zeros((n + 1, n + 1), dtype=torch.complex128, device="cuda")
    i = torch.arange(n, device="cuda")
    shift[i, i + 1] = shift[i + 1, i] = 1.0
    shift[0, 1] = shift[n, n - 1] = 2.0
    lo = [0.0] + [1.0] * (n - 1) + [2.0]
    up = [2.0] + [1.0] * (n - 1) + [0.0]
    inv = []
    for j in range(n + 1):
        S = shift + torch.diag(d[j])
        if j:
            S = S - lo[j] * up[j - 1] * inv[-1]
        inv.append(torch.linalg.inv(S))

    def solve(f):
        y = []
        for j in range(n + 1):
            y.append(inv[j] @ (f[j] - lo[j] * y[-1] if j else f[j]))
        for j in range(n - 1, -1, -1):
            y[j] = y[j] - up[j] * (inv[j] @ y[j + 1])
        return torch.stack(y)

    f = b / float(n) ** 2
    x = solve(f)
    for _ in range(2):
        x = x + solve(f - _nb(x) - d * x)
    return x


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    variant = case.get("variant", "hyb")
    if kind == "cycle":
        # the solution of the system, which ten contracting cycles approach to the tolerance
        kfs, f = _inputs(case, seed)
        return {"x": _direct(kfs[0], f[0]), "cycles": None}
    kfs, f = _inputs(case, seed)
    if kind == "apply":
        v = _nb(f[0]) + _diag(torch.from_numpy(kfs[0]).cuda() / n, BETA if case["op"] == "M" else 0.0) * f[0]
        return {"v": v * float(n) ** 2}
    if kind == "vcycle":
        return {"z": _vcycle(_levels(kfs[0], case["kh"] * n, variant), f[0] / float(n) ** 2)}
    res = [_bicgstab(kf, case["kh"] * (kf.shape[0] - 1), variant, b, case["maxit"]) for kf, b in zip(kfs, f)]
    if kind == "solve":
        return {"x": res[0][0][0], "history": res[0][1][:, 0].cpu().numpy()}
    return {"x": [x if kind == "group" else x[0] for x, _ in res]}
