"""The measured workloads of the library: what a program with fixed nonequispaced points has it do.

A case is one call (or one graph replay) through the Python binding on device buffers, the plan and
its weights or B_opt coefficients made beforehand, as a program that reconstructs many sample
vectors on one set of points keeps them.  Points, samples and weights are synthetic: the sampling
schemes of the paper's experiments (jittered, random, polar, golden-angle, linogram, stack of
spirals), samples and coefficients with real and imaginary part uniform in (-1, 1), compensation
weights of the size the schemes lead to.

``exact`` evaluates the exact Fourier sums (or the linear algebra that defines the result) in
float64 with plain torch.
"""
import math

import torch

import paper_2302_00414_gb300 as L

DEV = "cuda"
MODES = {"plain": L.MODE_PLAIN, "dcf": L.MODE_DCF, "bopt": L.MODE_BOPT}


def listed():
    return [
        # the smallest reconstruction: one dimension, a few hundred jittered points, float64
        {"name": "adjoint_1d_fp64", "kind": "adjoint", "d": 1, "M": 64, "Ms": 128, "N": 256, "m": 6, "prec": "fp64",
         "mode": "dcf", "points": "jitter"},
        # the smallest two-dimensional set of the batched workload, called alone
        {"name": "adjoint_2d_small", "kind": "adjoint", "d": 2, "M": 32, "Ms": 64, "N": 5117, "m": 4, "prec": "fp32",
         "mode": "dcf", "points": "random"},
        # a polar acquisition (512 angles, 256 radii) at the wider window: dense centre, points on grid nodes
        {"name": "adjoint_2d_polar", "kind": "adjoint", "d": 2, "M": 128, "Ms": 256, "N": 131072, "m": 6,
         "prec": "fp32", "mode": "dcf", "points": "polar"},
        # reconstruction to round-off: a linogram grid, float64, the window of Table 5.1's accuracy
        {"name": "adjoint_2d_fp64", "kind": "adjoint", "d": 2, "M": 256, "Ms": 512, "N": 524288, "m": 8,
         "prec": "fp64", "mode": "dcf", "points": "linogram"},
        # three dimensions: a stack of 64 spirals of 32768 points
        {"name": "adjoint_3d_spirals", "kind": "adjoint", "d": 3, "M": 64, "Ms": 128, "N": 64 * 32768, "m": 4,
         "prec": "fp32", "mode": "dcf", "points": "spirals"},
        # the throughput workload: 64 random sets of four sizes in one graph-replayed batch
        {"name": "batch_2d", "kind": "batch", "sets": 64, "M_top": 256, "m": 4, "prec": "fp32"},
        # Algorithm 4.4: the window's entries replaced by stored coefficients, streamed from memory
        {"name": "adjoint_2d_bopt", "kind": "adjoint", "d": 2, "M": 256, "Ms": 512, "N": 327677, "m": 4,
         "prec": "fp32", "mode": "bopt", "points": "random"},
        # Remark 4.6: samples from coefficients of the adjoint problem, with stored coefficients
        {"name": "inverse_adjoint_2d", "kind": "inverse", "d": 2, "M": 128, "Ms": 256, "N": 81919, "m": 4,
         "prec": "fp32", "points": "random"},
        # the forward transform: data consistency of iterative schemes, synthetic data
        {"name": "forward_2d", "kind": "forward", "d": 2, "M": 256, "Ms": 512, "N": 327679, "m": 4, "prec": "fp32",
         "points": "random"},
        {"name": "forward_3d", "kind": "forward", "d": 3, "M": 32, "Ms": 64, "N": 327673, "m": 4, "prec": "fp32",
         "points": "random"},
        # admitting a new point set: compensation weights by a capped float64 CG at degree 2M
        {"name": "weights_2d", "kind": "weights", "d": 2, "M": 128, "Ms": 256, "N": 81921, "m": 4, "prec": "fp32",
         "points": "random", "iters": 10},
        # admitting a new point set for Algorithm 4.4: one least-squares problem per grid column
        {"name": "optimize_b_2d", "kind": "optimize", "d": 2, "M": 64, "Ms": 128, "N": 66 * 66, "m": 4,
         "prec": "fp32", "points": "jitter"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _degree(rng, Ms):
    """An even degree with oversampling between 2 and 8/3; half of the draws exactly 2."""
    return Ms // 2 if rng.random() < 0.5 else 2 * rng.randint(-(-3 * Ms // 16), Ms // 4)


def draw(rng):
    kind = rng.choice(["adjoint", "adjoint", "adjoint", "adjoint", "batch", "bopt", "inverse", "forward", "forward",
                       "weights", "optimize"])
    if kind == "batch":
        return {"kind": "batch", "sets": _log(rng, 2, 64), "M_top": rng.choice([64, 128, 256]),
                "m": rng.choice([3, 4, 4, 5, 6]), "prec": "fp32"}
    if kind == "optimize":
        Ms = rng.choice([32, 64, 128])
        n = rng.randint(Ms // 2, Ms // 2 + Ms // 16)
        return {"kind": "optimize", "d": 2, "M": Ms // 2, "Ms": Ms, "N": n * n, "m": rng.choice([2, 3, 4]),
                "prec": rng.choice(["fp32", "fp64"]), "points": "jitter"}
    if kind == "weights":
        d = rng.choice([1, 2, 2, 3])
        Ms = rng.choice({1: [128, 512, 2048], 2: [64, 128, 256], 3: [32, 64]}[d])
        M = Ms // 2
        K = (2 * M) ** d
        return {"kind": "weights", "d": d, "M": M, "Ms": Ms, "N": _log(rng, K, 1.5 * K) + rng.randint(0, 31), "m": 4,
                "prec": "fp32", "points": "random", "iters": 5 if K >= 1 << 18 else rng.choice([5, 10])}
    d = 2 if kind in ("bopt", "inverse") else rng.choice([1, 2, 2, 2, 3])
    Ms = rng.choice({1: [128, 512, 2048], 2: [64, 128, 256, 512], 3: [32, 64, 128]}[d])
    M = _degree(rng, Ms)
    prec = "fp32" if rng.random() < 0.7 else "fp64"
    m = rng.choice([3, 4, 4, 5, 6] if d == 3 else [3, 4, 4, 5, 6, 8])
    if d == 3:   # largest: about the size of the listed spirals
        prec = "fp32" if Ms == 128 else prec
        m = min(m, 4) if Ms == 128 else m
        N = _log(rng, 0.2 * M ** 3, {32: 64, 64: 8, 128: 4}[Ms] * M ** 3)
    elif d == 2:
        N = _log(rng, 0.5 * M * M, (6 if prec == "fp32" else 4) * M * M)
    else:
        N = _log(rng, 2 * M, 64 * M)
    c = {"kind": "adjoint" if kind == "bopt" else kind, "d": d, "M": M, "Ms": Ms, "N": N + rng.randint(0, 31), "m": m,
         "prec": prec, "points": "random"}
    if kind in ("bopt", "inverse"):
        c["m"] = min(m, 4)
    if kind != "adjoint":
        if kind == "bopt":
            c["mode"] = "bopt"
        return c
    c["mode"] = rng.choice(["dcf", "dcf", "plain"])
    c["points"] = rng.choice({1: ["jitter", "random"], 2: ["random", "polar", "golden", "linogram"],
                              3: ["random", "spirals"]}[d])
    if c["points"] in ("polar", "golden"):       # angles x radii near the drawn count
        c["N"] = max(1, c["N"] // (2 * M)) * 2 * M
    elif c["points"] == "linogram":
        c["N"] = max(4, c["N"] // (2 * M) // 4 * 4) * 2 * M
    elif c["points"] == "spirals":
        c["N"] = max(1, c["N"] // M) * M
    return c


# ---- inputs ---------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _complex(g, *shape):
    return torch.complex(2 * _rand(g, *shape) - 1, 2 * _rand(g, *shape) - 1)


def _arange(a, b):
    return torch.arange(a, b, device=DEV, dtype=torch.float64)


def _points(c, g):
    d, M, N, kind = c["d"], c["M"], c["N"], c["points"]
    if kind == "random":
        return _rand(g, N, d) - 0.5
    if kind == "jitter":         # one point per cell of an equispaced grid, moved by up to a quarter cell
        n = round(N ** (1.0 / d))
        ax = (_arange(0, n) + 0.5) / n - 0.5
        x = torch.stack([a.reshape(-1) for a in torch.meshgrid(*[ax] * d, indexing="ij")], 1)
        return x + (_rand(g, n ** d, d) - 0.5) / (2 * n)
    if kind in ("polar", "golden"):
        R = 2 * M
        T = N // R
        r = _arange(-R // 2, R - R // 2) / R
        if kind == "polar":
            th = math.pi * _arange(-(T // 2), T - T // 2) / T
        else:
            th = torch.remainder(math.pi / 2 + _arange(0, T) * (2 * math.pi / (1 + math.sqrt(5.0))), math.pi) - math.pi / 2
        return torch.stack([(torch.cos(th)[:, None] * r).reshape(-1), (torch.sin(th)[:, None] * r).reshape(-1)], 1)
    if kind == "linogram":
        R = 2 * M
        T = N // R
        j = _arange(-R // 2, R - R // 2)[:, None] / R
        t = _arange(-(T // 4), T // 2 - T // 4)[None, :] * 4.0 / T
        a, b = (j + 0 * t).reshape(-1), (j * t).reshape(-1)
        return torch.cat([torch.stack([a, b], 1), torch.stack([-b, a], 1)])
    if kind == "spirals":        # M planes, M turns each
        per = N // M
        s = _arange(0, per)
        r, ph = s / (2.0 * per), 2 * math.pi * M * s / per
        z = (-0.5 + _arange(0, M) / M)[:, None].expand(M, per).reshape(-1)
        return torch.stack([z, (r * torch.sin(ph)).repeat(M), (r * torch.cos(ph)).repeat(M)], 1)
    raise ValueError(kind)


def _weights(c, x, g):
    """Compensation weights: the radius where the scheme is dense at its centre, else equal, both with some spread."""
    n = x.shape[0]
    w = (0.75 + 0.5 * _rand(g, n)) / n
    if c.get("points") in ("polar", "golden", "linogram", "spirals"):
        w = w * (0.01 + 4 * torch.linalg.vector_norm(x[:, -2:], dim=1))
    return torch.complex(w, 0.1 * w * (2 * _rand(g, n) - 1))


def _sigma(c):
    return (c["Ms"] - 0.5) / c["M"]      # ceil(sigma M) = Ms


def _beta(c):
    return math.pi * c["m"] * (2.0 - c["M"] / c["Ms"])


def _kb(c, delta):
    """The Kaiser-Bessel window in grid units."""
    s = 1 - (delta / c["m"]) ** 2
    return torch.where(s >= 0, torch.special.i0(_beta(c) * torch.sqrt(s.clamp(min=0))), torch.zeros_like(s))


def _wrapped_cells(c, x):
    """Base cell and fractional offset of every coordinate."""
    y = c["Ms"] * (x - torch.floor(x + 0.5))
    b = torch.floor(y)
    return b.to(torch.int64), y - b


def _coefficients(c, x, g):
    """N x (2m+2)^2 complex coefficients near the window's own entries, as optimised ones are."""
    S, m = 2 * c["m"] + 2, c["m"]
    _, u = _wrapped_cells(c, x)
    p = _kb(c, u[:, :, None] + m - _arange(0, S))
    b = p[:, 0, :, None] * p[:, 1, None, :]
    return b * (1 + 0.05 * _complex(g, *b.shape)) + 1e-3 * float(p.max()) ** 2 * _complex(g, *b.shape)


def _dtype(c):
    return torch.complex64 if c["prec"] == "fp32" else torch.complex128


def _plan(c, x):
    return L.Plan(x, c["M"], _sigma(c), c["m"], c["prec"])


def _batch_sets(case):
    """Degrees and point counts of a batch: four sizes in turn from the top down, 4 to 6 M^2 points."""
    out = []
    for i in range(case["sets"]):
        M = max(32, case["M_top"] >> (i * 7 % 4))
        out.append({"d": 2, "M": M, "Ms": 2 * M, "N": int((4 + 2 * ((i * 0.6180339887) % 1)) * M * M) + i, "m": case["m"],
                    "prec": case["prec"], "points": "random"})
    return out


def _inputs(c, seed):
    """Everything a case's call takes, before the library sees it."""
    g = _gen(seed)
    if c["kind"] == "batch":
        sets = []
        for s in _batch_sets(c):
            x = _points(s, g)
            sets.append((s, x, _weights(s, x, g), _complex(g, s["N"]).to(_dtype(s))))
        return {"sets": sets}
    x = _points(c, g)
    n = x.shape[0]
    v = {"x": x}
    if c["kind"] == "adjoint":
        v["f"] = _complex(g, n).to(_dtype(c))
        if c["mode"] == "dcf":
            v["w"] = _weights(c, x, g)
        if c["mode"] == "bopt":
            v["coef"] = _coefficients(c, x, g)
    elif c["kind"] == "inverse":
        v["coef"] = _coefficients(c, x, g)
        v["h"] = _complex(g, *[c["M"]] * c["d"]).to(_dtype(c))
    elif c["kind"] == "forward":
        v["h"] = _complex(g, *[c["M"]] * c["d"]).to(_dtype(c))
    return v


def prepare(case, seed):
    v = _inputs(case, seed)
    if case["kind"] == "batch":
        plans, fs, hs = [], [], []
        for s, x, w, f in v["sets"]:
            p = _plan(s, x)
            p.set_weights(w)
            plans.append(p)
            fs.append(f)
            hs.append(torch.empty((s["M"], s["M"]), dtype=f.dtype, device=DEV))
        return {"kind": "batch", "batch": L.Batch(plans, fs, hs, L.MODE_DCF), "out": hs, "keep": (plans, fs)}
    p = _plan(case, v["x"])
    if "w" in v:
        p.set_weights(v["w"])
    if "coef" in v:
        p.set_bopt(v["coef"])
    st = {"kind": case["kind"], "plan": p, "mode": MODES[case.get("mode", "plain")], "iters": case.get("iters"),
          "f": v.get("f"), "h": v.get("h")}
    if case["kind"] == "optimize":
        S = 2 * case["m"] + 2
        st["coef"] = torch.empty((v["x"].shape[0], S, S), dtype=torch.complex128, device=DEV)
    return st


def run(state):
    k = state["kind"]
    if k == "batch":
        state["batch"].run()
        return state["out"]
    p = state["plan"]
    if k == "adjoint":
        return p.adjoint(state["f"], mode=state["mode"])
    if k == "forward":
        return p.forward(state["h"])
    if k == "inverse":
        return p.inverse_adjoint(state["h"])
    if k == "weights":
        info = p.weights(max_iter=state["iters"], rel_tol=1e-13)
        return {"w": p.get_weights(), "iters": info["iters"], "residual_inf": info["residual_inf"]}
    residual = p.optimize_B()
    L.load().infft_get_bopt(p.handle, state["coef"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    return {"coef": state["coef"], "residual": residual}


# ---- what a pass cannot do without ----------------------------------------------------------------

def _transform_work(c, mode):
    d, M, Ms, N = c["d"], c["M"], c["Ms"], c["N"]
    r = 4 if c["prec"] == "fp32" else 8
    taps = (2 * c["m"] + 2) ** d if mode == "bopt" else (2 * c["m"] + 1) ** d
    per_point = 2 * r + (2 * r * taps if mode == "bopt" else d * r) + (2 * r if mode == "dcf" else 0)
    fl = N * taps * (8 if mode == "bopt" else 4)
    # one pruned FFT pass per axis
    fl += sum(Ms ** t * M ** (d - 1 - t) * 5 * Ms * math.log2(Ms) for t in range(d))
    return {"bytes": N * per_point + 2 * r * M ** d, "flops": fl}


def work(case):
    k = case["kind"]
    if k == "batch":
        ws = [_transform_work(s, "dcf") for s in _batch_sets(case)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    if k in ("adjoint", "forward"):
        return _transform_work(case, case.get("mode", "plain"))
    if k == "inverse":
        return _transform_work(case, "bopt")
    d, M, N, m = case["d"], case["M"], case["N"], case["m"]
    if k == "weights":
        # two float64 FFTs of period 4M per iteration, one adjoint and one forward NFFT of the points for t and w
        K, n = (2 * M) ** d, 4 * M
        fft = sum(n ** t * (2 * M) ** (d - 1 - t) * 5 * n * math.log2(n) for t in range(d))
        pts = N * ((17 if d <= 2 else 9) ** d) * 4
        return {"bytes": N * (8 * d + 16) + 16 * K, "flops": 2 * case["iters"] * fft + 2 * (pts + fft)}
    S = 2 * m + 2
    n = N * S ** d / case["Ms"] ** d            # members of a column
    return {"bytes": N * (8 * d + 16 * S ** d), "flops": case["Ms"] ** d * (4 / 3 * n ** 3 + 8 * n * n)}


# ---- the exact result in float64 -------------------------------------------------------------------

def _waves(M, x, sign):
    """exp(sign 2 pi i k x), k = -M/2 .. M/2 - 1, for the points x of one axis."""
    ph = x[:, None] * _arange(-(M // 2), M - M // 2)
    ph = 2 * math.pi * (ph - torch.round(ph))
    return torch.polar(torch.ones_like(ph), sign * ph)


def _chunks(n, M, d):
    step = max(256, min(n, (1 << 25) // max(1, M ** (d - 1))))
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _adjoint_sum(x, c, M):
    """h_k = sum_j c_j exp(-2 pi i k x_j)"""
    n, d = x.shape
    h = torch.zeros((M ** (d - 1), M), dtype=torch.complex128, device=DEV)
    for a, b in _chunks(n, M, d):
        e = c[a:b, None]
        for t in range(d - 1):
            w = _waves(M, x[a:b, t], -1)
            e = (e[:, :, None] * w[:, None, :]).reshape(b - a, -1)
        h += e.T @ _waves(M, x[a:b, d - 1], -1)
    return h.reshape([M] * d)


def _forward_sum(x, h, M):
    """f_j = sum_k h_k exp(2 pi i k x_j)"""
    n, d = x.shape
    out = []
    for a, b in _chunks(n, M, d):
        v = _waves(M, x[a:b, 0], 1) @ h.reshape(M, -1)
        for t in range(1, d):
            v = (v.reshape(b - a, M, -1) * _waves(M, x[a:b, t], 1)[:, :, None]).sum(1)
        out.append(v.reshape(-1))
    return torch.cat(out)


def _window_ft(c):
    k = _arange(-(c["M"] // 2), c["M"] - c["M"] // 2)
    s = torch.sqrt(_beta(c) ** 2 - (2 * math.pi * c["m"] * k / c["Ms"]) ** 2)   # positive for sigma >= 2
    return (2.0 * c["m"] / c["Ms"]) * torch.sinh(s) / s


def _columns(c, x):
    """Grid cell (row-major) of every point's (2m+2)^2 slots."""
    S, m, Ms = 2 * c["m"] + 2, c["m"], c["Ms"]
    b, _ = _wrapped_cells(c, x)
    s = torch.arange(S, device=DEV)
    q = torch.remainder(b[:, :, None] - m + s, Ms)
    return q[:, 0, :, None] * Ms + q[:, 1, None, :]


def _crop(c):
    return torch.remainder(torch.arange(-(c["M"] // 2), c["M"] - c["M"] // 2, device=DEV), c["Ms"])


def _exact_weights(c, x):
    """The best of the first iterates of plain CG on A^* A u = e_0 at degree 2M, w = conj(A u)."""
    M2, d = 2 * c["M"], c["d"]
    b = torch.zeros([M2] * d, dtype=torch.complex128, device=DEV)
    b[tuple([M2 // 2] * d)] = 1
    u, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rr = float((r.abs() ** 2).sum())
    best, kept = math.inf, u
    for _ in range(c["iters"]):
        q = _adjoint_sum(x, _forward_sum(x, p, M2), M2)
        al = rr / float((p.conj() * q).sum().real)
        u, r = u + al * p, r - al * q
        new = float((r.abs() ** 2).sum())
        if new < best:
            best, kept = new, u
        p = r + (new / rr) * p
        rr = new
    w = _forward_sum(x, kept, M2).conj()
    res = float((_adjoint_sum(x, w.conj(), M2) - b).abs().max())
    return {"w": w.cpu().numpy(), "iters": None, "residual_inf": res}


def _exact_optimize(c, x):
    """Column by column the solution of the normal equations of eq. opt_overdet_columnwise."""
    M, Ms, m, S = c["M"], c["Ms"], c["m"], 2 * c["m"] + 2
    n = x.shape[0]
    xw = x - torch.floor(x + 0.5)
    _, u = _wrapped_cells(c, x)
    cols = _columns(c, x).reshape(-1)
    order = torch.argsort(cols, stable=True)
    count = torch.bincount(cols, minlength=Ms * Ms)
    top = int(count.max())
    rank = torch.arange(cols.numel(), device=DEV) - (torch.cumsum(count, 0) - count)[cols[order]]
    member = torch.full((Ms * Ms, top), -1, dtype=torch.int64, device=DEV)
    member[cols[order], rank] = order
    what = _window_ft(c)
    k = _arange(-(M // 2), M - M // 2)
    y = (u[:, :, None] + m - _arange(0, S)) / Ms
    V = torch.zeros_like(y, dtype=torch.complex128)
    for i in range(M):
        V += what[i] * torch.polar(torch.ones_like(y), 2 * math.pi * k[i] * y)
    v = (V[:, 0, :, None] * V[:, 1, None, :]).reshape(-1)
    coef = torch.zeros(n * S * S, dtype=torch.complex128, device=DEV)
    rhs2 = float((what ** 2).sum()) ** 2
    worst = -math.inf
    for a in range(0, Ms * Ms, 2048):
        e = member[a:a + 2048]
        ok = e >= 0
        pt = torch.where(ok, e, 0) // (S * S)
        G = torch.ones((e.shape[0], top, top), dtype=torch.complex128, device=DEV)
        for t in range(2):
            xt = xw[:, t][pt]
            dx = xt[:, :, None] - xt[:, None, :]
            s = torch.zeros_like(G)
            for i in range(M):
                s += torch.polar(torch.ones_like(dx), 2 * math.pi * k[i] * dx)
            G = G * s
        both = ok[:, :, None] & ok[:, None, :]
        G = torch.where(both, G, torch.eye(top, dtype=G.dtype, device=DEV))
        rhs = torch.where(ok, v[torch.where(ok, e, 0)], 0)
        b = torch.cholesky_solve(rhs[:, :, None], torch.linalg.cholesky(G))[:, :, 0]
        coef[e[ok]] = b[ok]
        worst = max(worst, float((rhs2 - (b.conj() * rhs).sum(1).real).max()))
    return {"coef": coef.reshape(n, S, S), "residual": worst}


def exact(case, seed):
    v = _inputs(case, seed)
    if case["kind"] == "batch":
        return [_adjoint_sum(x, w * f, s["M"]) for s, x, w, f in v["sets"]]
    x = v["x"]
    if case["kind"] == "weights":
        return _exact_weights(case, x)
    if case["kind"] == "optimize":
        return _exact_optimize(case, x)
    if case["kind"] == "forward":
        return _forward_sum(x, v["h"].to(torch.complex128), case["M"])
    Ms = case["Ms"]
    if case["kind"] == "inverse":
        dinv = 1 / (Ms * _window_ft(case))
        i = _crop(case)
        g = torch.zeros((Ms, Ms), dtype=torch.complex128, device=DEV)
        g[i[:, None], i[None, :]] = v["h"].to(torch.complex128) * dinv[:, None] * dinv[None, :]
        g = torch.fft.ifft2(g, norm="forward").reshape(-1)
        return (v["coef"] * g[_columns(case, x)]).sum((1, 2))
    f = v["f"].to(torch.complex128)
    if case["mode"] == "bopt":
        g = torch.zeros(Ms * Ms, dtype=torch.complex128, device=DEV)
        g.index_add_(0, _columns(case, x).reshape(-1), (v["coef"].conj() * f[:, None, None]).reshape(-1))
        dinv = 1 / (Ms * _window_ft(case))
        i = _crop(case)
        return torch.fft.fft2(g.reshape(Ms, Ms))[i[:, None], i[None, :]] * dinv[:, None] * dinv[None, :]
    return _adjoint_sum(x, v["w"] * f if "w" in v else f, case["M"])
