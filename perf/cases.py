"""Performance cases of the WaveZip library: what its users call, over the sizes they call it with.

listed()            the named cases
draw(rng)           one more case of the same ranges
prepare(case, seed) inputs, weights and kept buffers on the GPU
run(state)          one pass through the public entry points, and its outputs
work(case)          bytes and flops of one pass that no implementation can do without
tolerance(case)     how far another correct implementation may be off
exact(case, seed)   the outputs in 64 bits, from torch and numpy alone

A case is one call (or one forward and inverse pair) of an entry point:

  condense   one video: wz_condense (nothing kept between calls) or wz_condense_ex with the
             workspace, outputs and status word that a serving loop keeps
  batch      wz_condense_batch on V videos of equal shape, everything kept
  relevance  wz_relevance: the scores and pooled frames alone
  project    wz_project: the two-layer projector on condensed tokens
  dwt2d      wz_dwt2d followed by wz_idwt2d on its bands

The features are spatially smooth Gaussian fields that follow an AR(1) over the frames with
fresh fields at scene cuts, plus noise, as in the repository's benchmark recipe.  On top of
that every video drifts towards and away from its query over time, so that about half of its
frames are relevant, and some have 3 x 3 patches that match the query (objects).
"""

import math

import numpy as np
import torch

import paper_2607_23265_gb300 as wz

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
LAMBDA = 1.5


def _condense(name, T, H, W, D, **kw):
    case = {"name": name, "kind": "condense", "V": 1, "T": T, "H": H, "W": W, "D": D, "dtype": "bf16", "Lq": 32,
            "ratio": 0.1, "scorer": "mean", "wta": 1, "wsm": 4, "wta_levels": 1, "wsm_levels": 1, "tau": 0.0,
            "patches": 0, "kept": True}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest: a 16-frame clip in fp32 (the CUDA-core path), where launches and latency count
        _condense("clip16_14x14_f32", 16, 14, 14, 896, dtype="f32", Lq=16, ratio=0.25),
        # a short clip through the one-line call, which keeps nothing between calls
        _condense("clip16_13x13_plain", 16, 13, 13, 896, Lq=16, ratio=0.25, kept=False),
        # one request at the paper's default of 64 frames
        _condense("video64_13x13", 64, 13, 13, 3584),
        # a longer video with objects that match the query
        _condense("video128_16x16_objects", 128, 16, 16, 3584, Lq=64, patches=4),
        # the largest single video: 256 frames of 729 tokens (the benchmark's workload)
        _condense("video256_27x27", 256, 27, 27, 3584, Lq=64),
        # a serving batch of 32 videos with their own query lengths and keep ratios: the largest call
        _condense("serving32x64_13x13", 64, 13, 13, 3584, kind="batch", V=32, Lq=0, ratio=0.0),
        # the max-over-query scorer on one video ...
        _condense("maxsim_video128_16x16", 128, 16, 16, 3584, Lq=64, scorer="maxsim", patches=4),
        # ... and on a serving batch
        _condense("maxsim_serving8x64_13x13", 64, 13, 13, 3584, kind="batch", V=8, Lq=0, ratio=0.0, scorer="maxsim"),
        # two decomposition levels in both wavelet modules
        _condense("levels2_video128_16x16", 128, 16, 16, 3584, Lq=64, wta_levels=2, wsm_levels=2),
        # the scorer alone, at a width and a frame count that are no powers of two
        {"name": "relevance_video100_24x24", "kind": "relevance", "V": 1, "T": 100, "H": 24, "W": 24, "D": 1152,
         "dtype": "bf16", "Lq": 20},
        # the projector on the condensed tokens of the 256-frame video
        {"name": "project_18662x3584", "kind": "project", "B": 18662, "D": 3584, "C": 3584, "E": 3584, "bias": True},
        # the wavelet analysis of a video's maps and its inverse
        {"name": "dwt2d_video32_27x27", "kind": "dwt2d", "V": 1, "T": 32, "H": 27, "W": 27, "D": 3584,
         "dtype": "bf16", "wsm": 4, "mode": "symmetric"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _width(rng, lo, hi, step):
    """A channel count: a multiple of `step` and, now and then, of 8 only."""
    s = step if rng.random() < 0.75 else 8
    return max(s, _log_int(rng, lo, hi) // s * s)


def draw(rng):
    kind = rng.choice(["condense"] * 9 + ["batch"] * 4 + ["maxsim"] * 4 + ["relevance"] * 3 + ["project"] * 3 + ["dwt2d"] * 3)
    H = rng.randint(7, 27)
    W = H if rng.random() < 0.7 else rng.randint(7, 27)
    T = _log_int(rng, 8, 256)
    if kind == "project":
        mult = lambda: 64 * _log_int(rng, 8, 56)  # noqa: E731
        return {"kind": "project", "B": _log_int(rng, 64, 18662), "D": mult(), "C": mult(), "E": mult(),
                "bias": rng.random() < 0.7}
    if kind == "relevance":
        return {"kind": "relevance", "V": 1, "T": T, "H": H, "W": W, "D": _width(rng, 512, 3584, 64),
                "dtype": rng.choice(["bf16", "bf16", "f32"]), "Lq": _log_int(rng, 1, 128)}
    if kind == "dwt2d":
        D = _width(rng, 256, 3584, 64)
        most = max(2, 32 * 27 * 27 * 3584 // (H * W * D))
        return {"kind": "dwt2d", "V": 1, "T": min(T, most), "H": H, "W": W, "D": D,
                "dtype": rng.choice(["bf16", "f32"]), "wsm": rng.choice([1, 2, 4, 4]),
                "mode": rng.choice(["symmetric", "symmetric", "zero", "periodic"])}
    case = _condense("", T, H, W, _width(rng, 512, 3584, 64), Lq=_log_int(rng, 4, 128),
                     ratio=rng.choice([0.05, 0.1, 0.1, 0.25]), patches=rng.choice([0, 0, 4]), kept=rng.random() < 0.7)
    del case["name"]
    if kind == "batch" or (kind == "maxsim" and rng.random() < 0.5):
        T = _log_int(rng, 8, 64)
        most = max(2, 32 * 64 * 169 * 3584 // (T * H * W * case["D"]))
        case.update(kind="batch", V=min(_log_int(rng, 2, 32), most), T=T, Lq=0, ratio=0.0, kept=True)
    if kind == "maxsim":
        case.update(scorer="maxsim", D=max(64, case["D"] // 64 * 64), kept=True)
        return case
    if kind == "condense":
        extra = rng.choice(["", "", "", "f32", "f32", "levels", "wavelets", "tau"])
        if case["T"] * H * W * case["D"] > 128 * 256 * 3584 and extra in ("f32", "levels"):
            case["T"] = max(8, 128 * 256 * 3584 // (H * W * case["D"]))
        if extra:
            case["kept"] = True
        if extra == "f32":
            case["dtype"] = "f32"
        elif extra == "levels":
            case.update(wta_levels=rng.randint(1, 3), wsm_levels=rng.randint(2, 3))
        elif extra == "wavelets":
            case.update(wta=rng.choice([1, 2, 4]), wsm=rng.choice([1, 2, 6]))
        elif extra == "tau":
            case["tau"] = 0.03
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _lengths(case):
    """Query rows and keep ratios of the videos of a case (a batch's differ from video to video)."""
    V = case["V"]
    if case["kind"] != "batch":
        return [case["Lq"]], [case.get("ratio", 0.1)]
    return [8 + (37 * v) % 121 for v in range(V)], [(0.05, 0.1, 0.25)[v % 3] for v in range(V)]


def _smoothing(n, length_scale=3.0):
    radius = int(math.ceil(3 * length_scale))
    K = np.zeros((n, n))
    for y in range(n):
        for o in range(-radius, radius + 1):
            k = (y + o) % (2 * n)
            K[y, k if k < n else 2 * n - 1 - k] += math.exp(-0.5 * (o / length_scale) ** 2)
        K[y] /= np.linalg.norm(K[y])
    return torch.from_numpy(K).float()


def _inputs(case, seed):
    """features [V, T, H, W, D] and query rows [sum Lq, D], on the GPU."""
    V, T, H, W, D = (case[k] for k in "VTHWD")
    dev = torch.device("cuda")
    dt = DTYPES[case["dtype"]]
    rng = np.random.Generator(np.random.PCG64(seed))
    g = torch.Generator(device=dev).manual_seed(seed)
    Lq = _lengths(case)[0] if "Lq" in case else [1] * V
    Q = (torch.randn((sum(Lq), D), generator=g, device=dev) / math.sqrt(D)).to(dt)
    qhat = torch.stack([q.float().mean(0) for q in Q.split(Lq)])
    qhat = qhat / qhat.norm(dim=1, keepdim=True)
    kh, kw = _smoothing(H).to(dev), _smoothing(W).to(dev)
    # scene cuts, the drift towards the query, and the patches that match it
    cut = torch.zeros((T, V), dtype=torch.bool)
    for v in range(V):
        n = min(max(1, T // 20), T - 1)
        cut[torch.from_numpy(rng.choice(np.arange(1, T), size=n, replace=False)), v] = True
    phase = torch.from_numpy(rng.uniform(0, 2 * math.pi, size=(2, V))).float()
    period = torch.from_numpy(rng.uniform(0.2, 0.9, size=V)).float() * T
    t = torch.arange(T).float()[:, None]
    drift = (4 * torch.cos(2 * math.pi * t / period + phase[0]) + 2 * torch.cos(14 * math.pi * t / period + phase[1]))
    drift, cut = drift.to(dev), cut.to(dev)
    span = max(1, T // 8)
    patches = [(int(rng.integers(0, max(1, T - span + 1))), int(rng.integers(0, max(1, H - 2))),
                int(rng.integers(0, max(1, W - 2)))) for _ in range(case.get("patches", 0))]
    X = torch.empty((V, T, H, W, D), dtype=dt, device=dev)
    a = 0.95
    F = None
    for t in range(T):
        E = torch.randn((V, H, W * D), generator=g, device=dev)
        E = torch.matmul(kw, torch.matmul(kh, E).reshape(V * H, W, D)).reshape(V, H, W, D)
        if F is None:
            F = E
        else:
            F = torch.where(cut[t].view(V, 1, 1, 1), E, a * F + math.sqrt(1 - a * a) * E)
        frame = F + 0.1 * torch.randn((V, H, W, D), generator=g, device=dev)
        frame += (drift[t].view(V, 1) * qhat).view(V, 1, 1, D)
        for (t0, y0, x0) in patches:
            if t0 <= t < t0 + span:
                frame[:, y0:y0 + 3, x0:x0 + 3, :] += 2.0 * qhat.view(V, 1, 1, D)
        X[:, t] = frame.to(dt)
    return X, Q


def _weights(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, D, C, E = (case[k] for k in "BDCE")
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    p = {"tokens": rnd(B, D).bfloat16(), "w1": (rnd(C, D) / math.sqrt(D)).bfloat16(), "b1": None,
         "w2": (rnd(E, C) / math.sqrt(C)).bfloat16(), "b2": None}
    if case["bias"]:
        p["b1"], p["b2"] = 0.1 * rnd(C), 0.1 * rnd(E)
    return p


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "project":
        st.update(_weights(case, seed))
        # a program that projects request after request keeps the hidden layer's memory
        st["workspace"] = torch.empty((wz.wz_project_workspace_size(case["B"], case["C"]),), dtype=torch.uint8, device="cuda")
        return st
    X, Q = _inputs(case, seed)
    V, T, H, W, D = X.shape
    if case["kind"] != "batch":
        X = X[0]
    st.update(X=X, Q=Q)
    if case["kind"] not in ("condense", "batch") or not case["kept"]:
        return st
    Lq, ratio = _lengths(case)
    code = wz.DTYPE_BF16 if case["dtype"] == "bf16" else wz.DTYPE_F32
    new = lambda shape, dt: torch.empty(shape, dtype=dt, device="cuda")  # noqa: E731
    opts = {"relevance": case["scorer"], "wta_wavelet": case["wta"], "wsm_wavelet": case["wsm"],
            "wta_levels": case["wta_levels"], "wsm_levels": case["wsm_levels"], "tau": case["tau"],
            "device_status": torch.zeros((1,), dtype=torch.int32, device="cuda")}
    if case["kind"] == "batch":
        rows = wz.wz_batch_rows(V, T, H, W, ratio)[0]
        size = wz.wz_batch_workspace_size(V, T, H, W, D, code, ratio)
        lead = (V,)
    else:
        rows = wz.wz_budget_size(T, H, W, ratio[0])
        size = wz.wz_condense_workspace_size(T, H, W, D, code, ratio[0])
        lead = ()
    opts.update(workspace=new((size,), torch.uint8), out_tokens=new((rows, D), X.dtype),
                out_index=new((rows, 3), torch.int32), out_budgets=new(lead + (T,), torch.int32),
                out_count=new((V,), torch.int32), out_relevance=new(lead + (T, 4), torch.float32))
    st.update(opts=opts, Lq=Lq, ratio=ratio)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "project":
        return wz.wz_project(state["tokens"], state["w1"], state["b1"], state["w2"], state["b2"], workspace=state["workspace"])
    if kind == "relevance":
        return wz.wz_relevance(state["X"], state["Q"], frame_mean=True)
    if kind == "dwt2d":
        bands = wz.wz_dwt2d(state["X"], case["wsm"], case["mode"])
        return bands + (wz.wz_idwt2d(*bands, case["H"], case["W"], case["wsm"]),)
    if kind == "batch":
        out = wz.wz_condense_batch(state["X"], state["Q"], state["Lq"], state["ratio"], **state["opts"])
        return {k: out[k] for k in ("tokens", "index", "budgets", "count", "relevance")}
    if case["kept"]:
        return wz.wz_condense_ex(state["X"], state["Q"], state["ratio"][0], **state["opts"])
    tokens, index = wz.wz_condense(state["X"], state["Q"], case["ratio"])
    return {"tokens": tokens, "index": index}


def _rows(case):
    N = case["T"] * case["H"] * case["W"]
    return sum(int(math.floor(float(np.float32(r)) * N + 0.5)) for r in _lengths(case)[1])


def work(case):
    """Each input read once and each output written once; the operations that every
    implementation makes (dots, norms, sums, four-point interpolation, products)."""
    if case["kind"] == "project":
        B, D, C, E = (case[k] for k in "BDCE")
        return {"bytes": 2 * (B * D + C * D + E * C + B * E) + (4 * (C + E) if case["bias"] else 0),
                "flops": 2 * B * C * (D + E)}
    V, T, H, W, D = (case[k] for k in "VTHWD")
    esz = 2 if case["dtype"] == "bf16" else 4
    elems = V * T * H * W * D
    if case["kind"] == "dwt2d":
        F = 2 * case["wsm"]
        hp, wp = (H + F - 1) // 2, (W + F - 1) // 2
        bands = 4 * V * T * hp * wp * D
        # width pass on H rows, height pass on two planes; the inverse alike
        flops = 2 * (2 * F * 2 * V * T * H * wp * D + 2 * F * bands)
        return {"bytes": elems * esz + 2 * 4 * bands + 4 * elems, "flops": flops}
    Lq, _ = _lengths(case)
    read = elems * esz + sum(Lq) * D * esz
    if case["kind"] == "relevance":
        return {"bytes": read + 4 * V * T * (H * W + 1 + D), "flops": 5 * elems}
    rows = _rows(case)
    dots = 2 * sum(Lq) * T * H * W * D if case["scorer"] == "maxsim" else 2 * elems
    return {"bytes": read + rows * (D * esz + 12) + (V * T * 20 if case["kept"] else 0),
            "flops": dots + 3 * elems + 8 * rows * D}


def tolerance(case):
    """About four times what each path was measured to be off exact(): bf16 results are off by
    their own rounding; fp32 results by sums of a few thousand terms.  The per-frame relevance
    outputs of a bf16 call are fp32 and far inside its bound."""
    if case["kind"] == "project":
        return {"rel": 0.01, "max": 0.06}      # hidden layer and result rounded to bf16
    if case["kind"] in ("relevance", "dwt2d"):
        return {"rel": 1e-5, "max": 1e-4}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 2e-4}
    return {"rel": 7e-3, "max": 0.03}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _filters(p):
    """Daubechies filters with p vanishing moments (minimum phase), by spectral factorisation."""
    zeros = []
    if p > 1:
        for y in np.roots([math.comb(p - 1 + k, k) for k in range(p)][::-1]):
            z = np.roots([1.0, 4.0 * y - 2.0, 1.0])
            zeros.append(z[np.argmin(np.abs(z))])
    h = np.real(np.poly([-1.0] * p + zeros))
    h = h * (math.sqrt(2.0) / h.sum())
    g = np.array([(-1.0) ** k * h[2 * p - 1 - k] for k in range(2 * p)])
    return h[::-1], g[::-1], h, g


def _extend(i, n, mode):
    if 0 <= i < n:
        return i
    if mode == "zero":
        return -1
    if mode == "periodic":
        return i % n
    k = i % (2 * n)
    return k if k < n else 2 * n - 1 - k


def _matrices(n, p, mode="symmetric"):
    """Analysis (lo, hi) [n', n] and synthesis (lo, hi) [n, n'] of one level."""
    dl, dh, rl, rh = _filters(p)
    F = 2 * p
    m = (n + F - 1) // 2
    A, S = np.zeros((2, m, n)), np.zeros((2, n, m))
    for i in range(m):
        for j in range(F):
            s = _extend(2 * i + 1 - j, n, mode)
            if s >= 0:
                A[0, i, s] += dl[j]
                A[1, i, s] += dh[j]
    for k in range(n):
        for i in range(m):
            t = k + F - 2 - 2 * i
            if 0 <= t < F:
                S[0, k, i], S[1, k, i] = rl[t], rh[t]
    return A, S


def _mat(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _along_h(m, x):
    return torch.matmul(m, x.reshape(x.shape[0], x.shape[1], -1)).reshape(x.shape[0], m.shape[0], *x.shape[2:])


def _along_w(m, x):
    return torch.matmul(m, x)


def _dwt2(x, p, mode):
    Ah, _ = _matrices(x.shape[1], p, mode)
    Aw, _ = _matrices(x.shape[2], p, mode)
    lo, hi = _along_h(_mat(Ah[0]), x), _along_h(_mat(Ah[1]), x)
    return [_along_w(_mat(Aw[u]), y) for y in (lo, hi) for u in (0, 1)]


def _idwt2(bands, H, W, p):
    _, Sh = _matrices(H, p)
    _, Sw = _matrices(W, p)
    lo = _along_w(_mat(Sw[0]), bands[0]) + _along_w(_mat(Sw[1]), bands[1])
    hi = _along_w(_mat(Sw[0]), bands[2]) + _along_w(_mat(Sw[1]), bands[3])
    return _along_h(_mat(Sh[0]), lo) + _along_h(_mat(Sh[1]), hi)


def _cos(dot, nu, nv):
    den = nu * nv
    return torch.where(den > 0, dot / torch.where(den > 0, den, torch.ones_like(den)), torch.zeros_like(den))


def _scores(X, Q, scorer):
    """a [T, N], r [T] and the pooled frames [T, D] of one video (float64)."""
    rows = Q.double() if scorer == "maxsim" else Q.double().mean(0, keepdim=True)
    qn = rows.norm(dim=1)
    a, mean = [], []
    for x in X.flatten(1, 2).split(16):
        x = x.double()
        a.append(_cos(x @ rows.T, x.norm(dim=2, keepdim=True), qn).amax(2))
        mean.append(x.mean(1))
    mean = torch.cat(mean)
    r = _cos(mean @ rows.T, mean.norm(dim=1, keepdim=True), qn).amax(1)
    return torch.cat(a), r, mean


def _rectified(r, gamma, p, levels):
    A, g, kept = r, gamma, []
    for _ in range(levels):
        n = A.size
        An, S = _matrices(n, p)
        gb = np.array([0.5 * (g[_extend(2 * k, n, "symmetric")] + g[_extend(2 * k + 1, n, "symmetric")])
                       for k in range(An.shape[1])])
        kept.append((S, gb * (An[1] @ A)))
        A, g = An[0] @ A, gb
    for S, d in reversed(kept):
        A = S[0] @ A + S[1] @ d
    return A


def _budgets(w, B, N):
    """Largest remainder over max(w, 0), capped at N with the rest apportioned again."""
    n = np.full(w.size, -1, dtype=np.int64)
    if B >= w.size * N:
        return np.full(w.size, N, dtype=np.int64)
    w = np.maximum(w, 0.0)
    if not (w > 0).any():
        w = np.ones_like(w)
    left = B
    while True:
        act = (n < 0) & (w > 0)
        u = w
        if not act.any():
            act, u = n < 0, np.ones_like(w)
        idx = np.nonzero(act)[0]
        q = left * u[idx] / u[idx].sum()
        over = q > N
        if over.any():
            n[idx[over]] = N
            left -= N * int(over.sum())
            continue
        fl = np.floor(q).astype(np.int64)
        order = np.lexsort((idx, -(q - fl)))
        fl[order[:left - fl.sum()]] += 1
        n[idx] = fl
        return np.maximum(n, 0)


def _grid(n, H, W):
    h = 1
    while h * h * W < n * H:
        h += 1
    h = min(H, h)
    return h, -(-n // h)


def _source(size, out):
    """Rows i0, i1 and the weight of i1 for every output position (half-pixel centres)."""
    num = np.maximum((2 * np.arange(out) + 1) * size - out, 0)
    i0 = np.minimum(num // (2 * out), size - 1)
    w = np.where(num // (2 * out) > size - 1, 0.0, (num - i0 * 2 * out) / (2.0 * out))
    return torch.from_numpy(i0).cuda(), torch.from_numpy(np.minimum(i0 + 1, size - 1)).cuda(), torch.from_numpy(w).cuda()


def _pooled(M, h, w):
    """Adaptive average pooling of maps [F, H, W] to [F, h, w]."""
    def bins(n, m):
        P = np.zeros((m, n))
        for i in range(m):
            lo, hi = (i * n) // m, -((-(i + 1) * n) // m)
            P[i, lo:hi] = 1.0 / (hi - lo)
        return _mat(P)
    return bins(M.shape[1], h) @ M @ bins(M.shape[2], w).T


def _modulated(x, M, p, levels):
    bands, sizes = [], []
    for _ in range(levels):
        sizes.append(x.shape[1:3])
        b = _dwt2(x, p, "symmetric")
        G = (LAMBDA * _pooled(M, b[0].shape[1], b[0].shape[2]))[..., None]
        bands.append([G * y for y in b[1:]])
        x = b[0]
    for (H, W), b in zip(reversed(sizes), reversed(bands)):
        x = _idwt2([x] + b, H, W, p)
    return x


def _condensed(X, Q, ratio, case):
    """One video: tokens, index rows, budgets, count, and (r, delta, gamma, r~) per frame."""
    T, H, W, D = X.shape
    N = H * W
    a, r, mean = _scores(X, Q, case["scorer"])
    nrm = mean.norm(dim=1)
    delta = torch.zeros(T, dtype=torch.float64)
    delta[1:] = (1 - _cos((mean[1:] * mean[:-1]).sum(1), nrm[1:], nrm[:-1])).clamp(0, 2).cpu()
    delta, r = delta.numpy(), r.cpu().numpy()
    lo, hi = delta.min(), delta.max()
    gamma = (delta - lo) / (hi - lo) if hi > lo else np.zeros(T)
    keep = np.nonzero((delta >= float(np.float32(case["tau"]))) | (np.arange(T) == 0))[0]
    rt = np.full(T, np.nan)
    rt[keep] = _rectified(r[keep], gamma[keep], case["wta"], case["wta_levels"])
    B = int(math.floor(float(np.float32(ratio)) * T * N + 0.5))
    n = np.zeros(T, dtype=np.int64)
    n[keep] = _budgets(rt[keep], B, N)
    tokens = torch.zeros((B, D), dtype=torch.float64, device=X.device)
    index = np.full((B, 3), -1, dtype=np.int64)
    off = np.concatenate([[0], np.cumsum(n)])
    live = np.nonzero(n)[0]
    for part in np.array_split(live, max(1, len(live) // 24)):
        if not len(part):
            continue
        at = torch.from_numpy(part).cuda()
        m = a[at]
        lo, hi = m.amin(1, keepdim=True), m.amax(1, keepdim=True)
        m = torch.where(hi > lo, (m - lo) / (hi - lo), torch.zeros_like(m)).reshape(len(part), H, W)
        x = _modulated(X[at].double(), m, case["wsm"], case["wsm_levels"])
        for k, f in enumerate(part):
            c = int(n[f])
            h, w = _grid(c, H, W)
            y0, y1, ly = _source(H, h)
            x0, x1, lx = _source(W, w)
            ly, lx = ly[:, None, None], lx[:, None]
            rows = (1 - ly) * x[k][y0] + ly * x[k][y1]
            z = (1 - lx) * rows[:, x0] + lx * rows[:, x1]
            tokens[off[f]:off[f + 1]] = z.reshape(h * w, D)[:c]
            p = np.arange(c)
            index[off[f]:off[f + 1]] = np.stack([np.full(c, f), p // w, p % w], 1)
    return tokens, torch.from_numpy(index), torch.from_numpy(n), int(off[-1]), torch.from_numpy(np.stack([r, delta, gamma, rt], 1))


def exact(case, seed):
    if case["kind"] == "project":
        p = _weights(case, seed)
        gelu = torch.nn.functional.gelu
        b = [0.0 if p[k] is None else p[k].double() for k in ("b1", "b2")]
        w1, w2 = p["w1"].double().T, p["w2"].double().T
        return torch.cat([gelu(z.double() @ w1 + b[0]) @ w2 + b[1] for z in p["tokens"].split(4096)])
    X, Q = _inputs(case, seed)
    if case["kind"] == "relevance":
        return _scores(X[0], Q, "mean")
    if case["kind"] == "dwt2d":
        bands = _dwt2(X[0].double(), case["wsm"], case["mode"])
        return tuple(bands) + (_idwt2(bands, case["H"], case["W"], case["wsm"]),)
    Lq, ratio = _lengths(case)
    got = [_condensed(x, q, rho, case) for x, q, rho in zip(X, Q.split(Lq), ratio)]
    out = {"tokens": torch.cat([v[0] for v in got]), "index": torch.cat([v[1] for v in got])}
    if case["kept"]:
        batch = case["kind"] == "batch"
        out["budgets"] = torch.stack([v[2] for v in got]) if batch else got[0][2]
        out["count"] = torch.tensor([v[3] for v in got])
        out["relevance"] = torch.stack([v[4] for v in got]) if batch else got[0][4]
    return out
