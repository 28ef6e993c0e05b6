"""What this library is used for, as cases that can be timed and checked one by one.

A case is one call (or one short sequence of calls) of the public binding on one attention block:
the teacher pass, the candidate losses of a sensitivity score, an iteration of the scale fit with or
without the KL term, the Fisher-coupling probe, the Hutchinson trace, and the weight-side work of a
block (starting scales, codes, Omega). The blocks are the two of `workloads/` (GPT-2 small and
Mistral-7B shapes) and small generic ones that reach the other head ratios; batches run from one
short sequence to the 128 x 2048 calibration batch.

listed() and draw(rng) give cases, prepare(case, seed) the inputs, run(state) one pass, work(case)
the bytes and operations that the pass cannot do without, tolerance(case) what another correct
implementation may differ by, exact(case, seed) the same outputs in 64 bits by plain torch.
"""
import math

import torch

import paper_2609_34866_gb300 as J

#           d_model, query heads, KV heads, head_dim, RoPE theta (0: none), std of the weights
BLOCKS = {
    "gpt2": (768, 12, 12, 64, 0.0, 0.02),
    "mistral": (4096, 32, 8, 128, 10000.0, 0.015),
    "gqa2": (512, 4, 2, 128, 10000.0, 0.02),
    "gqa4_dh64": (256, 4, 1, 64, 500.0, 0.02),
    "gqa3": (1024, 12, 4, 128, 10000.0, 0.02),
}
#            Student-t degrees of freedom (0: normal), share of outlier channels, their factor
ACTIVATIONS = {
    "normal": (0, 0.0, 1.0),
    "normal_outliers": (0, 0.01, 20.0),
    "t4": (4, 0.0, 1.0),
    "t4_outliers": (4, 0.005, 30.0),
    "t4_some_outliers": (4, 0.005, 10.0),
    "t3_outliers": (3, 0.01, 20.0),
}
LAMBDA_KL = 0.1
PROBES = 4


def _case(name, kind, block, x, B, T, G, bits):
    return {"name": name, "kind": kind, "block": block, "x": x, "B": B, "T": T, "G": G, "bits": bits}


def listed():
    return [
        # an iteration of the scale fit on the smallest calibration batch: launches and latency
        _case("fit_gpt2_4x128", "fit", "gpt2", "normal", 4, 128, 128, "3"),
        # the teacher pass of a GPT-2 block, made once per block and batch
        _case("teacher_gpt2_16x1024", "teacher", "gpt2", "normal_outliers", 16, 1024, 128, ""),
        # one knapsack-scoring pass of a GPT-2 block: four widths in one call
        _case("score_gpt2_64x1024", "score", "gpt2", "normal_outliers", 64, 1024, 128, "2,3,4,8"),
        # scoring with both terms of the paper's default objective, ragged sequence length
        _case("score_kl_gpt2_16x777", "score_kl", "gpt2", "normal", 16, 777, 128, "2,3,4"),
        # one row of the 32 x 5 Mistral sensitivity table
        _case("score_mistral_32x2048", "score", "mistral", "t4_outliers", 32, 2048, 128, "2,3,4,5,8"),
        # an iteration of the scale fit on the full calibration batch: the largest call
        _case("fit_mistral_128x2048", "fit", "mistral", "t4", 128, 2048, 128, "3"),
        # the same at long context, 2 bits in groups of 64, with outlier channels
        _case("fit_mistral_16x4096", "fit", "mistral", "t4_some_outliers", 16, 4096, 64, "2"),
        # the same on a few sequences of an odd length
        _case("fit_mistral_3x1337", "fit", "mistral", "t4", 3, 1337, 128, "3"),
        # an iteration of the scale fit on the default objective (MSE + 0.1 KL)
        _case("fit_kl_mistral_8x2048", "fit_kl", "mistral", "t4", 8, 2048, 128, "3"),
        # the Fisher-coupling probe with the STE weight gradient it comes from
        _case("fisher_mistral_8x2048", "fisher", "mistral", "t4", 8, 2048, 128, "2"),
        # the Hutchinson trace of one block (sensitivity criterion)
        _case("trace_mistral_8x2048", "trace", "mistral", "t4_outliers", 8, 2048, 128, ""),
        # the weight side of one block: min-MSE warm-start scales, deployed codes, Omega scores
        _case("scales_mistral_g64", "scales", "mistral", "normal", 1, 1, 64, "2"),
    ]


KINDS = ("fit", "fit", "score", "score", "teacher", "fit_kl", "score_kl", "fisher", "trace", "scales")


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(KINDS)
        block = rng.choice(("gpt2", "gpt2", "mistral", "mistral", "gqa2", "gqa4_dh64", "gqa3"))
        T = _log_int(rng, 16, 4096)
        N = _log_int(rng, 128, 262144)
        G = rng.choice((64, 128))
        if kind in ("score", "score_kl"):
            bits = rng.choice(("2,3,4,8", "2,3,4,5,8", "3", "2,4", "2,3,4"))
        elif kind in ("teacher", "trace"):
            bits = ""
        else:
            bits = rng.choice(("2", "3", "4"))
        # gradients with the heaviest tails can leave the fp16 range, which the library reports
        heavy = ("t4", "t4_some_outliers") if kind in ("fit", "fit_kl", "fisher") else \
            ("t4", "t4_outliers", "t3_outliers")
        x = rng.choice(heavy if block == "mistral" else ("normal", "normal_outliers"))
        B = max(1, min(512, N // T))
        if kind == "scales":
            B = T = 1
        case = {"kind": kind, "block": block, "x": x, "B": B, "T": T, "G": G, "bits": bits}
        if work(case)["flops"] <= most:
            return case


# ------------------------------------------------------------------ inputs
def _shape(case):
    d, hq, hkv, dh, theta, std = BLOCKS[case["block"]]
    return d, hq, hkv, dh, theta, std, (hq + 2 * hkv) * dh


def _bits(case):
    return [int(b) for b in case["bits"].split(",")] if case["bits"] else []


def _inputs(case, seed):
    """X [B, T, d] and W [D, d] in bf16 and the fp32 scales [D, d / G] of every width."""
    d, hq, hkv, dh, theta, std, D = _shape(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)

    W = (normal(D, d) * std).to(torch.bfloat16)
    amax = W.float().reshape(D, d // case["G"], case["G"]).abs().amax(dim=2)
    # absmax scales for scores and probes; a fit is somewhere on its way around the min-MSE scales
    fitted = {2: 0.5, 3: 0.75, 4: 0.9}
    scales = []
    for b in _bits(case):
        s = amax / float((1 << (b - 1)) - 1)
        if case["kind"] in ("fit", "fit_kl"):
            s = s * (fitted[b] * (0.9 + 0.2 * torch.rand(s.shape, generator=g, device="cuda")))
        scales.append(s.contiguous())
    if case["kind"] == "scales":
        return None, W, scales
    df, frac, factor = ACTIVATIONS[case["x"]]
    perm = torch.randperm(d, generator=g, device="cuda")
    outliers = perm[:math.ceil(frac * d)] if frac else None
    X = torch.empty((case["B"], case["T"], d), dtype=torch.bfloat16, device="cuda")
    step = max(1, (1 << 25) // (case["T"] * d))
    for b0 in range(0, case["B"], step):
        shape = (min(step, case["B"] - b0), case["T"], d)
        x = normal(*shape)
        if df:  # Student-t, unit variance
            chi2 = normal(*shape) ** 2
            for _ in range(df - 1):
                chi2 += normal(*shape) ** 2
            x = x / torch.sqrt(chi2 / df) / math.sqrt(df / (df - 2.0))
        if outliers is not None:
            x[:, :, outliers] *= factor
        X[b0:b0 + shape[0]] = x.to(torch.bfloat16)
    return X, W, scales


def prepare(case, seed):
    """The calibration batch, the weights, the scales, the workspace and, where the call needs it,
    the teacher's output: what a fitting or scoring program holds when it makes the call."""
    d, hq, hkv, dh, theta, std, D = _shape(case)
    X, W, scales = _inputs(case, seed)
    kind, B, T = case["kind"], case["B"], case["T"]
    desc = J.BlockDesc(d, hq, hkv, dh, case["G"], 1 if theta else 0, float(theta), 0.0)
    s = {"kind": kind, "desc": desc, "B": B, "T": T, "X": X, "W": W, "scales": scales,
         "bits": _bits(case), "seed": int(seed)}

    def new(*shape, dtype=torch.float32):
        return torch.empty(shape, dtype=dtype, device="cuda")

    f64 = torch.float64
    if kind == "scales":
        s["ws"] = J.Workspace(desc, 1, 1, 1, False)
        s["trace"] = torch.tensor([2.5], dtype=f64, device="cuda")
        s["s0"] = new(D, d // case["G"])
        s["codes"] = new(D, d, dtype=torch.int8)
        s["c1"], s["c2"] = new(1, dtype=f64), new(1, dtype=f64)
        return s
    bwd = kind in ("fit", "fit_kl", "fisher")
    C = 2 if kind == "trace" else max(1, len(s["bits"]))
    s["ws"] = J.Workspace(desc, B, T, C, bwd)
    s["A"], s["lse"] = new(B, T, hq * dh), new(B, hq, T)
    s["loss"] = new(max(1, len(s["bits"])), dtype=f64)
    if kind == "teacher":
        s["sq"] = new(1, dtype=f64)
        return s
    J.jab_reference_forward(desc, B, T, X, W, s["A"], s["ws"], lse=s["lse"])
    if kind in ("score_kl", "fit_kl"):
        s["QKV"] = new(B, T, D, dtype=torch.float16)
        J.jab_reference_projection(desc, B, T, X, W, s["QKV"], s["ws"])
    if kind == "score":
        s["parts"] = new(C, B, hq, dtype=f64)
    if kind == "score_kl":
        s["mse"], s["kl"] = new(C, dtype=f64), new(C, dtype=f64)
    if kind == "fit_kl":
        s["kl"] = new(1, dtype=f64)
    if kind in ("fit", "fit_kl"):
        s["grad"] = new(D, d // case["G"])
    if kind == "fit":  # the batch stays the same over the fit: converted once
        J.jab_prepare_x(desc, B, T, X, s["ws"])
    if kind == "fisher":
        s["grad"], s["sq"] = new(D, d), new(1, dtype=f64)
    if kind == "trace":
        s["trace"], s["vhv"] = new(1, dtype=f64), new(PROBES, dtype=f64)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    kind, desc, B, T, X, W = s["kind"], s["desc"], s["B"], s["T"], s["X"], s["W"]
    if kind == "scales":
        b = s["bits"][0]
        J.jab_init_scales(desc, b, 1, W, s["s0"])
        J.jab_quantize(desc, b, W, s["s0"], codes=s["codes"])
        J.jab_omega_scores(desc, W, [b], [s["s0"]], s["trace"], 3, s["c1"], s["ws"], c2=s["c2"])
        return {"scales": s["s0"], "codes": s["codes"], "c1": s["c1"], "c2": s["c2"]}
    ws, A = s["ws"], s["A"]
    if kind == "teacher":
        J.jab_reference_forward(desc, B, T, X, W, A, ws, lse=s["lse"], a_sqnorm=s["sq"])
        return {"A": A, "lse": s["lse"], "sq": s["sq"]}
    if kind == "score":
        J.jab_loss_forward(desc, B, T, X, W, A, s["bits"], s["scales"], s["loss"], ws,
                           sse_parts=s["parts"])
        return {"loss": s["loss"], "parts": s["parts"]}
    if kind == "score_kl":
        J.jab_loss_forward_kl(desc, B, T, X, W, A, s["QKV"], s["bits"], s["scales"], LAMBDA_KL,
                              s["loss"], ws, mse=s["mse"], kl=s["kl"])
        return {"loss": s["loss"], "mse": s["mse"], "kl": s["kl"]}
    if kind == "fit":
        J.jab_loss_backward_scales_prepared(desc, B, T, X, W, A, s["bits"][0], s["scales"][0], 0.0,
                                            s["loss"], s["grad"], ws)
        return {"loss": s["loss"], "grad": s["grad"]}
    if kind == "fit_kl":
        J.jab_loss_backward_scales_kl(desc, B, T, X, W, A, s["QKV"], s["lse"], s["bits"][0],
                                      s["scales"][0], 0.0, LAMBDA_KL, s["loss"], s["grad"], ws,
                                      kl=s["kl"])
        return {"loss": s["loss"], "kl": s["kl"], "grad": s["grad"]}
    if kind == "fisher":
        J.jab_loss_backward_weights(desc, B, T, X, W, A, s["bits"][0], s["scales"][0], s["loss"],
                                    grad_w=s["grad"], grad_sqnorm=s["sq"], ws=ws)
        return {"loss": s["loss"], "grad": s["grad"], "sq": s["sq"]}
    if kind == "trace":
        J.jab_hutchinson_trace(desc, B, T, X, W, A, s["lse"], PROBES, s["seed"], s["trace"], ws,
                               vhv=s["vhv"])
        return {"trace": s["trace"], "vhv": s["vhv"]}
    raise ValueError(kind)


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    d, hq, hkv, dh, theta, std, D = _shape(case)
    kind, B, T = case["kind"], case["B"], case["T"]
    N, C, ng = B * T, max(1, len(_bits(case))), d // case["G"]
    if kind == "scales":  # W in; scales and codes out; 80 trial scales of about five operations each
        return {"bytes": D * d * (2 + 1) + 4 * D * ng, "flops": 80 * 5 * D * d}
    proj = 2.0 * N * D * d                       # X W^T, and as much for dQKV^T X
    attn = 4.0 * B * hq * dh * T * (T + 1) / 2   # Q K^T and P V over the visible keys
    nbytes = 2 * N * d + 2 * D * d               # X, W
    if kind == "teacher":
        return {"bytes": nbytes + 4 * N * hq * dh + 4 * B * hq * T, "flops": proj + attn}
    if kind == "trace":                          # five products per probe: S, two halves of dS, dO's two
        return {"bytes": nbytes + 4 * N * hq * dh,
                "flops": proj + PROBES * (proj + 2.5 * attn)}
    nbytes += 4 * N * hq * dh + C * 4 * D * ng   # A_ref, scales
    if kind == "score":
        return {"bytes": nbytes, "flops": C * (proj + attn)}
    if kind == "score_kl":                       # the student's and the teacher's scores again
        return {"bytes": nbytes + 2 * N * (hq + hkv) * dh, "flops": C * (proj + 1.5 * attn)}
    flops = 2 * proj + 3.5 * attn                # forward, and the backward's five products
    if kind == "fisher":
        return {"bytes": nbytes + 4 * D * d, "flops": flops}
    if kind == "fit_kl":                         # the teacher's scores once more
        return {"bytes": nbytes + 4 * D * ng + 2 * N * (hq + hkv) * dh, "flops": flops + 0.5 * attn}
    return {"bytes": nbytes + 4 * D * ng, "flops": flops}


def tolerance(case):
    """About four times the largest distance from exact() seen over the listed and a hundred drawn
    cases (fp16 operands, bf16 for dQKV): as far as another correct order of the same roundings may
    be off. The scales are argmins, the codes whole numbers: equal but for ties."""
    return {"teacher": {"rel": 3e-3, "max": 0.15}, "score": {"rel": 2e-3, "max": 0.06},
            "score_kl": {"rel": 1e-3, "max": 0.02}, "fit": {"rel": 1.6e-2, "max": 0.5},
            "fit_kl": {"rel": 1.6e-2, "max": 0.5}, "fisher": {"rel": 1.4e-2, "max": 0.4},
            "trace": {"rel": 3e-3, "max": 0.01},
            "scales": {"rel": 1e-5, "max": 0.02, "differ": 1e-5}}[case["kind"]]


# ------------------------------------------------------------------ the same in 64 bits
def _quantize(W, s, b, G):
    """w_hat (64 bits) and the LSQ factor d w_hat / d s; the quotient is the 32-bit one."""
    D, d = W.shape
    qmax = float((1 << (b - 1)) - 1)
    v = W.float().reshape(D, d // G, G) / s[:, :, None]
    q = torch.clamp(torch.round(v), -qmax, qmax)
    r = torch.where(v.abs() <= qmax, q - v, torch.sign(v) * qmax)
    w_hat = q.double() * s.double()[:, :, None]
    return w_hat.reshape(D, d), r.double().reshape(D, d), q.reshape(D, d)


def _rope(x, T, dh, theta, back=False):
    """Rotate-half RoPE of [T, heads, dh] (or its transpose)."""
    half = dh // 2
    inv = theta ** (-2.0 * torch.arange(half, device="cuda", dtype=torch.float64) / dh)
    phi = torch.arange(T, device="cuda", dtype=torch.float64)[:, None] * inv[None, :]
    c, s = torch.cos(phi)[:, None, :], torch.sin(phi)[:, None, :]
    if back:
        s = -s
    x1, x2 = x[..., :half], x[..., half:]
    return torch.cat([x1 * c - x2 * s, x2 * c + x1 * s], dim=-1)


def _qkv(case, x, w):
    """Heads of one sequence: Q [hq, T, dh], K and V [hkv, T, dh], rotated."""
    d, hq, hkv, dh, theta, std, D = _shape(case)
    T = x.shape[0]
    y = (x @ w.T).reshape(T, hq + 2 * hkv, dh)
    q, k, v = y[:, :hq], y[:, hq:hq + hkv], y[:, hq + hkv:]
    if theta:
        q, k = _rope(q, T, dh, theta), _rope(k, T, dh, theta)
    return q.transpose(0, 1), k.transpose(0, 1), v.transpose(0, 1)


def _probs(q, k, mask, dh):
    """Scores and attention map of one KV group: q [r, T, dh], k [T, dh]."""
    s = (q @ k.T) / math.sqrt(dh)
    s.masked_fill_(mask, -math.inf)
    lse = torch.logsumexp(s, dim=2)
    return s, lse, torch.exp(s - lse[:, :, None])


def _kl(pt, st, lt, ss, ls, mask):
    t = torch.where(mask, torch.zeros_like(pt), pt * ((st - lt[:, :, None]) - (ss - ls[:, :, None])))
    return t.sum()


def _splitmix_signs(seed, first, n):
    """Signs of outputs first + 1 .. first + n of SplitMix64 seeded with `seed`."""
    def signed(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    def lsr(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    i = torch.arange(first + 1, first + n + 1, device="cuda", dtype=torch.int64)
    z = i * signed(0x9E3779B97F4A7C15) + int(seed)
    z = (z ^ lsr(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ lsr(z, 27)) * signed(0x94D049BB133111EB)
    z = z ^ lsr(z, 31)
    return torch.where(z < 0, -1.0, 1.0).double()


def _exact_flops(case):
    d, hq, hkv, dh, theta, std, D = _shape(case)
    kind, B, T = case["kind"], case["B"], case["T"]
    C = len(_bits(case))
    proj, prod = 2.0 * B * T * D * d, 2.0 * B * hq * dh * T * T  # products are not triangular here
    n_proj, n_prod = {"teacher": (1, 2), "score": (1 + C, 2 + 2 * C), "score_kl": (1 + C, 2 + 2 * C),
                      "fit": (3, 8), "fit_kl": (3, 8), "fisher": (3, 8),
                      "trace": (1 + PROBES, 2 + 5 * PROBES)}[kind]
    return n_proj * proj + n_prod * (prod + 40.0 * B * hq * T * T) + 3e8 * B * hkv * (1 + C)


def exact(case, seed):
    d, hq, hkv, dh, theta, std, D = _shape(case)
    kind, B, T, G = case["kind"], case["B"], case["T"], case["G"]
    if kind != "scales" and _exact_flops(case) > 1.5e13:
        return None
    X, W, scales = _inputs(case, seed)
    bits = _bits(case)
    if kind == "scales":
        return _exact_scales(W, bits[0], G)
    r, n = hq // hkv, float(B) * T * hq * dh
    W64 = W.double()
    mask = torch.ones((T, T), dtype=torch.bool, device="cuda").triu(1)
    quant = [_quantize(W, s, b, G) for s, b in zip(scales, bits)]
    f64 = {"dtype": torch.float64, "device": "cuda"}
    A_all = torch.empty((B, T, hq * dh), **f64) if kind == "teacher" else None
    lse_all = torch.empty((B, hq, T), **f64)
    parts, kls = torch.zeros((max(1, len(bits)), B, hq), **f64), torch.zeros(max(1, len(bits)), **f64)
    sq = torch.zeros(1, **f64)
    gw = torch.zeros((D, d), **f64) if kind in ("fit", "fit_kl", "fisher") else None
    vhv = torch.zeros(PROBES, **f64)
    probes = [_splitmix_signs(seed, i * D * d, D * d).reshape(D, d)
              for i in range(PROBES if kind == "trace" else 0)]
    for b in range(B):
        x = X[b].double()
        qt, kt, vt = _qkv(case, x, W64)
        tangents = [_qkv(case, x, p) for p in probes]
        students = [_qkv(case, x, w_hat) for w_hat, _, _ in quant]
        dq, dk, dv = ((torch.zeros_like(t) for t in students[0]) if gw is not None else (None,) * 3)
        for g in range(hkv):
            hs = slice(g * r, g * r + r)
            st, lt, pt = _probs(qt[hs], kt[g], mask, dh)
            A = pt @ vt[g]
            lse_all[b, hs] = lt
            sq += (A ** 2).sum()
            if A_all is not None:
                A_all[b].reshape(T, hq, dh)[:, hs] = A.transpose(0, 1)
            for i, (dqt, dkt, dvt) in enumerate(tangents):
                ds = (dqt[hs] @ kt[g].T + qt[hs] @ dkt[g].T) / math.sqrt(dh)
                u = pt * ds
                do = u @ vt[g] + pt @ dvt[g] - u.sum(dim=2, keepdim=True) * A
                vhv[i] += 2.0 * (do ** 2).sum() / n
            for c, (q, k, v) in enumerate(students):
                ss, ls, ps = _probs(q[hs], k[g], mask, dh)
                o = ps @ v[g]
                e = o - A
                parts[c, b, hs] = (e ** 2).sum(dim=(1, 2))
                if kind in ("score_kl", "fit_kl"):
                    kls[c] += _kl(pt, st, lt, ss, ls, mask) / B
                if gw is not None:
                    do = e * (2.0 / n)
                    dp = do @ v[g].T
                    dss = ps * (dp - (do * o).sum(dim=2, keepdim=True))
                    if kind == "fit_kl":
                        dss += (LAMBDA_KL / B) * (ps - pt)
                    dq[hs] = dss @ k[g] / math.sqrt(dh)
                    dk[g] = torch.einsum("rij,rid->jd", dss, q[hs]) / math.sqrt(dh)
                    dv[g] = torch.einsum("rij,rid->jd", ps, do)
        if gw is not None:
            dq, dk, dv = dq.transpose(0, 1), dk.transpose(0, 1), dv.transpose(0, 1)
            if theta:
                dq, dk = _rope(dq, T, dh, theta, True), _rope(dk, T, dh, theta, True)
            gw += torch.cat([dq, dk, dv], dim=1).reshape(T, D).T @ x
    loss = parts.sum(dim=(1, 2)) / n
    if kind == "teacher":
        return {"A": A_all, "lse": lse_all, "sq": sq}
    if kind == "score":
        return {"loss": loss, "parts": parts}
    if kind == "score_kl":
        return {"loss": loss + LAMBDA_KL * kls, "mse": loss, "kl": kls}
    if kind == "trace":
        return {"trace": vhv.mean().reshape(1), "vhv": vhv}
    if kind == "fisher":
        return {"loss": loss, "grad": gw, "sq": (gw ** 2).sum().reshape(1)}
    kappa = 1.0 / math.sqrt(G * float((1 << (bits[0] - 1)) - 1))
    grad = kappa * (gw * quant[0][1]).reshape(D, d // G, G).sum(dim=2)
    if kind == "fit_kl":
        return {"loss": loss + LAMBDA_KL * kls, "kl": kls, "grad": grad}
    return {"loss": loss, "grad": grad}


def _exact_scales(W, b, G):
    D, d = W.shape
    qmax = float((1 << (b - 1)) - 1)
    w = W.float().reshape(D, d // G, G)
    amax = w.abs().amax(dim=2)
    s0 = torch.where(amax > 0, amax / torch.full_like(amax, qmax), torch.ones_like(amax))
    best, best_err = s0.clone(), torch.full(s0.shape, math.inf, dtype=torch.float64, device="cuda")
    for k in range(80):
        s = (s0.double() * float(100 - k) / 100.0).float()
        q = torch.clamp(torch.round(w / s[:, :, None]), -qmax, qmax)
        err = ((q.double() * s.double()[:, :, None] - w.double()) ** 2).sum(dim=2)
        better = (err < best_err) & (amax > 0)
        best, best_err = torch.where(better, s, best), torch.where(better, err, best_err)
    w_hat, _, q = _quantize(W, best, b, G)
    c1 = 2.5 * ((w_hat - W.double()) ** 2).sum().reshape(1)
    return {"scales": best, "codes": q.to(torch.int8), "c1": c1, "c2": 3.0 * c1}
