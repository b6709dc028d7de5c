"""Performance cases: the calls a serving process or a calibration job makes into the library, through the public
binding, with inputs drawn on the GPU from a seed.

Online, once per prefill: lukv_compress (uniform batches, batches of different lengths, the KeyDiff metric) and the
deployment mode (profile lookup, scoring, selection and gather with the caller's own buffers).  Offline, once per model:
oracle importance, utility curves, the profile build and the exact solver that cross-checks the relaxation.
"""
import math

import torch

from paper_2602_08585_b200 import lukv

DTYPES = {"bf16": torch.bfloat16, "fp32": torch.float32}


# ---- the cases --------------------------------------------------------------------------------

def listed():
    return [
        # A toy-sized call (one layer, 1k tokens, fp32, head size 64): nothing but launches and latencies.
        dict(name="compress_tiny_1k", kind="compress", S=1, L=1, H=4, G=1, d=64, T=1024, w=16, kp=7, dtype="fp32", P=65,
             keep=0.2, keep_odd=0.2, needles=8, channels="none", n_sink=0, min_keep=0.0),
        # One layer of an 8B-class model at 8k, as a layer-by-layer prefill calls it.
        dict(name="compress_layer_8k", kind="compress", S=1, L=1, H=8, G=4, d=128, T=8192, w=32, kp=7, dtype="bf16",
             P=129, keep=0.2, keep_odd=0.2, needles=64, channels="x8", n_sink=0, min_keep=0.0),
        # The benchmark's configuration: the whole 8B-class cache at 32k in one call.
        dict(name="compress_model_32k", kind="compress", S=1, L=32, H=8, G=4, d=128, T=32768, w=32, kp=7, dtype="bf16",
             P=257, keep=0.2, keep_odd=0.2, needles=64, channels="x8", n_sink=0, min_keep=0.0),
        # A serving batch: eight sequences of 16k, a wider window, light and heavy compression side by side.
        dict(name="compress_batch_16k", kind="compress", S=8, L=32, H=8, G=4, d=128, T=16384, w=64, kp=5, dtype="bf16",
             P=257, keep=0.1, keep_odd=0.5, needles=64, channels="x8", n_sink=0, min_keep=0.0),
        # Long documents: 128k tokens, seven query heads per KV head, heavy-tailed key channels.
        dict(name="compress_model_128k", kind="compress", S=1, L=28, H=4, G=7, d=128, T=131072, w=32, kp=7, dtype="bf16",
             P=513, keep=0.1, keep_odd=0.1, needles=256, channels="t3", n_sink=0, min_keep=0.0),
        # A deployed batch of requests of eight different lengths, with attention sinks and a minimum retention.
        dict(name="ragged_batch", kind="ragged", S=8, L=16, H=8, G=4, d=128, T=16000, w=32, kp=7, dtype="bf16", P=126,
             lens="16000,7625,11875,3500,14125,5250,9875,1750", keep=0.2, keep_odd=0.2, needles=32, channels="x8",
             n_sink=4, min_keep=0.01),
        # The second proxy metric (keys only, window of one) over the 32k cache.
        dict(name="keydiff_model_32k", kind="keydiff", S=1, L=32, H=8, d=128, T=32768, dtype="bf16", P=257, keep=0.2,
             keep_odd=0.2, channels="x8", n_sink=0, min_keep=0.0),
        # The deployment mode with a stored profile: head size 64, an odd context length, sinks.
        dict(name="online_model_20k", kind="online", S=1, L=16, H=8, G=4, d=64, T=20011, w=32, kp=7, dtype="bf16",
             sigma=0.75, needles=32, channels="x8", n_sink=4),
        # Calibration: the profile from 30 queries' curves at token resolution (a context of 4,000 tokens, 256 heads).
        dict(name="profile_build_4k", kind="profile", Q=30, N=256, T=4000, w=32, P=4001, R=99),
        # Calibration: oracle importance of one query (64 decode steps, model width 4096).
        dict(name="importance_4k", kind="importance", S=1, L=32, H=8, G=4, d=128, T=4000, w=32, dtype="bf16", steps=64,
             width=4096, decode_keys=True, normalize=True),
        # Calibration: utility curves of the proxy ranking for all 30 queries.
        dict(name="curves_4k", kind="curves", Q=30, N=256, T=4000, w=32, P=4001, n_sink=0),
        # Cross-check of the relaxation: the exact solver on one query's curves.
        dict(name="exact_4k", kind="exact", N=256, T=4000, w=32, keep=0.3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cache_sizes(rng, lo_T, hi_T, rows_max):
    """(S, L, H, T, P) with S*L*H*T <= rows_max; T is a multiple of P - 1 and rarely a power of two."""
    S = rng.choice([1, 1, 1, 2, 3, 4, 8])
    L = _log_int(rng, 1, 32)
    H = rng.choice([2, 4, 8, 8])
    T = min(_log_int(rng, lo_T, hi_T), rows_max // H)
    seg_count = rng.choice([32, 50, 64, 100, 125, 128, 200, 256, 500, 512])
    T = max(1, T // seg_count) * seg_count
    T = max(T, lo_T // seg_count * seg_count + seg_count)
    L = max(1, min(L, rows_max // (H * T)))
    S = max(1, min(S, rows_max // (L * H * T)))
    return S, L, H, T, seg_count + 1


def draw(rng):
    kind = rng.choice(["compress"] * 5 + ["ragged", "keydiff", "online", "profile", "importance", "curves", "exact"])
    dtype = rng.choice(["bf16"] * 4 + ["fp32"])
    d = rng.choice([128, 128, 128, 64])
    keep = round(math.exp(rng.uniform(math.log(0.05), math.log(0.5))), 3)
    keep_odd = rng.choice([keep, min(0.6, round(2 * keep, 3))])
    if kind in ("compress", "ragged", "online"):
        # the FP32 scores of a batch cost an order of magnitude more per key: smaller caches there
        rows = (1 << 20) if dtype == "fp32" else (1 << 24)
        S, L, H, T, P = _cache_sizes(rng, 1024, 131072 if kind != "ragged" else 32768, rows)
        w, G = rng.choice([(16, 1), (16, 4), (32, 1), (32, 2), (32, 4), (32, 4), (32, 7), (32, 8), (64, 4)])
        sinks = rng.choice([(0, 0.0), (4, 0.01)])
        c = dict(kind=kind, S=S, L=L, H=H, G=G, d=d, T=T, w=w, kp=rng.choice([5, 7, 7]), dtype=dtype, needles=32,
                 channels=rng.choice(["x8", "x8", "t3"]), n_sink=sinks[0])
        if kind == "online":
            c["T"] = T + rng.randrange(0, 16)  # any length: nothing here depends on the curve grid
            c["sigma"] = round(1.0 - keep, 3)
            return c
        c.update(P=P, keep=keep, keep_odd=keep_odd, min_keep=sinks[1])
        if kind == "ragged":
            c["S"] = S = rng.randrange(2, 9)
            c["L"] = max(1, min(L, rows // (S * H * T)))
            seg = P - 1
            c["lens"] = ",".join(str(seg * rng.randrange(max(1, -(-512 // seg)), T // seg + 1)) for _ in range(S))
        return c
    if kind == "keydiff":
        S, L, H, T, P = _cache_sizes(rng, 1024, 131072, (1 << 23) // (2 if dtype == "fp32" else 1))
        return dict(kind=kind, S=S, L=L, H=H, d=d, T=T, dtype=dtype, P=P, keep=keep, keep_odd=keep_odd,
                    channels=rng.choice(["x8", "t3"]), n_sink=0, min_keep=0.0)
    N = 8 * _log_int(rng, 2, 32)
    T = _log_int(rng, 500, 4000)
    if kind == "profile":
        return dict(kind=kind, Q=_log_int(rng, 4, 30), N=N, T=T, w=rng.choice([16, 32, 64]), P=T + 1,
                    R=rng.choice([19, 49, 99]))
    if kind == "curves":
        if rng.random() < 0.25:  # a longer context on a coarser grid
            seg = rng.choice([4, 5, 8])
            return dict(kind=kind, Q=4, N=N, T=seg * _log_int(rng, 1000, 2500), w=32, P=0, seg=seg, n_sink=4)
        return dict(kind=kind, Q=_log_int(rng, 4, 30), N=N, T=T, w=rng.choice([16, 32, 64]), P=T + 1,
                    n_sink=rng.choice([0, 4]))
    if kind == "exact":
        return dict(kind=kind, N=N, T=T, w=rng.choice([16, 32, 64]), keep=keep)
    # importance: the FP32 inputs of a small model, or bf16 inputs up to the listed size
    G = rng.choice([1, 4, 4, 7])
    L, H = (2, 4) if dtype == "fp32" else (_log_int(rng, 2, 32), rng.choice([4, 8]))
    return dict(kind=kind, S=1, L=L, H=H, G=G, d=d, T=min(T, 2000) if dtype == "fp32" or G == 7 else T, w=32, dtype=dtype,
                steps=_log_int(rng, 8, 64), width=rng.choice([1024, 2048, 3584, 4096]) if dtype == "bf16" else 1024,
                decode_keys=rng.random() < 0.7, normalize=rng.random() < 0.7)


# ---- inputs -------------------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _normal(shape, dtype, g):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(generator=g)


def _student_t3(shape, g):
    z = _normal(shape, torch.float32, g)
    chi = sum(_normal(shape, torch.float32, g).square_() for _ in range(3))
    return z / (chi / 3).sqrt_()


def _cache(c, g):
    """q_win [S][L][H*G][w][d], k, v [S][L][H][T][d]: unit normals, four outlier channels per KV head (shared by its query
    heads), needle keys aligned with the window's mean query."""
    S, L, H, T, d = c["S"], c["L"], c["H"], c["T"], c["d"]
    G, w = c.get("G", 1), c.get("w", 1)
    dt = DTYPES[c["dtype"]]
    heads = S * L * H
    q = _normal((heads, G * w, d), dt, g)
    k = _normal((heads, T, d), dt, g)
    v = _normal((heads, T, d), dt, g)
    if c["channels"] != "none":
        ch = torch.rand((heads, d), generator=g, device="cuda").topk(4, dim=1).indices
        gain = torch.ones((heads, 1, d), device="cuda").scatter_(2, ch[:, None, :], 8.0)
        q.mul_(gain.to(dt))
        if c["channels"] == "x8":
            k.mul_(gain.to(dt))
        else:
            k.scatter_(2, ch[:, None, :].expand(heads, T, 4), _student_t3((heads, T, 4), g).to(dt))
    needles = c.get("needles", 0)
    if needles:
        each = (T - w) // needles  # one needle in each of `needles` stretches: no position twice
        pos = torch.randint(0, each, (heads, needles), generator=g, device="cuda")
        pos += each * torch.arange(needles, device="cuda")
        rows = 3.0 * q.float().mean(dim=1, keepdim=True) + 0.1 * _normal((heads, needles, d), torch.float32, g)
        k[torch.arange(heads, device="cuda")[:, None], pos] = rows.to(dt)
    return q.view(S, L, H * G, w, d), k.view(S, L, H, T, d), v.view(S, L, H, T, d)


def _curves(N, P, g):
    """Utility-versus-budget curves [N][P]: Exp(1) increments, one in five scaled x3 (non-concave)."""
    inc = torch.empty((N, P - 1), dtype=torch.float64, device="cuda").exponential_(generator=g)
    inc *= torch.where(torch.rand((N, P - 1), generator=g, device="cuda") < 0.2, 3.0, 1.0)
    out = torch.zeros((N, P), dtype=torch.float32, device="cuda")
    out[:, 1:] = inc.cumsum(dim=1).float()
    return out


def _calibration_curves(Q, N, P, T, g):
    """Curves [Q][N][P] of Q calibration queries: each head has its own decay and scale, shared by the queries."""
    r = torch.rand((2, N), generator=g, device="cuda", dtype=torch.float64)
    k = torch.arange(1, P, device="cuda", dtype=torch.float64) * (T // (P - 1))
    trend = 0.25 * 16.0 ** r[1][:, None] * k[None, :] ** -(0.2 + 1.4 * r[0][:, None])
    out = torch.zeros((Q, N, P), dtype=torch.float32, device="cuda")
    for i in range(Q):
        inc = torch.empty((N, P - 1), dtype=torch.float64, device="cuda").exponential_(generator=g)
        out[i, :, 1:] = (inc * trend).cumsum(dim=1).float()
    return out


def _lens(c):
    return [int(x) for x in c["lens"].split(",")]


def _budgets(c):
    N, w, keeps = c["L"] * c["H"], c.get("w", 1), (c["keep"], c["keep_odd"])
    lens = _lens(c) if c["kind"] == "ragged" else [c["T"]] * c["S"]
    floors = [math.ceil(c["min_keep"] * (t - w)) + 1 if c["min_keep"] else 0 for t in lens]
    return [min(N * (t - w), max(N * f, int(keeps[i % 2] * N * t))) for i, (t, f) in enumerate(zip(lens, floors))]


def _online_rows(c):
    """Rows the deployment mode can produce: at most (1 - sigma) * n per head on average, plus the window."""
    N, n = c["L"] * c["H"], c["T"] - c["w"]
    return c["S"] * (int((1.0 - c["sigma"]) * N * n) + N + N * c["w"])


def _bytes(t):
    return torch.empty(int(t), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    c, g, kind = case, _generator(seed), case["kind"]
    s = {"kind": kind}
    if kind in ("compress", "ragged", "keydiff"):
        s["q"], s["k"], s["v"] = _cache(c, g)
        N = c["L"] * c["H"]
        flags = lukv.FLAG_KEYDIFF if kind == "keydiff" else 0
        s["p"] = lukv.make_params(c["S"], c["L"], c["H"], c.get("G", 1), c["d"], c["T"], c.get("w", 1), c.get("kp", 1),
                                  c["dtype"], c["P"], n_sink=c["n_sink"], min_keep=c["min_keep"], flags=flags)
        if kind == "keydiff":
            s["q"] = None
        s["curves"] = _curves(N, c["P"], g)
        s["budgets"] = _budgets(c)
        s["lens"] = _lens(c) if kind == "ragged" else None
        s["ws"] = lukv.alloc_workspace(s["p"])
        s["out"] = lukv.Outputs(s["p"], s["budgets"])
    elif kind == "online":
        s["q"], s["k"], s["v"] = _cache(c, g)
        N = c["L"] * c["H"]
        p = s["p"] = lukv.make_params(c["S"], c["L"], c["H"], c["G"], c["d"], c["T"], c["w"], c["kp"], c["dtype"], 2,
                                      n_sink=c["n_sink"])
        # a stored profile: every head leans to keep more or less than the target, the mean is the target
        s["ratios"] = [i / 100.0 for i in range(1, 100)]
        rho = torch.tensor(s["ratios"], dtype=torch.float64, device="cuda")[:, None]
        lean = torch.rand((N,), generator=g, device="cuda", dtype=torch.float64) * 1.2 - 0.6
        s["profile"] = (rho + (lean - lean.mean())[None, :] * rho * (1 - rho)).float()
        s["sigma"] = [c["sigma"]] * c["S"]
        s["rows"] = _online_rows(c)
        dt = DTYPES[c["dtype"]]
        s["k_out"], s["v_out"] = (torch.zeros((s["rows"], c["d"]), dtype=dt, device="cuda") for _ in range(2))
        s["kept"] = torch.zeros(s["rows"], dtype=torch.int32, device="cuda")
        s["scores"] = torch.empty((c["S"], N, p.n), dtype=torch.float32, device="cuda")
        s["head_budgets"] = torch.empty((c["S"], N), dtype=torch.int32, device="cuda")
        s["offsets"] = torch.empty(c["S"] * N + 1, dtype=torch.int32, device="cuda")
        s["ws"] = lukv.alloc_workspace(p)
    elif kind == "profile":
        s["p"] = lukv.make_params(1, 1, c["N"], 1, 64, c["T"], c["w"], 1, "fp32", c["P"])
        s["Q"], s["ratios"] = c["Q"], [(i + 1) / (c["R"] + 1.0) for i in range(c["R"])]
        s["curves"] = _calibration_curves(c["Q"], c["N"], c["P"], c["T"], g)
        s["profile"] = torch.empty((c["R"], c["N"]), dtype=torch.float32, device="cuda")
        s["ws"] = _bytes(lukv.lukv_profile_workspace_bytes(s["p"], c["Q"], c["R"]))
    elif kind == "importance":
        S, L, H, G, d, T = c["S"], c["L"], c["H"], c["G"], c["d"], c["T"]
        dt = DTYPES[c["dtype"]]
        s["p"] = lukv.make_params(S, L, H, G, d, T, c["w"], 1, c["dtype"], 2 if T % 2 else 3)
        s["steps"], s["width"], s["normalize"] = c["steps"], c["width"], c["normalize"]
        s["q"] = _normal((S, L, H * G, c["steps"], d), dt, g)
        s["k"], s["v"] = (_normal((S, L, H, T, d), dt, g) for _ in range(2))
        s["k_dec"] = _normal((S, L, H, c["steps"], d), dt, g) if c["decode_keys"] else None
        s["w_o"] = _normal((L, H * G, d, c["width"]), dt, g).mul_(d ** -0.5)
        s["importance"] = torch.empty((S, L * H, T - c["w"]), dtype=torch.float32, device="cuda")
        s["ws"] = _bytes(lukv.lukv_importance_workspace_bytes(s["p"], c["steps"]))
    elif kind == "curves":
        P = c["P"] or c["T"] // c["seg"] + 1
        s["p"] = lukv.make_params(c["Q"], 1, c["N"], 1, 64, c["T"], c["w"], 1, "fp32", P, n_sink=c["n_sink"])
        shape = (c["Q"], c["N"], c["T"] - c["w"])
        # attention-like values over several orders of magnitude; the importance follows the proxy with noise
        z = _normal(shape, torch.float32, g)
        s["scores"] = (2.0 * z).exp_()
        s["importance"] = (1.5 * z + _normal(shape, torch.float32, g)).exp_()
        s["curves"] = torch.empty((c["Q"], c["N"], P), dtype=torch.float32, device="cuda")
    else:  # exact
        s["p"] = lukv.make_params(1, 1, c["N"], 1, 64, c["T"], c["w"], 1, "fp32", c["T"] + 1)
        s["budgets"] = [int(c["keep"] * c["N"] * (c["T"] - c["w"]))]
        s["curves"] = _calibration_curves(1, c["N"], c["T"] + 1, c["T"], g)[0]
        s["head_budgets"] = torch.empty((1, c["N"]), dtype=torch.int32, device="cuda")
        s["offsets"] = torch.empty(c["N"] + 1, dtype=torch.int32, device="cuda")
        s["values"] = torch.empty(1, dtype=torch.float64, device="cuda")
        s["ws"] = _bytes(lukv.lukv_exact_workspace_bytes(s["p"], s["budgets"][0]))
    return s


# ---- one pass -------------------------------------------------------------------------------------

def _bits(t):
    """Packed rows are byte copies of cache rows: handed over as whole numbers."""
    return t.view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


def run(s):
    kind, p = s["kind"], s["p"]
    if kind in ("compress", "keydiff"):
        o = s["out"]
        lukv.lukv_compress(p, s["q"], s["k"], s["v"], s["curves"], s["budgets"], o.k_out, o.v_out, o.kept_idx, o.budgets,
                           o.offsets, o.rows, o.dev_status, s["ws"])
        return [_bits(o.k_out), _bits(o.v_out), o.kept_idx, o.budgets, o.offsets, o.dev_status]
    if kind == "ragged":
        o = s["out"]
        lukv.lukv_compress_ragged(p, s["lens"], s["q"], s["k"], s["v"], s["curves"], s["budgets"], o.k_out, o.v_out,
                                  o.kept_idx, o.budgets, o.offsets, o.rows, o.dev_status, s["ws"])
        return [_bits(o.k_out), _bits(o.v_out), o.kept_idx, o.budgets, o.offsets, o.dev_status]
    if kind == "online":
        lukv.lukv_profile_budgets(p, s["profile"], s["ratios"], s["sigma"], s["head_budgets"], s["offsets"])
        lukv.lukv_score(p, s["q"], s["k"], s["scores"], s["ws"])
        lukv.lukv_select_gather(p, s["scores"], s["head_budgets"], s["offsets"], s["k"], s["v"], s["k_out"], s["v_out"],
                                s["kept"], s["rows"], s["ws"])
        return [s["scores"], _bits(s["k_out"]), _bits(s["v_out"]), s["kept"], s["head_budgets"], s["offsets"]]
    if kind == "profile":
        lukv.lukv_profile_build(p, s["curves"], s["Q"], s["ratios"], s["profile"], s["ws"])
        return s["profile"]
    if kind == "importance":
        lukv.lukv_oracle_importance(p, s["steps"], s["width"], s["q"], s["k"], s["v"], s["k_dec"], s["w_o"],
                                    s["normalize"], s["importance"], s["ws"])
        return s["importance"]
    if kind == "curves":
        lukv.lukv_build_curves(p, s["scores"], s["importance"], s["curves"])
        return s["curves"]
    lukv.lukv_exact_allocate(p, s["curves"], s["budgets"], s["head_budgets"], s["offsets"], s["values"], s["ws"])
    return [s["head_budgets"], s["offsets"], s["values"]]


# ---- what a pass cannot do without ------------------------------------------------------------------

def work(case):
    c, kind = case, case["kind"]
    if kind in ("compress", "ragged", "keydiff", "online"):
        es = 2 if c["dtype"] == "bf16" else 4
        N, d, w, G = c["L"] * c["H"], c["d"], c.get("w", 1), c.get("G", 1)
        lens = _lens(c) if kind == "ragged" else [c["T"]] * c["S"]
        keys, row = N * sum(lens), d * es
        rows = _online_rows(c) if kind == "online" else sum(_budgets(c)) + c["S"] * N * w
        # every key once, the kept values once (the kept keys are among the keys), both packed outputs and the positions
        total = keys * row + rows * row + 2 * rows * row + 4 * rows + 8 * c["S"] * N
        if kind == "keydiff":
            return {"bytes": total + 4 * N * c["P"], "flops": 4.0 * keys * d}
        total += c["S"] * N * G * w * row
        total += 4 * (keys - c["S"] * N * w) if kind == "online" else 4 * N * c["P"]  # scores are an output there
        return {"bytes": total, "flops": 2.0 * keys * G * w * d}
    if kind == "profile":
        return {"bytes": 4 * (c["Q"] * c["N"] * c["P"] + c["R"] * c["N"]), "flops": 4.0 * c["Q"] * c["N"] * c["P"]}
    if kind == "importance":
        es = 2 if c["dtype"] == "bf16" else 4
        N, n = c["S"] * c["L"] * c["H"], c["T"] - c["w"]
        total = N * (2 * c["T"] + c["G"] * c["steps"] + (c["steps"] if c["decode_keys"] else 0)) * c["d"] * es
        total += c["L"] * c["H"] * c["G"] * c["d"] * c["width"] * es + 4 * N * n
        return {"bytes": total, "flops": 2.0 * N * c["G"] * c["d"] * (n * c["width"] + c["steps"] * c["T"])}
    if kind == "curves":
        n, P = c["T"] - c["w"], c["P"] or c["T"] // c["seg"] + 1
        return {"bytes": 4 * c["Q"] * c["N"] * (2 * n + P), "flops": float(c["Q"] * c["N"] * n) * math.log2(n)}
    # exact: one addition and one comparison for every reachable (head, budget so far, tokens of this head)
    N, n = c["N"], c["T"] - c["w"]
    B = int(c["keep"] * N * n)
    pairs = sum((min(B, (h + 1) * n) - max(0, B - (N - 1 - h) * n) + 1) * min(n, B) for h in range(N))
    return {"bytes": 4 * N * (c["T"] + 1) + 8 * N + 8, "flops": 2.0 * pairs}


def tolerance(case):
    kind = case["kind"]
    if kind in ("compress", "ragged", "keydiff"):
        # positions, budgets and row bits are whole numbers; two positions whose scores agree to the last digits may
        # change places, which moves the rows between them
        return {"rel": 0.0, "differ": 0.01}
    if kind == "online":
        # a 32-bit logit of size 100 carries 1e-5, and so does its exponential
        return {"rel": 5e-5, "max": 2e-3, "differ": 0.01}
    if kind == "importance":
        return {"rel": 5e-5, "max": 2e-3}
    if kind == "curves":
        return {"rel": 1e-6, "max": 1e-5}  # 64-bit sums, rounded once
    return {"rel": 1e-6, "differ": 0.0}    # profile, exact: the rules fix every whole number
