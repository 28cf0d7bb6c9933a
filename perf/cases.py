"""The work that programs have this library do, as cases to be timed and compared.

A pass of a case is one of five things a serving or analysis program does:

  generate  a prompt's keys and values are compressed (`taskkv_compress_ex`, into buffers the program keeps) and
            `steps` tokens are decoded with the fused step, either every layer at once or layer by layer as a
            model's loop does it
  stream    the same, with the layers compressed one at a time as a prefill loop produces them
            (`taskkv_cache_create`, `taskkv_compress_layer`)
  paged     a batch of requests served from a page pool: compression into pages, `steps` fused steps, pages given back
  decode    attention over a cache that is already there (`taskkv_decode`, or `taskkv_decode_ex` per layer)
  semantic  the exact semantic vectors and column means of one sequence (`taskkv_exact_semantic`)

What a program sees of a compacted cache is the attention over it, so that is what the first four return, for every
step, layer and head: every retained row, the classes, the lengths and the appended rows enter it.

Inputs are seeded.  A query is its head's mean query plus noise of the same size, so that window rows and decode
queries favour the same keys, as attention does; scores have a standard deviation of about one; the first four keys
are attention sinks; the heads that Eq. 16 counts as heterogeneous carry an offset on V.
"""
import math

import numpy as np
import torch

from paper_2501_15113_b200 import binding as tk

_SINKS = 4           # leading keys that attract every query


def _case(name, kind, **kw):
    case = dict(name=name, kind=kind, layers=1, heads=32, kv_heads=8, dim=128, seq_lens="8192", dtype="bf16", window=32,
                sink=4, recent=256, mid=256, budget=0.0, top_t=256, beta=0.3, m=1, steps=1, by_layer=False)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: one fp32 layer of eight heads, launches and host work are all there is
        _case("toy_f32_generate", "generate", heads=8, kv_heads=8, dim=64, seq_lens="512", dtype="f32", window=16,
              recent=32, mid=32, beta=0.25, m=2, steps=16),
        # a chat-sized prompt of a 32-layer multi-head model, tokens decoded layer by layer
        _case("mha_4k_generate", "generate", layers=32, kv_heads=32, seq_lens="4096", mid=512, beta=0.125, m=4, steps=8,
              by_layer=True),
        # the long prompt of the same model: 32 layers x 32 heads x 32768 keys
        _case("mha_32k_prefill", "generate", layers=32, kv_heads=32, seq_lens="32768", mid=512, beta=0.125, m=4),
        # grouped queries at 131072 keys with 40 % of the cache kept
        _case("gqa_128k_prefill", "generate", layers=32, seq_lens="131072", budget=0.4),
        # a ragged batch of sixteen documents on a grouped-query model (8 of its layers)
        _case("gqa_ragged_batch", "generate", layers=8, recent=128, beta=0.25, m=2,
              seq_lens="8192 9001 10240 11777 12345 14336 16384 17003 18500 20011 21504 23333 25600 27777 30001 32768"),
        # a point of the budget sweep: eight sequences of 65536 keys, one layer
        _case("gqa_64k_sweep", "generate", seq_lens=" ".join(["65536"] * 8), beta=0.25, m=2, steps=4),
        # layers compressed as a prefill loop hands them over, then tokens layer by layer
        _case("gqa_8k_stream", "stream", layers=32, seq_lens="8191", steps=4, by_layer=True),
        # three requests in and out of a page pool
        _case("gqa_paged_requests", "paged", layers=16, seq_lens="1500 3071 6000", steps=32),
        # decode over the long multi-head cache, every layer in one call
        _case("mha_32k_decode", "decode", layers=32, kv_heads=32, seq_lens="32768", mid=512, beta=0.125, m=4),
        # decode over a ragged batch, layer by layer
        _case("gqa_ragged_decode", "decode", layers=32, recent=128, beta=0.25, m=2, by_layer=True,
              seq_lens="8192 1000 5003 2048 12345 3333 7001 4096"),
        # fp32 compression of a medium prompt, grouped queries
        _case("f32_6k_generate", "generate", layers=8, heads=16, kv_heads=4, dim=64, seq_lens="6001", dtype="f32",
              recent=128, steps=4),
        # exact semantic vectors of one layer
        _case("semantic_16k", "semantic", kv_heads=32, seq_lens="16384"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["generate"] * 6 + ["decode"] * 2 + ["stream", "paged", "semantic"])
    heads, kv_heads = rng.choice([(32, 32), (32, 8), (32, 8), (16, 8), (8, 8), (16, 4), (32, 4)])
    dim = rng.choice([128, 128, 128, 64])
    if kind == "semantic":
        return _drawn(kind, heads=heads, kv_heads=kv_heads, dim=dim, seq_lens=str(log_int(400, 14000)))
    dtype = "bf16" if kind == "paged" else rng.choice(["bf16"] * 6 + ["f32"])
    group = heads // kv_heads
    window = rng.choice([32, 32, 32, 16]) if group <= 4 else 16
    batch = rng.choice([1, 1, 1, 2, 3, 8, 16])
    top = {1: 131072, 2: 65536, 3: 65536, 8: 65536, 16: 32768}[batch]
    if dtype == "f32":
        top = 16384
    if kind == "paged":
        top = 16384
    longest = log_int(400, top)
    lens = [longest] + [log_int(max(300, longest // 4), longest) for _ in range(batch - 1)]
    per_layer = sum(lens) * kv_heads * dim * 2 * (2 if dtype == "bf16" else 4)
    most = 3e9 if dtype == "bf16" else 3e8
    layers = rng.choice([r for r in (1, 2, 4, 8, 16, 32) if r * per_layer <= most or r == 1])
    by_layer = kind == "stream" or rng.random() < 0.4
    steps = 1 if kind == "decode" else rng.choice([1, 1, 4, 8])
    return _drawn(kind, layers=layers, heads=heads, kv_heads=kv_heads, dim=dim, dtype=dtype, window=window,
                  seq_lens=" ".join(map(str, lens)), recent=rng.choice([32, 128, 256]), mid=log_int(32, 2048),
                  budget=rng.choice([0.0, 0.0, 0.4]), beta=rng.choice([0.125, 0.25, 0.3]), m=rng.choice([1, 2]),
                  steps=steps, by_layer=by_layer)


def _drawn(kind, **kw):
    case = _case("", kind, **kw)
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------------------- sizes
def _lens(case):
    return [int(x) for x in case["seq_lens"].split()]


def _far_heads(case, r):
    """Eq. 16 for layer r."""
    n, R = case["kv_heads"], case["layers"]
    top = n * float(np.float32(case["beta"]))
    f = top if R <= 1 else top - (top - case["m"]) / (R - 1) * r
    return max(0, min(n, int(math.floor(f + 0.5))))


def _kept(case, r, N):
    """(heads of layer r that keep everything, rows the others keep of N)."""
    n, s = case["kv_heads"], case["sink"] + case["recent"]
    f = _far_heads(case, r)
    full = min(n, f + 1)
    mid = case["mid"]
    if case["budget"] > 0:                                                   # Eq. 17
        mid = 0 if full >= n else math.floor((float(np.float32(case["budget"])) * n * N - N * full) / (n - full)) - s
    return full, N if N <= s else s + max(0, min(mid, N - s))


def work(case):
    n, kv, d, R = case["heads"], case["kv_heads"], case["dim"], case["layers"]
    es, rows = (2 if case["dtype"] == "bf16" else 4), case["heads"] * case["window"]
    if case["kind"] == "semantic":
        N = _lens(case)[0]
        return {"bytes": R * (N * d * 2 * (n + 2 * kv) + kv * (N + d) * 4), "flops": R * n * N * (N + 1) / 2 * 2 * d}
    moved, flops = 0.0, 0.0
    for N in _lens(case):
        for r in range(R):
            full, kept = _kept(case, r, N)
            held = full * N + (kv - full) * kept
            if case["kind"] != "decode":
                # the window's queries, K once, the V rows that are kept or enter a semantic vector, the kept rows out
                v_rows = full * N + (kv - full) * min(N, kept + case["top_t"])
                moved += (rows * d + kv * N * d + v_rows * d + 2 * held * d) * es
                flops += 2.0 * rows * N * d
            for t in range(case["steps"]):
                grown = held + (0 if case["kind"] == "decode" else (t + 1) * kv)
                moved += (2 * grown * d + 2 * n * d) * es
                flops += 4.0 * grown * (n // kv) * d
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # Measured against 64 bits: bf16 outputs 1.8e-3, fp32 outputs 1.6e-7, exact vectors and column means 5e-7.  A score
    # within the rounding of the selection boundary may fall on either side of it; such a row moves its head's output by
    # that row's share, which is what the room above four times those figures is for.
    if case["kind"] == "semantic":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1e-2, "max": 0.5} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-2}


# ---------------------------------------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _inputs(case, seed):
    """(q_win, k, v per sequence; q, k_new, v_new per step), laid out as the calls take them."""
    g = _generator(seed)
    R, n, kv, d, L = case["layers"], case["heads"], case["kv_heads"], case["dim"], case["window"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    lens, T = _lens(case), case["steps"]
    B = len(lens)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dt)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device="cuda") + 0.5

    mean_q = 0.7 * torch.randn(R, n, 1, d, generator=g, device="cuda")
    k_scale, v_scale = uniform(R, kv, 1, 1), uniform(R, kv, 1, 1)
    offset = torch.zeros(R, kv, 1, d, device="cuda")
    order = torch.rand(R, kv, generator=g, device="cuda").argsort(dim=1)
    sign = (torch.rand(R, kv, 1, d, generator=g, device="cuda") < 0.5).float() * 2 - 1
    for r in range(R):
        far = order[r, :_far_heads(case, r)]
        offset[r, far] = sign[r, far]
    sink = mean_q.view(R, kv, n // kv, d).mean(2, keepdim=True)
    sink = 4.0 * math.sqrt(d) * sink / sink.square().sum(-1, keepdim=True)

    q_win, k, v = [], [], []
    for N in lens:
        q_win.append(normal(R, n, L, d).mul_(0.7).add_(mean_q.to(dt)))
        kb = normal(R, kv, N, d).mul_(k_scale.to(dt))
        kb[:, :, :_SINKS] += sink.to(dt)
        k.append(kb)
        v.append(normal(R, kv, N, d).mul_(v_scale.to(dt)).add_(offset.to(dt)))
    # one tensor per step, [layers, batch, ...] for the layer-by-layer loop and [batch, layers, ...] otherwise
    lead = (T, R, B) if case["by_layer"] else (T, B, R)
    mq = mean_q.view(R, 1, n, d) if case["by_layer"] else mean_q.view(R, n, d)
    ks = k_scale.view(R, 1, kv, 1) if case["by_layer"] else k_scale.view(R, kv, 1)
    q = normal(*lead, n, d).mul_(0.7).add_(mq.to(dt))
    k_new = normal(*lead, kv, d).mul_(ks.to(dt))
    v_new = normal(*lead, kv, d)
    return q_win, k, v, q, k_new, v_new


def _semantic_inputs(case, seed):
    g = _generator(seed)
    R, n, kv, d, N = case["layers"], case["heads"], case["kv_heads"], case["dim"], _lens(case)[0]

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)

    mean_q = 0.7 * torch.randn(R, n, 1, d, generator=g, device="cuda")
    q = normal(R, n, N, d).mul_(0.7).add_(mean_q.bfloat16())
    return q, normal(R, kv, N, d), normal(R, kv, N, d)


def _params(case):
    lens = _lens(case)
    return tk.Params(n_layers=case["layers"], n_heads=case["heads"], n_kv_heads=case["kv_heads"], head_dim=case["dim"],
                     seq_lens=lens, sink=case["sink"], recent=case["recent"], mid_budget=case["mid"], window=case["window"],
                     dtype=case["dtype"], top_t=case["top_t"], beta=case["beta"], m_top=case["m"],
                     budget_frac=case["budget"], max_new_tokens=0 if case["kind"] == "decode" else case["steps"])


def prepare(case, seed):
    if case["kind"] == "semantic":
        q, k, v = _semantic_inputs(case, seed)
        R, kv, N, d = k.shape
        scratch = torch.empty(int(tk.lib.taskkv_exact_semantic_bytes(R, case["heads"], kv, d, N)), dtype=torch.uint8,
                              device="cuda")
        return {"case": case, "q": q, "k": k, "v": v, "scratch": scratch}
    q_win, k, v, q, k_new, v_new = _inputs(case, seed)
    params = _params(case)
    state = {"case": case, "params": params, "q_win": q_win, "k": k, "v": v, "q": q, "k_new": k_new, "v_new": v_new,
             "out": torch.empty_like(q), "cache": None, "pool": None}
    if case["kind"] == "paged":
        info, pages = tk.taskkv_plan_paged(params, 64)
        pages += int(info.n_units)                                          # room for one more page per head
        state["pool"] = tk.Pool(64, pages, case["dim"], case["dtype"], "cuda")
    else:
        info = tk.taskkv_plan(params)
    state["cache_mem"] = torch.empty(int(info.cache_bytes), dtype=torch.uint8, device="cuda")
    state["workspace"] = torch.empty(int(info.workspace_bytes), dtype=torch.uint8, device="cuda")
    if case["kind"] == "stream":                                            # a prefill loop has one layer at a time
        state["layers"] = [([x[r] for x in q_win], [x[r] for x in k], [x[r] for x in v]) for r in range(case["layers"])]
    if case["kind"] == "decode":
        state["cache"] = tk.taskkv_compress_ex(params, q_win, k, v, cache_mem=state["cache_mem"],
                                               workspace_mem=state["workspace"])
        torch.cuda.synchronize()
        for name in ("q_win", "k", "v"):                                    # the prompt's own cache is dropped
            state[name] = None
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "semantic":
        return tk.taskkv_exact_semantic(state["q"], state["k"], state["v"], workspace_mem=state["scratch"])
    q, k_new, v_new, out = state["q"], state["k_new"], state["v_new"], state["out"]
    if case["kind"] == "decode":
        if case["by_layer"]:
            for r in range(case["layers"]):
                state["cache"].taskkv_decode_ex(q[0, r], r, 1, out=out[0, r])
        else:
            state["cache"].taskkv_decode(q[0], out=out[0])
        return out
    memory = {"cache_mem": state["cache_mem"], "workspace_mem": state["workspace"]}
    if case["kind"] == "stream":
        cache = tk.taskkv_cache_create(state["params"], "cuda", **memory)
        for r, (q_r, k_r, v_r) in enumerate(state["layers"]):
            cache.taskkv_compress_layer(r, q_r, k_r, v_r)
    elif case["kind"] == "paged":
        cache = tk.taskkv_compress_paged(state["params"], state["q_win"], state["k"], state["v"], state["pool"], **memory)
    else:
        cache = tk.taskkv_compress_ex(state["params"], state["q_win"], state["k"], state["v"], **memory)
    for t in range(case["steps"]):
        if case["by_layer"]:
            for r in range(case["layers"]):
                cache.taskkv_decode_step_ex(q[t, r], k_new[t, r], v_new[t, r], r, 1, out=out[t, r])
        else:
            cache.taskkv_decode_step(q[t], k_new[t], v_new[t], out=out[t])
    if case["kind"] == "paged":
        cache.close()                                                       # the requests are done: their pages go back
    return out


# ---------------------------------------------------------------------------------------------------- 64 bits
def exact(case, seed):
    if case["kind"] == "semantic":
        return _exact_semantic(case, seed)
    q_win, k, v, q, k_new, v_new = _inputs(case, seed)
    R, n, kv, d, L = case["layers"], case["heads"], case["kv_heads"], case["dim"], case["window"]
    G, T, s1, s2 = n // kv, case["steps"], case["sink"], case["recent"]
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    future = torch.ones(L, L, device="cuda", dtype=torch.bool).triu(1)
    for b, N in enumerate(_lens(case)):
        for r in range(R):
            Q, K, V = q_win[b][r].double().view(kv, G * L, d), k[b][r].double(), v[b][r].double()
            C = torch.empty(kv, N, dtype=torch.float64, device="cuda")
            for h in range(kv):
                S = (Q[h] @ K[h].T).view(G, L, N) / math.sqrt(d)
                S[:, :, N - L:].masked_fill_(future, -math.inf)
                C[h] = torch.softmax(S, -1).mean((0, 1))
            top = C.topk(min(case["top_t"], N), dim=1).indices
            sem = torch.stack([C[h, top[h]] @ V[h, top[h]] for h in range(kv)])
            dist = (sem - sem.mean(0)).norm(dim=1)
            f = _far_heads(case, r)
            full, kept = _kept(case, r, N)
            by_dist = dist.argsort(descending=True).tolist()
            whole = set(by_dist[:f]) | set(by_dist[-1:] if full > f else [])
            pooled = torch.nn.functional.avg_pool1d(C[:, None], 7, 1, 3, count_include_pad=True)[:, 0]
            for h in range(kv):
                Kh, Vh = K[h], V[h]
                if h not in whole and kept < N:
                    pos = pooled[h, s1:N - s2].topk(kept - s1 - s2).indices.sort().values + s1
                    pos = torch.cat([torch.arange(s1, device="cuda"), pos, torch.arange(N - s2, N, device="cuda")])
                    Kh, Vh = Kh[pos], Vh[pos]
                at = (slice(None), r, b) if case["by_layer"] else (slice(None), b, r)
                held = Kh.shape[0]
                if case["kind"] != "decode":
                    Kh, Vh = torch.cat([Kh, k_new[at][:, h].double()]), torch.cat([Vh, v_new[at][:, h].double()])
                S = q[at][:, h * G:(h + 1) * G].double() @ Kh.T / math.sqrt(d)          # [T, G, rows]
                if case["kind"] != "decode":
                    late = torch.arange(T, device="cuda")[None] > torch.arange(T, device="cuda")[:, None]
                    S[:, :, held:].masked_fill_(late[:, None], -math.inf)
                out[at][:, h * G:(h + 1) * G] = torch.softmax(S, -1) @ Vh
    return out


def _exact_semantic(case, seed):
    q, k, v = _semantic_inputs(case, seed)
    R, n, N, d = q.shape
    kv = k.shape[1]
    C = torch.zeros(R, kv, N, dtype=torch.float64, device="cuda")
    for r in range(R):
        for a in range(n):
            K = k[r, a // (n // kv)].double()
            for i in range(0, N, 2048):
                rows = q[r, a, i:i + 2048].double()
                S = rows @ K[:i + rows.shape[0]].T / math.sqrt(d)
                S.masked_fill_(torch.ones(S.shape, device="cuda", dtype=torch.bool).triu(i + 1), -math.inf)
                C[r, a // (n // kv), :S.shape[1]] += torch.softmax(S, -1).sum(0)
    C /= (n // kv) * N
    return torch.einsum("rhn,rhnd->rhd", C, v.double()), C
