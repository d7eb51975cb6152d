"""The measured cases: what users of the memory layer have it do.

Every case is one call of a public entry point of ``UltraMemLayer`` on a layer
of the sizes that the repository's workloads name (``workloads.CONFIGS``) or,
for drawn cases, of sizes between and beside them.  All inputs are Gaussians
at the layer's scale, made on the GPU from the seed alone.

A case's fields: the layer's hyper-parameters in the C ABI's names, ``tokens``
(a batch is ``n_seq`` sequences of ``tokens / n_seq`` tokens) and ``entry``:

  forward         S1-S9 on device tensors
  forward_seq     the same with the query convolution's state in and out
  forward_host    the same on pinned host buffers, both copies inside
  retrieve        S1-S6: the selected slots and their weights
  lookup_reduce   S7-S9 on given slots
  backward        the gradients of the lookup-reduce on given slots
  exact           the brute-force top-m of each head's whole grid
"""
from __future__ import annotations

import math

import torch

from paper_2411_12364_gb300.binding import UltraMemLayer

LAYER = ("d_in", "d_k", "heads", "rank", "n", "expand_e", "d_v", "d_out", "topk", "topm",
         "has_proj", "share_query", "act", "dtype", "cores", "conv_k", "query_ln", "score_mode",
         "shuffle_seed")

_BASE = dict(d_in=2048, d_k=128, heads=4, rank=2, n=2048, expand_e=4, d_v=256, d_out=2048,
             topk=64, topm=64, has_proj=1, share_query=1, act=0, dtype=1, cores=0, conv_k=0,
             query_ln=0, score_mode=0, shuffle_seed=1002)
_DECODE = dict(d_in=1024, heads=2, n=1024, d_out=1024, topk=32, topm=32, shuffle_seed=1001)
_TINY = dict(d_in=256, d_k=64, heads=2, n=256, expand_e=1, d_out=256, topk=16, topm=16,
             has_proj=0, dtype=0, shuffle_seed=1000)


def _case(name, entry, tokens, n_seq=1, **over):
    c = dict(_BASE, entry=entry, tokens=tokens, n_seq=n_seq)
    c.update(over)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one decode step of 64 sequences through the decode-shaped layer: the
        # benchmark's headline
        _case("decode_1m_b64", "forward", 64, **_DECODE),
        # one token of one interactive stream through the mid-size layer: the
        # smallest call of a served model
        _case("mid_4m_b1", "forward", 1),
        # a decode step of a large batch through the 20M-row table
        _case("large_20m_b256", "forward", 256, n=4480),
        # a ragged prefill chunk with the paper's default two-core scoring
        _case("mid_4m_mcs2_b1000", "forward", 1000, cores=2),
        # a whole prefill chunk: 4 sequences of 4096 tokens
        _case("prefill_16k", "forward", 16384, n_seq=4),
        # prompts of four sequences through the layer with every query-side
        # option: 4-tap convolution with its state, query LayerNorm
        _case("decode_1m_conv_ln_4x500", "forward_seq", 2000, n_seq=4, conv_k=4, query_ln=1,
              **_DECODE),
        # the small fp32 layer, no virtual expansion
        _case("tiny_fp32_b16", "forward", 16, **_TINY),
        # a decode step in fp32 storage (the precision mode), ragged batch
        _case("decode_1m_fp32_b77", "forward", 77, dtype=0, **_DECODE),
        # a decode step called on host buffers: what the benchmark's end-to-end
        # figure measures
        _case("decode_1m_host_b64", "forward_host", 64, **_DECODE),
        # the lookup half of the layer on slots selected elsewhere (a training
        # forward, a sharded selection): one 2048-token sequence
        _case("mid_4m_lookup_b2048", "lookup_reduce", 2048),
        # the training backward of the lookup for one 2048-token sequence
        _case("decode_1m_backward_b2048", "backward", 2048, **_DECODE),
        # the recall measurement's reference: the exact top-m of every grid
        _case("decode_1m_exact_b64", "exact", 64, **_DECODE),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: an entry point, a layer between the named workloads'
    sizes and a batch of any length.  Work stays below prefill_16k's."""
    entry = rng.choice(["forward"] * 5 + ["forward_seq", "forward_seq", "forward_host",
                                          "retrieve", "lookup_reduce", "lookup_reduce",
                                          "backward", "backward", "exact"])
    heads = rng.choice([1, 2, 2, 3, 4])
    d_in = rng.choice([512, 768, 1024, 1536, 2048])
    topk = rng.choice([16, 24, 32, 48, 64])
    over = dict(d_in=d_in, d_out=d_in, heads=heads, topk=topk, topm=topk,
                d_k=rng.choice([64, 128]), d_v=rng.choice([128, 256]),
                n=_log_int(rng, 200, 2048), expand_e=rng.choice([1, 4, 4, 4, 9]),
                rank=rng.choice([2, 2, 2, 4]), share_query=rng.choice([1, 1, 1, 0]),
                shuffle_seed=rng.randrange(1, 1 << 20))
    tokens, n_seq = _log_int(rng, 1, 4096), 1
    kind = rng.random()
    if entry in ("forward", "retrieve", "forward_host") and kind < 0.15:
        over.update(rank=1, score_mode=1, act=1)          # product keys with their softmax
    elif entry in ("forward", "lookup_reduce", "backward") and kind < 0.4:
        over.update(cores=2)                              # Multi-Core Scoring
    if entry == "forward" and rng.random() < 0.2 or entry == "backward" and rng.random() < 0.2:
        over.update(dtype=0, n=min(over["n"], 1100))      # the precision mode
        tokens = min(tokens, 300)
    if entry == "forward" and rng.random() < 0.15:
        over.update(n=_log_int(rng, 2049, 4480), expand_e=4, dtype=1)   # up to the largest table
    if entry == "forward_seq":
        over.update(conv_k=rng.choice([2, 4]), query_ln=rng.choice([0, 1]))
        n_seq = _log_int(rng, 1, 64)
        tokens = n_seq * max(1, tokens // n_seq)
    if entry == "forward_host":
        tokens = min(tokens, 512)
    if entry == "backward":
        over["n"] = min(over["n"], 1200)
    if entry == "exact":
        over.update(n=min(over["n"], 1024), expand_e=rng.choice([1, 4]), share_query=1)
        tokens = max(1, min(tokens, 64 // heads))
    return _case(None, entry, tokens, n_seq=n_seq, **over)


# -- inputs -----------------------------------------------------------------

def _randn(gen, shape, std, dtype):
    return torch.randn(*shape, generator=gen, device="cuda").mul_(std).to(dtype)


def _keys(case):
    return math.isqrt(case["expand_e"]) * case["n"]


def _inputs(case, seed):
    """The layer's parameters and the call's inputs, on the GPU."""
    c = case
    gen = torch.Generator(device="cuda").manual_seed(1 + seed)
    dt = torch.bfloat16 if c["dtype"] else torch.float32
    H, dk, K, r, E = c["heads"], c["d_k"], _keys(c), c["rank"], c["expand_e"]
    hd, h, N = H * dk, max(1, c["cores"]), c["n"] ** 2
    w = dict(w_q=_randn(gen, (hd, c["d_in"]), c["d_in"] ** -0.5, dt),
             w_q_col=None if c["share_query"]
             else _randn(gen, (hd, c["d_in"]), c["d_in"] ** -0.5, dt),
             k_row=_randn(gen, (H, K, dk), dk ** -0.5, dt),
             k_col=_randn(gen, (H, K, dk), dk ** -0.5, dt),
             core=_randn(gen, (H, h, r, r) if c["cores"] > 1 else (H, r, r), h ** -0.5,
                         torch.float32).cpu(),
             w_proj=_randn(gen, (E, c["d_v"], c["d_out"]), (E * c["d_v"]) ** -0.5, dt)
             if c["has_proj"] else None)
    if c["score_mode"]:
        w["core"] = None
    if c["conv_k"]:
        w["conv_w"] = _randn(gen, (c["conv_k"], c["d_in"]), c["conv_k"] ** -0.5, torch.float32)
        w["conv_b"] = _randn(gen, (c["d_in"],), 0.1, torch.float32)
    if c["query_ln"]:
        A = 1 if c["share_query"] else 2
        w["ln_g"] = 1 + _randn(gen, (A, hd), 0.1, torch.float32)
        w["ln_b"] = _randn(gen, (A, hd), 0.1, torch.float32)
    values = torch.empty((N, c["d_v"]), dtype=dt, device="cuda")
    rows = (1 << 26) // c["d_v"]
    for r0 in range(0, N, rows):
        r1 = min(N, r0 + rows)
        values[r0:r1] = _randn(gen, (r1 - r0, c["d_v"]), 0.02, dt)
    w["values"] = values
    B, m = c["tokens"], c["topm"]
    call = {}
    if c["entry"] in ("lookup_reduce", "backward"):
        # slots as a selection leaves them: addresses spread over the whole
        # virtual grid, positive scores in falling order (with component cores
        # each slot's score split over them)
        call["idx"] = torch.randint(0, E * N, (B, H, m), generator=gen, device="cuda")
        s = _randn(gen, (B, H, m), 1.0, torch.float32).abs_().add_(2.0)
        s = s.sort(-1, descending=True).values
        if c["cores"] > 1:
            part = torch.softmax(_randn(gen, (B, H, m, h), 1.0, torch.float32), -1)
            s = s.unsqueeze(-1) * part
        call["w"] = s.contiguous()
    else:
        call["x"] = _randn(gen, (B, c["d_in"]), 1.0, dt)
    if c["entry"] == "backward":
        call["g"] = _randn(gen, (B, c["d_out"]), 1.0, dt)
    if c["entry"] == "forward_seq" and c["conv_k"] > 1:
        call["state"] = _randn(gen, (c["n_seq"], c["conv_k"] - 1, c["d_in"]), 1.0, dt)
    return w, call


def prepare(case, seed):
    w, call = _inputs(case, seed)
    layer = UltraMemLayer({k: case[k] for k in LAYER}, w, case["tokens"])
    st = dict(layer=layer, entry=case["entry"], n_seq=case["n_seq"], **call)
    if case["entry"] == "forward_host":
        st["x"] = call["x"].cpu().pin_memory()
        st["out"] = torch.empty((case["tokens"], case["d_out"]),
                                dtype=st["x"].dtype).pin_memory()
    if "state" in call:
        st["next"] = torch.empty_like(call["state"])
    return st


def run(state):
    layer, entry = state["layer"], state["entry"]
    if entry == "forward":
        return layer.forward(state["x"])
    if entry == "forward_seq":
        out = layer.forward_seq(state["x"], state["n_seq"], state.get("state"),
                                state.get("next"))
        return (out, state["next"]) if "next" in state else out
    if entry == "forward_host":
        return layer.forward_host(state["x"], state["out"])
    if entry == "retrieve":
        return layer.retrieve(state["x"])
    if entry == "exact":
        return layer.retrieve_exact(state["x"])
    if entry == "lookup_reduce":
        return layer.lookup_reduce(state["idx"], state["w"])
    dv, dw, dwp = layer.lookup_reduce_backward(state["idx"], state["w"], state["g"])
    return (dv, dw, dwp) if dwp is not None else (dv, dw)


# -- what a pass cannot do without ------------------------------------------

def work(case):
    c = case
    es = 2 if c["dtype"] else 4
    B, H, K, dk, r = c["tokens"], c["heads"], _keys(c), c["d_k"], c["rank"]
    E, dv, do, k, m = c["expand_e"], c["d_v"], c["d_out"], c["topk"], c["topm"]
    h, A, N = max(1, c["cores"]), 1 if c["share_query"] else 2, c["n"] ** 2
    slots, kd = B * H * m, E * dv
    proj = kd * do if c["has_proj"] else 0
    rows = min(slots, N) * dv * es
    by = fl = 0
    if c["entry"] not in ("lookup_reduce", "backward"):
        by += B * c["d_in"] * es + A * H * dk * c["d_in"] * es + 2 * H * K * dk * es
        fl += 2 * A * B * H * dk * c["d_in"] + 4 * B * H * K * dk
        if c["conv_k"]:
            by += (c["conv_k"] + 1) * c["d_in"] * 4 \
                + 2 * c["n_seq"] * (c["conv_k"] - 1) * c["d_in"] * es
            fl += 2 * B * c["conv_k"] * c["d_in"]
        if c["entry"] == "exact":
            fl += 2 * B * H * K * K * r
        else:
            fl += 4 * B * H * K * r + 2 * B * H * k * k * r
    if c["entry"] in ("retrieve", "exact"):
        by += slots * (8 + 4 * (h if c["entry"] == "retrieve" else 1))
    elif c["entry"] == "backward":
        by += slots * (8 + 8 * h) + B * do * es + rows + N * dv * 4 + proj * (es + 4)
        fl += 6 * slots * dv + 4 * B * proj
    else:
        by += rows + proj * es + B * do * es
        fl += 2 * slots * dv + 2 * B * proj
        if c["entry"] == "lookup_reduce":
            by += slots * (8 + 4 * h)
    return {"bytes": by, "flops": fl}


# -- the same in 64 bits, from the formulas ---------------------------------

def _shuffle(seed, M):
    """The seeded bijection v -> (a v + c) mod M (two SplitMix64 outputs)."""
    if seed == 0 or M <= 1:
        return 1, 0
    mask, gold = (1 << 64) - 1, 0x9E3779B97F4A7C15

    def out(s):
        z = (s + gold) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)

    a, c = 1 + out(seed) % (M - 1), out((seed + gold) & mask) % M
    while math.gcd(a, M) != 1:
        a = 1 if a + 1 >= M else a + 1
    return a, c


def _rank1(core):
    """Leading singular pair of each head's core, sum(u) > 0."""
    U, S, Vh = torch.linalg.svd(core)
    u, s = U[..., 0], S[..., 0]
    u = torch.where(u.sum(-1, keepdim=True) < 0, -u, u)
    return u, torch.einsum("hab,ha->hb", core, u) / s[:, None]


def _queries(case, w, call):
    """[q_row, q_col], each [B, H, D_k], and the next convolution state."""
    c, x = case, call["x"].double()
    nxt = None
    if c["conv_k"]:
        S, kc = c["n_seq"], c["conv_k"]
        xs = x.view(S, -1, c["d_in"])
        L = xs.shape[1]
        past = call["state"].double() if kc > 1 else xs[:, :0]
        full = torch.cat([past, xs], 1)
        nxt = full[:, full.shape[1] - (kc - 1):] if kc > 1 else None
        y = w["conv_b"].double() + torch.zeros_like(xs)
        for j in range(kc):
            y += w["conv_w"][j].double() * full[:, kc - 1 - j:kc - 1 - j + L]
        x = y.reshape(-1, c["d_in"])
    qs = []
    for a, wq in enumerate((w["w_q"], w["w_q_col"])):
        if wq is None:
            qs.append(qs[0])
            continue
        q = (x @ wq.double().T).view(-1, c["heads"], c["d_k"])
        if c["query_ln"]:
            d = q - q.mean(-1, keepdim=True)
            q = d / (d.square().mean(-1, keepdim=True) + 1e-5).sqrt()
            q = q * w["ln_g"][a].double().view(c["heads"], -1) \
                + w["ln_b"][a].double().view(c["heads"], -1)
        qs.append(q)
    return qs, nxt


def _chunk_scores(q, keys, r):
    """S [T, H, r, K]: each key's dot product with the query, per rank chunk."""
    T, H, dk = q.shape
    kk = keys.double().view(H, -1, r, dk // r)
    return torch.einsum("thrd,hkrd->thrk", q.view(T, H, r, dk // r), kk)


def _select(case, w, call):
    """(idx [B, H, m], weights [B, H, m] or [B, H, m, h], next state)."""
    c = case
    H, r, k, m, K = c["heads"], c["rank"], c["topk"], c["topm"], _keys(c)
    (qr, qc), nxt = _queries(c, w, call)
    if c["score_mode"]:
        cores = core = None
        u = t = torch.ones((H, 1), dtype=torch.float64, device="cuda")
    else:
        cores = w["core"].double().view(H, -1, r, r)
        core = cores.sum(1)
        u, t = (z.cuda() for z in _rank1(core))
        cores, core = cores.cuda(), core.cuda()
    exact = c["entry"] == "exact"
    step = max(1, (1 << 26) // (H * K * K)) if exact else max(1, (1 << 26) // (H * K * r))
    idxs, ws = [], []
    for b in range(0, qr.shape[0], step):
        sr = _chunk_scores(qr[b:b + step], w["k_row"], r)
        sc = _chunk_scores(qc[b:b + step], w["k_col"], r)
        T = sr.shape[0]
        if exact:
            i = j = torch.arange(K, device="cuda").expand(T, H, K)
        else:
            i = torch.einsum("thrk,hr->thk", sr, u).topk(k, -1).indices
            j = torch.einsum("thrk,hr->thk", sc, t).topk(k, -1).indices
            sr = sr.gather(3, i.unsqueeze(2).expand(T, H, r, k))
            sc = sc.gather(3, j.unsqueeze(2).expand(T, H, r, k))
        if core is None:
            g = sr[:, :, 0, :, None] + sc[:, :, 0, None, :]
        else:
            g = torch.einsum("thai,hab,thbj->thij", sr, core, sc)
        g, best = g.flatten(2).topk(m, -1)
        n2 = i.shape[2]
        pi, pj = best // n2, best % n2
        idxs.append(i.gather(2, pi) * K + j.gather(2, pj))
        if c["act"] and not exact:
            g = torch.softmax(g, -1)
        if c["cores"] > 1 and not exact:
            a = sr.gather(3, pi.unsqueeze(2).expand(T, H, r, m))
            d = sc.gather(3, pj.unsqueeze(2).expand(T, H, r, m))
            g = torch.einsum("tham,hcab,thbm->thmc", a, cores, d)
        ws.append(g)
    return torch.cat(idxs), torch.cat(ws), nxt


def _slots(case, idx):
    N = case["n"] ** 2
    a, c = _shuffle(case["shuffle_seed"], case["expand_e"] * N)
    v = (idx * a + c) % (case["expand_e"] * N)
    return v // N, v % N


def _slice_weights(case, w):
    """w [T, H, m(, h)] as one weight per value column."""
    if case["cores"] > 1:
        return w.repeat_interleave(case["d_v"] // case["cores"], dim=-1)
    return w.unsqueeze(-1)


def _pooled(case, values, idx, w):
    """acc [T, E, D_v]."""
    T, E, dv = idx.shape[0], case["expand_e"], case["d_v"]
    p, row = _slots(case, idx)
    rows = values[row.flatten()].double().view(*idx.shape, dv)
    rows = rows * _slice_weights(case, w.double())
    acc = torch.zeros((T * E, dv), dtype=torch.float64, device="cuda")
    dst = p + torch.arange(T, device="cuda")[:, None, None] * E
    acc.index_add_(0, dst.flatten(), rows.reshape(-1, dv))
    return acc.view(T, E, dv)


def _token_step(case):
    return max(1, (1 << 26) // (case["heads"] * case["topm"] * case["d_v"]))


def _lookup(case, wt, idx, w):
    outs = []
    for b in range(0, idx.shape[0], _token_step(case)):
        s = slice(b, b + _token_step(case))
        acc = _pooled(case, wt["values"], idx[s], w[s])
        outs.append(acc.flatten(1) if wt["w_proj"] is None else
                    acc.flatten(1) @ wt["w_proj"].double().flatten(0, 1))
    return torch.cat(outs)


def _backward(case, wt, idx, w, g):
    E, dv, h = case["expand_e"], case["d_v"], max(1, case["cores"])
    g, wp = g.double(), wt["w_proj"]
    dval = torch.zeros((case["n"] ** 2, dv), dtype=torch.float64, device="cuda")
    dws, dwp = [], None
    for b in range(0, idx.shape[0], _token_step(case)):
        s = slice(b, b + _token_step(case))
        T = g[s].shape[0]
        dacc = g[s].view(T, 1, dv) if wp is None else \
            torch.einsum("to,edo->ted", g[s], wp.double())
        p, row = _slots(case, idx[s])
        d = dacc.reshape(T * E, dv)[(p + torch.arange(T, device="cuda")[:, None, None] * E)]
        v = wt["values"][row.flatten()].double().view(*row.shape, dv)
        dws.append((d * v).view(*row.shape, h, dv // h).sum(-1))
        dval.index_add_(0, row.flatten(),
                        (d * _slice_weights(case, w[s].double())).reshape(-1, dv))
        if wp is not None:
            acc = _pooled(case, wt["values"], idx[s], w[s])
            part = torch.einsum("ted,to->edo", acc, g[s])
            dwp = part if dwp is None else dwp + part
    dw = torch.cat(dws)
    dw = dw if case["cores"] > 1 else dw.squeeze(-1)
    return (dval, dw, dwp) if dwp is not None else (dval, dw)


def exact(case, seed):
    """What ``run`` returns, in 64 bits; addresses have no such value."""
    wt, call = _inputs(case, seed)
    if case["entry"] == "lookup_reduce":
        return _lookup(case, wt, call["idx"], call["w"])
    if case["entry"] == "backward":
        return _backward(case, wt, call["idx"], call["w"], call["g"])
    idx, w, nxt = _select(case, wt, call)
    if case["entry"] in ("retrieve", "exact"):
        return None, w
    out = _lookup(case, wt, idx, w)
    if case["entry"] == "forward_host":
        return out.cpu()
    return (out, nxt) if nxt is not None else out
