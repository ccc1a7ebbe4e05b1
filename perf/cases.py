"""Performance cases of the Dynamic Mask Attention library: what a program that trains, prefills or decodes with it calls.

A case is a dict of plain values. `kind` says which of the library's call sequences one pass runs:

  train     dma_mask_build (or dma_mask_build_varlen for packed documents), dma_attn_fwd, dma_attn_bwd, dma_mask_bwd: one
            attention layer's training step; outputs O, lse, dQ, dK, dV, dW_delta, dA
  prefill   dma_mask_build, dma_attn_fwd; outputs O, lse
  mask      dma_mask_build alone; outputs bias, expiry, bitmap (bit patterns: the selection is specified to the bit)
  chunk     dma_mask_build over the keys so far, dma_attn_fwd_chunk for the newest rows; outputs O, lse
  decode    dma_delta_range for the appended key, dma_decode over the whole cache; outputs o, lse
  generate  dma_decode_state_init, then per token dma_delta_range and dma_decode_step; outputs every token's o, lse.
            With `graph` the loop is captured once in a CUDA graph, as a serving program keeps it

Inputs follow paper_2508_02124_b200/workloads.py: Q, K, V, dO ~ N(0, 1), W_delta ~ N(0, 1 / row length), A ~ U(0.5, 2),
drawn on the GPU. The training cases scale A by 1/4: with the full gates most rows of random inputs are nearly one-hot, and
dA is then a sum whose terms cancel to the rounding of O (measured 17 % off 64 bits at 16K keys), which compares nothing.
The gate's scale does not change which keys are kept.
"""
import heapq
import math

import torch

from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import workloads


def _case(kind, B, Hq, Hkv, L, d, w, dtype="bf16", causal=True, full=False, docs=0, rows=0, spare=0, tokens=0, graph=False):
    return {"kind": kind, "B": B, "Hq": Hq, "Hkv": Hkv, "L": L, "d": d, "w": w, "dtype": dtype, "causal": causal, "full": full,
            "docs": docs, "rows": rows, "spare": spare, "tokens": tokens, "graph": graph}


def listed():
    c = _case
    return [
        # long-context training layer: 32 query / 8 KV heads of 128 channels, 16K tokens (the headline benchmark's shapes)
        dict(c("train", 1, 32, 8, 16384, 128, 2048), name="train_16k"),
        # a window of half the sequence, no head grouping: one point of the benchmark's window sweep
        dict(c("train", 1, 16, 16, 8192, 128, 4096), name="train_8k_w4096"),
        # a small model's layer: short ragged sequences, 64 channels per head
        dict(c("train", 2, 16, 4, 1000, 64, 256), name="train_short_d64"),
        # the smallest configuration, in fp32 (debugging, unit-scale experiments): launches and latency
        dict(c("train", 1, 2, 2, 256, 64, 64, dtype="fp32"), name="train_tiny_fp32"),
        # pre-training on packed documents: 12 documents in one 16K row
        dict(c("train", 1, 32, 8, 16384, 128, 2048, docs=12), name="train_packed_16k"),
        # bidirectional layer with the sampling weights over the whole value row
        dict(c("train", 1, 16, 4, 4096, 128, 1024, causal=False, full=True), name="train_noncausal_4k"),
        # prompt processing, ordinary and long
        dict(c("prefill", 1, 16, 4, 4096, 128, 1024), name="prefill_4k"),
        dict(c("prefill", 1, 32, 8, 65536, 128, 4096), name="prefill_64k"),
        # prompt processing in pieces: the newest 2048 rows of 16K
        dict(c("chunk", 1, 32, 8, 16384, 128, 2048, rows=2048), name="prefill_chunk_16k"),
        # one token over a KV cache with spare room: a single stream, and a batch at long context
        dict(c("decode", 1, 32, 8, 16384, 128, 2048, spare=512), name="decode_16k"),
        dict(c("decode", 8, 32, 8, 65536, 128, 4096, spare=512), name="decode_64k_b8"),
        # a burst of tokens with the kept set carried along, captured in a CUDA graph
        dict(c("generate", 1, 32, 8, 16384, 128, 2048, spare=512, tokens=32, graph=True), name="generate_16k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "prefill", "prefill", "mask", "chunk", "decode", "decode", "generate"])
    Hkv, G, d = rng.choice([1, 2, 4, 8]), rng.choice([1, 2, 4]), rng.choice([64, 128, 128])
    Hq = Hkv * G
    if kind == "train":
        if rng.random() < 0.15:                           # fp32: small problems
            L = _log_int(rng, 64, 1024)
            return _case("train", rng.choice([1, 2]), min(Hq, 8), min(Hkv, Hq, 8), L, d, max(8, _log_int(rng, max(8, L // 8), L)), dtype="fp32")
        L = _log_int(rng, 128, 16384)
        w = max(16, _log_int(rng, max(16, L // 16), max(17, L // 2)))
        B = rng.choice([1, 1, 2, 4])
        while B > 1 and B * Hq * L > 32 * 16384:
            B //= 2
        mode = rng.random()
        if mode < 0.2:
            return _case("train", B, Hq, Hkv, L, d, w, docs=max(1, min(16, L // 100)))
        if mode < 0.4:
            L = min(L, 8192)
            return _case("train", B, Hq, Hkv, L, d, min(w, L // 2), causal=False, full=rng.random() < 0.5 and Hq * Hkv * d <= 16384)
        return _case("train", B, Hq, Hkv, L, d, w, full=rng.random() < 0.2 and Hq * Hkv * d <= 16384)
    if kind in ("prefill", "mask"):
        L = _log_int(rng, 128, 32768)
        return _case(kind, 1, Hq, Hkv, L, d, max(16, _log_int(rng, max(16, L // 16), max(17, L // 3))))
    if kind == "chunk":
        L = _log_int(rng, 1024, 32768)
        return _case(kind, 1, Hq, Hkv, L, d, max(64, L // rng.choice([4, 8, 16])), rows=min(L, _log_int(rng, 100, 4096)))
    if kind == "decode":
        L = _log_int(rng, 1024, 131072)
        B = _log_int(rng, 1, 16)
        while B > 1 and B * Hq * L > 8 * 32 * 65536:
            B = (B + 1) // 2
        return _case(kind, B, Hq, Hkv, L, d, max(64, L // rng.choice([4, 8, 16, 32])), spare=rng.choice([0, 512]))
    L = _log_int(rng, 1024, 32768)
    return _case(kind, rng.choice([1, 2, 4]), Hq, Hkv, L, d, max(64, L // rng.choice([4, 8, 16])), spare=512,
                 tokens=rng.choice([8, 16, 32]), graph=rng.random() < 0.7)


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _flags(case):
    f = dma.DMA_FLAG_FULL_DELTA if case["full"] else 0
    # the kept keys of packed documents cluster: the tile-walking kernels are the documented choice there
    return f | (dma.DMA_FLAG_TILE_PATH if case["docs"] > 1 else 0)


def _rows(case):
    """Query rows of the case."""
    return case["rows"] or {"decode": 1, "generate": case["tokens"]}.get(case["kind"], case["L"])


def _capacity(case):
    return case["L"] + case["tokens"] + case["spare"]


def _cu(case, seed):
    return workloads.packed_cu_seqlens(case["L"], case["docs"], seed) if case["docs"] else [0, case["L"]]


def _inputs(case, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    B, Hq, Hkv, d, dt, C = case["B"], case["Hq"], case["Hkv"], case["d"], _dtype(case), _capacity(case)

    def normal(*shape):
        out = torch.empty(*shape, dtype=dt, device="cuda")
        return out.copy_(torch.randn(*shape, generator=g, device="cuda"))

    x = {"K": normal(B, C, Hkv, d), "V": normal(B, C, Hkv, d)}
    n = Hkv * d if case["full"] else d
    x["W"] = torch.randn(Hq, n, generator=g, device="cuda") / math.sqrt(n)
    x["A"] = (torch.rand(Hq, generator=g, device="cuda") * 1.5 + 0.5) * (0.25 if case["kind"] == "train" else 1.0)
    x["Q"] = normal(_rows(case), B, Hq, d) if case["kind"] in ("decode", "generate") else normal(B, _rows(case), Hq, d)
    if case["kind"] == "train":
        x["dO"] = normal(B, case["L"], Hq, d)
    return x


def _problem(case, L=None):
    p = dma.problem(case["B"], case["Hq"], case["Hkv"], L or case["L"], case["d"], case["w"], dtype=_dtype(case),
                    causal=int(case["causal"]), flags=_flags(case))
    if case["kind"] in ("decode", "generate"):
        row = case["Hkv"] * case["d"]
        for s in (p.k_stride, p.v_stride):
            s[0], s[1], s[2] = _capacity(case) * row, row, case["d"]
    return p


def prepare(case, seed):
    kind, B, Hq, L = case["kind"], case["B"], case["Hq"], case["L"]
    s = dict(_inputs(case, seed), case=case)
    p = s["p"] = _problem(case)
    f32 = dict(dtype=torch.float32, device="cuda")
    ws = lambda n: torch.empty(n, dtype=torch.uint8, device="cuda")  # noqa: E731
    if kind in ("decode", "generate"):
        rows = _rows(case)
        s["delta"] = torch.zeros(B, Hq, (_capacity(case) + 3) // 4 * 4, **f32)
        dma.dma_delta_range(p, s["V"], s["W"], s["A"], s["delta"], 0, L)
        s["steps"] = [_problem(case, L + t + 1) for t in range(case["tokens"])]
        s["ws"] = ws(dma.dma_decode_workspace(s["steps"][-1] if s["steps"] else p))
        s["o"] = torch.empty_like(s["Q"])
        s["lse"] = torch.zeros(rows, (B * Hq + 3) // 4 * 4, **f32)
        if kind == "generate":
            s["state"] = dma.dma_decode_state(p, "cuda")
            s["graph"] = None
            if case["graph"]:
                _generate(s)
                torch.cuda.synchronize()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g):
                    _generate(s)
                s["graph"] = g
        return s
    s["bias"] = torch.empty(B, Hq, L, **f32)
    s["expiry"] = torch.empty(B, Hq, L, dtype=torch.int32, device="cuda")
    s["bitmap"] = torch.empty(dma.dma_bitmap_words(p), dtype=torch.int32, device="cuda")
    m, f, b = dma.dma_query_workspace(p)
    s["ws_m"], s["ws_f"] = ws(m), ws(f)
    if kind == "mask":
        return s
    s["O"], s["lse"] = torch.empty_like(s["Q"]), torch.empty(B, Hq, _rows(case), **f32)
    if kind == "chunk":
        pc = _problem(case)
        pc.flags |= dma.DMA_FLAG_COMPACT_KV
        s["ws_f"] = ws(dma.dma_query_workspace(pc)[1])
    if kind == "train":
        s["ws_b"], s["ws_g"] = ws(b), ws(dma.dma_mask_bwd_workspace(p))
        s["dQ"], s["dK"], s["dV"] = (torch.empty_like(s[k]) for k in ("Q", "K", "V"))
        s["dM"], s["dW"], s["dA"] = torch.empty(B, Hq, L, **f32), torch.empty_like(s["W"]), torch.empty_like(s["A"])
        if case["docs"]:
            s["cu"] = torch.tensor(_cu(case, seed), dtype=torch.int32, device="cuda")
    return s


def _generate(s):
    dma.dma_decode_state_init(s["p"], s["delta"], s["state"], ws=s["ws"])
    for t, p in enumerate(s["steps"]):
        dma.dma_delta_range(p, s["V"], s["W"], s["A"], s["delta"], p.L - 1, p.L)
        dma.dma_decode_step(p, s["Q"][t], s["K"], s["V"], s["delta"], s["state"], o=s["o"][t], lse=s["lse"][t], ws=s["ws"])


def run(s):
    case, p = s["case"], s["p"]
    kind, n = case["kind"], case["B"] * case["Hq"]
    if kind == "generate":
        if s["graph"] is not None:
            s["graph"].replay()
        else:
            _generate(s)
        return {"o": s["o"], "lse": s["lse"][:, :n]}
    if kind == "decode":
        dma.dma_delta_range(p, s["V"], s["W"], s["A"], s["delta"], p.L - 1, p.L)
        dma.dma_decode(p, s["Q"][0], s["K"], s["V"], s["delta"], o=s["o"][0], lse=s["lse"][0], ws=s["ws"])
        return {"o": s["o"], "lse": s["lse"][:, :n]}
    mask = s["bias"], s["expiry"], s["bitmap"]
    if case["docs"]:
        dma.dma_mask_build_varlen(p, s["V"], s["W"], s["A"], s["cu"], *mask, ws=s["ws_m"])
    else:
        dma.dma_mask_build(p, s["V"], s["W"], s["A"], *mask, ws=s["ws_m"])
    if kind == "mask":
        return {"bias": s["bias"], "expiry": s["expiry"], "bitmap": s["bitmap"]}
    if kind == "chunk":
        dma.dma_attn_fwd_chunk(p, p.L - case["rows"], s["Q"], s["K"], s["V"], s["bias"], s["expiry"], s["O"], s["lse"], ws=s["ws_f"])
        return {"O": s["O"], "lse": s["lse"]}
    dma.dma_attn_fwd(p, s["Q"], s["K"], s["V"], *mask, s["O"], s["lse"], ws=s["ws_f"])
    if kind == "train":
        dma.dma_attn_bwd(p, s["Q"], s["K"], s["V"], s["O"], s["dO"], s["lse"], *mask, s["dQ"], s["dK"], s["dV"], s["dM"], ws=s["ws_b"])
        dma.dma_mask_bwd(p, s["V"], s["W"], s["A"], s["bias"], s["dM"], s["dV"], s["dW"], s["dA"], ws=s["ws_g"])
        return {"O": s["O"], "lse": s["lse"], "dQ": s["dQ"], "dK": s["dK"], "dV": s["dV"], "dW": s["dW"], "dA": s["dA"]}
    return {"O": s["O"], "lse": s["lse"]}


def _kept_pairs(case):
    """(row, key) pairs that one (batch, head) keeps."""
    L, w = case["L"], case["w"]
    tri = lambda n: n * (n + 1) // 2 if n <= w else w * (w + 1) // 2 + (n - w) * w  # noqa: E731
    if case["kind"] in ("decode", "generate"):
        return sum(min(w, L + t + (case["kind"] == "generate")) for t in range(_rows(case)))
    if not case["causal"]:
        return L * min(w, L)
    if case["docs"]:
        cu = _cu(case, 0)
        return sum(tri(b - a) for a, b in zip(cu, cu[1:]))
    return tri(L) - tri(L - _rows(case))


def work(case):
    B, Hq, Hkv, L, d, w = (case[k] for k in ("B", "Hq", "Hkv", "L", "d", "w"))
    kind, e = case["kind"], 2 if case["dtype"] == "bf16" else 4
    kv, q = B * L * Hkv * d * e, B * _rows(case) * Hq * d * e
    zflops = 2 * B * L * Hq * (Hkv * d if case["full"] else d)
    pairs = B * Hq * _kept_pairs(case)
    if kind in ("decode", "generate"):
        # every token needs the delta of the appended key; the selection reads the delta row once; the kept K and V rows of a
        # KV head's query heads are read once a token, shared rows once
        share = 1 - (1 - min(1.0, w / L)) ** (Hq // Hkv)
        rows = _rows(case)
        return {"bytes": B * Hq * L * 4 + rows * B * Hkv * L * share * 2 * d * e + 2 * q, "flops": 4 * d * pairs}
    mask_out = B * Hq * L * 8
    if kind == "mask":
        return {"bytes": kv + mask_out, "flops": zflops}
    if kind in ("prefill", "chunk"):
        return {"bytes": 2 * kv + 2 * q, "flops": zflops + 4 * d * pairs}
    return {"bytes": 2 * kv + 3 * q + 2 * kv + q, "flops": 4 * zflops + 14 * d * pairs}


def tolerance(case):
    # about four times the distance from exact() of the path when it was written: 2.5e-3 (gradients), 1e-3 (o), 4e-7 (fp32)
    if case["kind"] == "mask":
        return "exact"
    if case["dtype"] == "fp32":
        return {"rel": 1e-5}
    return {"rel": 0.01, "max": 0.2} if case["kind"] == "train" else {"rel": 0.005, "max": 0.1}


# ---- the same results in 64 bits, from the definitions ------------------------------------------------------------------

def _delta64(case, x):
    """z and delta, [B, Hq, capacity] float64."""
    B, Hq, Hkv, d = (case[k] for k in ("B", "Hq", "Hkv", "d"))
    V, W, A = x["V"].double(), x["W"].double(), x["A"].double()
    if case["full"]:
        z = torch.einsum("bjc,hc->bhj", V.reshape(B, -1, Hkv * d), W)
    else:
        z = torch.einsum("bjkc,kgc->bkgj", V, W.view(Hkv, Hq // Hkv, d)).reshape(B, Hq, -1)
    sp = torch.nn.functional.softplus(z, threshold=1e9)
    return z, sp, torch.exp(A[None, :, None] * sp)


def _expiry64(case, delta, cu):
    """Row i keeps key j iff first_j <= i < expiry[j]: a heap of the w best keys walked over the rows."""
    w, L = case["w"], case["L"]
    out = torch.full(delta.shape, L, dtype=torch.int64)
    for b in range(case["B"]):
        for h in range(case["Hq"]):
            row, ex = delta[b, h, :L].tolist(), [L] * L
            if not case["causal"]:
                order = sorted(range(L), key=lambda j: (-row[j], j))
                for j in order[w:]:
                    ex[j] = 0
            else:
                for s0, s1 in zip(cu, cu[1:]):
                    heap = []
                    for i in range(s0, s1):
                        if len(heap) < w:
                            heapq.heappush(heap, (row[i], -i))
                        else:
                            ex[-heapq.heappushpop(heap, (row[i], -i))[1]] = i
                    for _, j in heap:
                        ex[-j] = s1
            out[b, h, :L] = torch.tensor(ex)
    return out.cuda()


def exact(case, seed):
    x = _inputs(case, seed)
    B, Hq, Hkv, L, d, w = (case[k] for k in ("B", "Hq", "Hkv", "L", "d", "w"))
    G, kind, scale = Hq // Hkv, case["kind"], 1 / math.sqrt(case["d"])
    z, sp, delta = _delta64(case, x)
    if kind == "mask":
        return {"bias": delta[..., :L], "expiry": None, "bitmap": None}
    if kind in ("decode", "generate"):
        o = torch.zeros(_rows(case), B, Hq, d, dtype=torch.float64, device="cuda")
        lse = torch.zeros(_rows(case), B * Hq, dtype=torch.float64, device="cuda")
        for t in range(_rows(case)):
            n = L + (t + 1 if kind == "generate" else 0)
            for b in range(B):
                for h in range(Hq):
                    sel = torch.sort(delta[b, h, :n], descending=True, stable=True)[1][:w]
                    K, V = x["K"][b, sel, h // G].double(), x["V"][b, sel, h // G].double()
                    s = K @ x["Q"][t, b, h].double() * scale + delta[b, h, sel]
                    lse[t, b * Hq + h] = torch.logsumexp(s, 0)
                    o[t, b, h] = torch.softmax(s, 0) @ V
        return {"o": o, "lse": lse}
    ex = _expiry64(case, delta.cpu(), _cu(case, seed))
    rows, train = _rows(case), kind == "train"
    q0, j = L - rows, torch.arange(L, device="cuda")
    O = torch.zeros(B, rows, Hq, d, dtype=torch.float64, device="cuda")
    lse = torch.zeros(B, Hq, rows, dtype=torch.float64, device="cuda")
    dQ, dK, dV = (torch.zeros_like(x[k], dtype=torch.float64) if train else None for k in ("Q", "K", "V"))
    dM = torch.zeros(B, Hq, L, dtype=torch.float64, device="cuda")
    step = max(64, min(rows, (1 << 27) // L))
    for b in range(B):
        for h in range(Hq):
            K, V, Q = x["K"][b, :L, h // G].double(), x["V"][b, :L, h // G].double(), x["Q"][b, :, h].double()
            for r in range(0, rows, step):
                i = torch.arange(q0 + r, q0 + min(rows, r + step), device="cuda")[:, None]
                n = int(i[-1]) + 1 if case["causal"] else L
                q, hide = Q[r:r + step], i >= ex[b, h, :n]
                if case["causal"]:
                    hide |= j[:n] > i
                P = (q @ K[:n].T).mul_(scale).add_(delta[b, h, :n]).masked_fill_(hide, -math.inf)
                lse[b, h, r:r + step] = torch.logsumexp(P, 1)
                P.sub_(lse[b, h, r:r + step, None]).exp_()
                o = O[b, r:r + step, h] = P @ V[:n]
                if train:
                    do = x["dO"][b, r:r + step, h].double()
                    dV[b, :n, h // G] += P.T @ do
                    dS = (do @ V[:n].T).sub_((do * o).sum(1, keepdim=True)).mul_(P)
                    dM[b, h, :n] += dS.sum(0)
                    dQ[b, r:r + step, h] = dS @ K[:n] * scale
                    dK[b, :n, h // G] += dS.T @ q * scale
    if not train:
        return {"O": O, "lse": lse}
    g = dM * delta[..., :L]
    dA = (g * sp[..., :L]).sum((0, 2))
    dz = g * x["A"].double()[None, :, None] * torch.sigmoid(z[..., :L])
    V, W = x["V"].double(), x["W"].double()
    if case["full"]:
        dW = torch.einsum("bhj,bjc->hc", dz, V.reshape(B, L, Hkv * d))
        dV += torch.einsum("bhj,hc->bjc", dz, W).view(B, L, Hkv, d)
    else:
        dz, Wg = dz.view(B, Hkv, G, L), W.view(Hkv, G, d)
        dW = torch.einsum("bkgj,bjkc->kgc", dz, V).reshape(Hq, d)
        dV += torch.einsum("bkgj,kgc->bjkc", dz, Wg)
    return {"O": O, "lse": lse, "dQ": dQ, "dK": dK, "dV": dV, "dW": dW, "dA": dA}
