"""GPU parity of the attention forward (Sec. 4.2) and backward (Sec. 4.3) against the CPU oracle (fp64
instantiation, fed the same rounded inputs), through the C-ABI."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import workloads as wl

from helpers import assert_close, f64, gpu_run, oracle_mask, problem_of, round_to, stored_forward

pytestmark = pytest.mark.gpu

C1, C2 = wl.CONFIGS["1"], wl.CONFIGS["2"]
CASES = [
    C1,
    wl.small(C1, L=1, w=1, name="fp32 L1"),
    wl.small(C1, L=77, w=200, name="fp32 w>=L ragged"),
    wl.small(C1, B=2, d=128, Hq=4, Hkv=2, L=321, w=50, name="fp32 d128 gqa ragged"),
    wl.small(C2, B=2, Hq=4, Hkv=2, L=1000, w=129, backward=True, name="bf16 ragged gqa"),
    wl.small(C2, B=1, Hq=8, Hkv=2, L=1024, w=256, backward=True, name="bf16 L1024"),
    wl.small(C2, B=1, Hq=2, Hkv=1, L=640, w=1, backward=True, name="bf16 w=1"),
    wl.small(C2, B=1, Hq=2, Hkv=2, L=130, w=999, backward=True, name="bf16 dense-causal"),
    wl.small(C2, B=1, Hq=4, Hkv=4, L=512, w=64, d=64, backward=True, name="bf16 d64"),
    wl.small(C2, B=1, Hq=4, Hkv=1, L=1536, w=200, backward=True, qk_scale=3.0, name="bf16 peaked"),
    # d = 64: the backward alternates between two P / dS buffers; schedules of one, two, three and five 64-row steps per CTA
    wl.small(C2, B=1, Hq=1, Hkv=1, L=64, w=16, d=64, backward=True, name="bf16 d64 one step"),
    wl.small(C2, B=2, Hq=2, Hkv=2, L=100, w=30, d=64, backward=True, name="bf16 d64 two steps"),
    wl.small(C2, B=1, Hq=2, Hkv=1, L=129, w=500, d=64, backward=True, name="bf16 d64 gqa three steps"),
    wl.small(C2, B=1, Hq=6, Hkv=2, L=300, w=41, d=64, backward=True, name="bf16 d64 group of 3 ragged"),
]


def oracle_all(case, inp, bias, e, backward=True):
    Q, K, V, dO = (f64(inp[k]) for k in ("Q", "K", "V", "dO"))
    O, lse = oracle.forward(Q, K, V, bias.astype(np.float64), expiry=e)
    out = {"O": O, "lse": lse}
    if backward:
        # Alg. 2 reads the stored forward output: D uses O rounded to the element type
        dQ, dK, dV, dM = oracle.backward(Q, K, V, dO, bias.astype(np.float64), expiry=e, O=round_to(case, O))
        out.update(dQ=dQ, dK=dK, dV=dV, dM=dM)
    return out


def compare(case, got, ref, backward=True, end_to_end=False):
    """end_to_end: the GPU backward read the GPU forward's own stored O (dma_step_host cannot be handed another), which
    differs from the oracle's stored O wherever the two forwards round an element to different neighbours; D = rowsum(dO o O)
    of Alg. 2 carries those one-ulp differences into every dS of the row, so the gradients are held to the bound relative
    to the tensor's largest magnitude there. Everywhere else both backward passes read the same stored O and the
    per-row / per-head bounds apply."""
    assert_close(got["O"], ref["O"], case.dtype, "O")
    assert_close(got["lse"], ref["lse"], case.dtype, "lse", lse=True)
    if backward:
        for k in ("dQ", "dK", "dV", "dM"):
            assert_close(got[k], ref[k], case.dtype, k, kind="tensor" if end_to_end else None)


@pytest.mark.parametrize("case", CASES, ids=lambda c: c.name)
def test_forward_backward_small(case):
    inp = wl.make_inputs(case)
    dl, e, bmp = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])          # both backward passes read the same stored forward output
    got = gpu_run(case, inp, stored=st)
    assert np.array_equal(got["expiry"].cpu().numpy(), e)
    compare(case, got, ref)
    # block skipping is an optimisation only: ignoring the bitmap must give the same result
    again = gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_IGNORE_BITMAP)
    compare(case, again, ref)


@pytest.mark.parametrize("case", [c for c in CASES if c.dtype == "bf16"], ids=lambda c: c.name)
def test_cuda_core_kernels_on_bf16(case):
    inp = wl.make_inputs(case)
    dl, e, bmp = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    compare(case, gpu_run(case, inp, stored=stored_forward(case, ref["O"], ref["lse"]), flags=dma.DMA_FLAG_SIMT), ref)


def test_injected_mask_zero_bias_is_dense_causal_attention():
    # any self-consistent (bias, expiry, bitmap) is accepted: zero bias + everything kept = textbook causal attention
    case = wl.small(C2, B=1, Hq=4, Hkv=2, L=700, w=700, backward=True, name="inject")
    inp = wl.make_inputs(case)
    B, Hq, L = case.B, case.Hq, case.L
    bias = np.zeros((B, Hq, L), np.float32)
    e = np.full((B, Hq, L), L, np.int32)
    bmp = oracle.bitmap_from_expiry(e).view(np.int32)
    ref_all = oracle_all(case, inp, bias, e)
    got = gpu_run(case, inp, mask=(bias, e, bmp), stored=stored_forward(case, ref_all["O"], ref_all["lse"]))
    q, k, v = (inp[n].double().permute(0, 2, 1, 3) for n in ("Q", "K", "V"))
    G = Hq // case.Hkv
    ref = torch.nn.functional.scaled_dot_product_attention(q, k.repeat_interleave(G, 1), v.repeat_interleave(G, 1), is_causal=True)
    assert_close(got["O"], ref.permute(0, 2, 1, 3).numpy(), "bf16", "O vs SDPA")
    compare(case, got, ref_all)


def test_skipped_tiles_do_not_change_the_result_on_a_banded_mask():
    # structured workload at reduced length: many inactive tiles
    case = wl.small(wl.CONFIGS["S"], L=2048, w=256, Hq=6, Hkv=2, name="S-small")
    inp = wl.make_inputs(case)
    dl, e, bmp = oracle_mask(case, inp)
    T = case.L // 128
    t = np.arange(T)
    active = ((bmp[..., t // 32] >> (t % 32)) & 1).sum()
    assert active < 0.8 * case.B * case.Hq * T * (T + 1) / 2           # the mask really has holes
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    compare(case, gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_TILE_PATH), ref)
    compare(case, gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_IGNORE_BITMAP), ref)


def dq_rows(case):
    """Sampled query rows for dQ: the dense-causal region (rows below w keep every visible key) AND the region where
    the mask drops keys (rows at and beyond w), including both sides of a tile boundary and the last row."""
    L, w = case.L, min(case.w, case.L)
    rows = [0, 5, 130, min(700, L - 1), w - 1, min(w, L - 1), min(w + 1, L - 1), L // 2, (L // 2) | 1, 3 * L // 4 + 77,
            L - 129, L - 128, L - 1]
    return np.unique(np.clip(np.array(rows, np.int64), 0, L - 1)).astype(np.int32)


class Samples:
    """Full-size parity on sampled outputs: query rows (O, lse, dQ) and keys (dK, dV, dM) that the oracle evaluates one
    by one, computed BEFORE the GPU runs. Keys are sampled near the end of the sequence, where only the last 600 rows can
    keep them; dQ rows cover the region where the mask drops keys. `stored` holds the oracle's forward output on every
    row the sampled gradients depend on: the GPU backward is given those rows as its stored O / lse (Alg. 2 takes them
    as inputs), so both backward passes work from the same values."""

    def __init__(self, case, inp, nrows=24, nkeys=6, seed=0, forward_only=False):
        rng = np.random.default_rng(seed)
        self.case, self.inp = case, inp
        self.backward = case.backward and not forward_only
        self.dl, self.e, _ = oracle_mask(case, inp)
        Q, K, V, dO = (f64(inp[k]) for k in ("Q", "K", "V", "dO"))
        L, bias = case.L, self.dl.astype(np.float64)
        rows = np.concatenate([[0, 1, 127, 128, L - 1], rng.integers(0, L, nrows)])
        if self.backward:
            self.keys = np.unique(np.concatenate([[L - 1, L - 130], rng.integers(L - 600, L, nkeys)])).astype(np.int32)
            tail = np.arange(L - 600, L)                             # the only rows that can keep those keys
            self.dq = dq_rows(case)
            rows = np.concatenate([rows, tail, self.dq])
        self.rows = np.unique(rows).astype(np.int32)
        self.O, self.lse = oracle.forward(Q, K, V, bias, expiry=self.e, rows=self.rows)
        self.stored = stored_forward(case, self.O, self.lse, rows=self.rows)
        if self.backward:
            Ostored = np.zeros_like(Q)
            Ostored[:, self.rows] = self.stored["O"]                 # Alg. 2 reads the stored (rounded) forward output
            _, self.dK, self.dV, self.dM = oracle.backward(Q, K, V, dO, bias, expiry=self.e, keys=self.keys, want_dq=False, O=Ostored)
            at = np.searchsorted(self.rows, self.dq)
            self.dQ = oracle.backward_dq_rows(Q, K, V, dO, bias, self.dq, expiry=self.e, O=self.stored["O"][:, at])

    def check(self, got, tag=""):
        case = self.case
        assert_close(got["O"][:, self.rows], self.O, case.dtype, tag + "O rows")
        assert_close(got["lse"][:, :, self.rows], self.lse, case.dtype, tag + "lse rows", lse=True)
        if not self.backward:
            return
        assert_close(got["dK"][:, self.keys], self.dK, case.dtype, tag + "dK keys")
        assert_close(got["dV"][:, self.keys], self.dV, case.dtype, tag + "dV keys")
        assert_close(got["dM"][:, :, self.keys], self.dM, case.dtype, tag + "dM keys")
        assert_close(got["dQ"][:, self.dq], self.dQ, case.dtype, tag + "dQ rows")
        # properties that hold at any size (Sec. 4.3): rows of dS sum to zero; q.dQ and k.dK balance per KV group
        # (D is formed from the stored, rounded O, so each row of dS sums to dO_i.(O_i - stored O_i), at most
        # half a bf16 ulp of every |dO_ic O_ic| term; in fp32 the bound is the accumulation error)
        Q, K, dO = (f64(self.inp[k]) for k in ("Q", "K", "dO"))
        L = case.L
        dMs = f64(got["dM"]).sum(-1)
        half_ulp = 2.0 ** -9 if case.dtype == "bf16" else 2.0 ** -20
        bound = half_ulp * (np.abs(dO) * np.abs(f64(got["O"]))).sum((1, 3)) + 1e-3
        assert (np.abs(dMs) <= bound).all(), (dMs, bound)
        G = case.Hq // case.Hkv
        lhs = (Q * f64(got["dQ"])).sum(-1).reshape(case.B, L, case.Hkv, G).sum((1, 3))
        rhs = (K * f64(got["dK"])).sum(-1).sum(1)
        assert np.abs(lhs - rhs).max() <= 2e-2 * max(1.0, np.abs(rhs).max())


@pytest.mark.parametrize("key", ["2", "3", "3x3", "4w256", "4w2048", "4w8192", "5", "S"])
def test_full_size_configs_sampled(key):
    case = wl.CONFIGS[key]
    inp = wl.make_inputs(case)
    ref = Samples(case, inp)
    # the tile-walking kernels (Alg. 1 / Alg. 2 with block skipping)
    ref.check(gpu_run(case, inp, backward=case.backward, stored=ref.stored, flags=dma.DMA_FLAG_TILE_PATH))


def test_default_flags_choose_the_path_from_the_descriptor():
    """Without DMA_FLAG_COMPACT_KV / DMA_FLAG_TILE_PATH the library picks token-compacted execution for causal bf16 problems
    with L >= 2048 and 4 w <= L and the tile-walking kernels otherwise: O and lse are the bits of the explicitly chosen path,
    the injected over-full mask is reported (DMA_ERR_MASK_OVERFLOW) instead of being truncated silently."""
    dev = torch.device("cuda:0")
    for key, chosen in (("4w2048", dma.DMA_FLAG_COMPACT_KV), ("4w4096", dma.DMA_FLAG_TILE_PATH)):
        case = wl.small(wl.CONFIGS[key], Hq=4, Hkv=4, name="auto " + key)
        inp = wl.make_inputs(case)
        a, b = gpu_run(case, inp, backward=False), gpu_run(case, inp, backward=False, flags=chosen)
        assert torch.equal(a["O"], b["O"]) and torch.equal(a["lse"], b["lse"]), key
        sizes = [dma.dma_query_workspace(problem_of(case, flags=f)) for f in (0, chosen)]
        assert sizes[0] == sizes[1], key
    # a mask that keeps every visible key, declared with w = 64: the gathered lists (w + 256 entries) overflow
    case = wl.small(C2, B=1, Hq=2, Hkv=1, L=2048, w=64, name="overfull")
    inp = wl.make_inputs(case)
    p = problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV)
    e = torch.full((1, 2, case.L), case.L, dtype=torch.int32, device=dev)
    bias = torch.zeros(1, 2, case.L, dtype=torch.float32, device=dev)
    bmp = torch.from_numpy(oracle.bitmap_from_expiry(e.cpu().numpy()).view(np.int32)).to(dev)
    ws = torch.empty(dma.dma_query_workspace(p)[1], dtype=torch.uint8, device=dev)
    dma.dma_attn_fwd(p, inp["Q"].to(dev), inp["K"].to(dev), inp["V"].to(dev), bias, e, bmp, ws=ws)
    assert dma.dma_read_status(ws) == -8


def test_mma_block_skipping_does_not_change_the_result():
    """With DMA_FLAG_BLOCK_SKIP the P V product of an executed tile leaves out the 16-key MMA blocks in which no key can be
    kept by the query tile's rows. P is exactly zero there, so O and lse must be the bits of the run with every block
    multiplied, on masks that really have such blocks: a banded importance
    pattern, packed documents whose boundaries fall inside key tiles, and the gathered lists of the token-compacted kernels.
    The same outputs are held to the oracle in the tests above."""
    dev = torch.device("cuda:0")
    banded = wl.small(wl.CONFIGS["S"], L=4096, w=200, Hq=6, Hkv=2, backward=False, name="block-skip banded")
    packed = wl.small(C2, B=1, Hq=4, Hkv=2, L=3000, w=300, backward=False, name="block-skip packed")
    for case, cu in ((banded, None), (packed, [0, 70, 1000, 1111, 1900, 2500, 3000])):
        inp = wl.make_inputs(case)
        Q, K, V = (inp[k].to(dev) for k in ("Q", "K", "V"))
        p0 = problem_of(case, flags=dma.DMA_FLAG_TILE_PATH)
        if cu is None:
            mask = dma.dma_mask_build(p0, V, inp["W_delta"].to(dev), inp["A"].to(dev))
        else:
            mask = dma.dma_mask_build_varlen(p0, V, inp["W_delta"].to(dev), inp["A"].to(dev), torch.tensor(cu, dtype=torch.int32, device=dev))
        # the mask must contain dead 16-key blocks inside active tiles, or the test checks nothing
        e = mask[1].cpu().numpy()
        bmp = mask[2].cpu().numpy().view(np.uint32)
        dead_blocks = 0
        for qt in range(case.L // 128):
            for kt in range(qt):                                                   # off-diagonal tiles: a key is dead iff it expired before the tile's rows
                if (bmp[0, 0, qt, kt // 32] >> np.uint32(kt % 32)) & np.uint32(1):
                    blk = (e[0, 0, kt * 128:(kt + 1) * 128].reshape(8, 16) <= qt * 128).all(1)
                    dead_blocks += int(blk.sum())
        assert dead_blocks > 0, case.name
        for path in (dma.DMA_FLAG_TILE_PATH, dma.DMA_FLAG_COMPACT_KV):
            outs = []
            for extra in (dma.DMA_FLAG_BLOCK_SKIP, 0):
                p = problem_of(case, flags=path | extra)
                ws = torch.empty(dma.dma_query_workspace(p)[1], dtype=torch.uint8, device=dev)
                outs.append(dma.dma_attn_fwd(p, Q, K, V, *mask, ws=ws))
                assert dma.dma_read_status(ws) == 0
            assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1]), (case.name, path)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("path", [dma.DMA_FLAG_TILE_PATH, dma.DMA_FLAG_COMPACT_KV])
def test_mma_block_skipping_leaves_dead_blocks_out(path, d):
    """Infinite value rows of 16 keys that the last query tile's rows no longer keep, one MMA block of an active tile and of the gathered list:
    a product over that block would be 0 x inf."""
    dev = torch.device("cuda:0")
    case = wl.small(C2, B=1, Hq=1, Hkv=1, L=512, w=512, d=d, backward=False, name="block-skip infinite")
    inp = wl.make_inputs(case)
    e = torch.full((1, 1, 512), 512, dtype=torch.int32)
    e[0, 0, :16], e[0, 0, 16] = 384, 17                       # (240 keys are kept by all rows of the second pair of tiles: the 16 are a block of its list)
    bmp = torch.from_numpy(oracle.bitmap_from_expiry(e.numpy()).view(np.int32)).to(dev)
    bias = torch.zeros(1, 1, 512)
    V = inp["V"].clone()
    V[:, :16] = float("inf")
    p = problem_of(case, flags=path | dma.DMA_FLAG_BLOCK_SKIP)
    ws = torch.empty(dma.dma_query_workspace(p)[1], dtype=torch.uint8, device=dev)
    O, lse = dma.dma_attn_fwd(p, inp["Q"].to(dev), inp["K"].to(dev), V.to(dev), bias.to(dev), e.to(dev), bmp, ws=ws)
    assert dma.dma_read_status(ws) == 0
    rows = np.arange(384, 512, dtype=np.int32)
    Or, lr = oracle.forward(*(f64(inp[k]) for k in ("Q", "K", "V")), f64(bias), expiry=e.numpy(), rows=rows)
    assert_close(O[:, 384:], Or, case.dtype, "O")
    assert_close(lse[:, :, 384:], lr, case.dtype, "lse", lse=True)


def test_largest_supported_lengths():
    """The longest sequences the tensor-core kernels take: L = 131072 (1024 key tiles, the forward schedule's capacity; with
    a group of 4 query heads per KV head also the capacity of the backward's step list), forward and backward, tile path and
    token-compacted. Sampled rows and keys against the oracle, dQ on rows where the mask drops keys."""
    case = wl.small(wl.CONFIGS["3"], B=1, Hq=4, Hkv=1, L=131072, w=2048, backward=True, name="max L")
    inp = wl.make_inputs(case)
    ref = Samples(case, inp, nrows=8, nkeys=4)
    got = gpu_run(case, inp, stored=ref.stored, flags=dma.DMA_FLAG_TILE_PATH)
    ref.check(got)
    ref.check(gpu_run(case, inp, stored=ref.stored, flags=dma.DMA_FLAG_COMPACT_KV), "compact ")
    with pytest.raises(dma.DmaError) as e:                        # one tile more is refused, not mis-executed
        too_long = wl.small(case, L=131072 + 128)
        dma.dma_attn_fwd(problem_of(too_long, flags=dma.DMA_FLAG_TILE_PATH), got["O"], got["O"], got["O"], got["bias"], got["expiry"], got["bitmap"])
    assert e.value.status == -4
    with pytest.raises(dma.DmaError) as e:                        # eight heads per KV head at this length: the tile path's step list is too short
        wide = problem_of(wl.small(case, Hq=8), flags=dma.DMA_FLAG_TILE_PATH)
        ws = torch.empty(dma.dma_query_workspace(wide)[2], dtype=torch.uint8, device="cuda:0")
        dma.dma_attn_bwd(wide, got["O"], got["O"], got["O"], got["O"], got["O"], got["lse"], got["bias"], got["expiry"], got["bitmap"], ws=ws)
    assert e.value.status == -4


def test_whole_step_can_be_captured_in_a_cuda_graph():
    """The stream entry points only enqueue work (no allocation, no synchronisation): mask build, forward and backward are
    captured once and replayed; the replay reproduces the eager results."""
    dev = torch.device("cuda:0")
    case = wl.small(C2, B=1, Hq=8, Hkv=2, L=1024, w=256, backward=True, name="graph")
    inp = wl.make_inputs(case)
    eager = gpu_run(case, inp)
    p = problem_of(case)
    Q, K, V, dO = (inp[k].to(dev) for k in ("Q", "K", "V", "dO"))
    W, A = inp["W_delta"].to(dev), inp["A"].to(dev)
    m_ws, f_ws, b_ws = (torch.empty(n, dtype=torch.uint8, device=dev) for n in dma.dma_query_workspace(p))
    bias, expiry, bitmap = (torch.empty_like(eager[k]) for k in ("bias", "expiry", "bitmap"))
    O, lse = torch.empty_like(eager["O"]), torch.empty_like(eager["lse"])
    dQ, dK, dV, dM = (torch.empty_like(eager[k]) for k in ("dQ", "dK", "dV", "dM"))
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dma.dma_mask_build(p, V, W, A, bias, expiry, bitmap, m_ws)
        dma.dma_attn_fwd(p, Q, K, V, bias, expiry, bitmap, O, lse, f_ws)
        dma.dma_attn_bwd(p, Q, K, V, O, dO, lse, bias, expiry, bitmap, dQ, dK, dV, dM, b_ws)
    for _ in range(2):
        for t in (bias, expiry, bitmap, O, lse, dQ, dK, dV, dM):
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert dma.dma_read_status(f_ws) == 0 and dma.dma_read_status(b_ws) == 0
        for k, t in (("bias", bias), ("expiry", expiry), ("bitmap", bitmap), ("O", O), ("lse", lse), ("dK", dK), ("dV", dV)):
            assert torch.equal(t, eager[k]), k
        assert_close(dQ, f64(eager["dQ"]), case.dtype, "dQ (replayed)")        # atomics: order-dependent rounding
        assert_close(dM, f64(eager["dM"]), case.dtype, "dM (replayed)")


def test_bounded_wait_reports_timeout_and_context_survives():
    # a wait that nothing satisfies gives up after its limit and leaves a status, instead of hanging the GPU
    dev = torch.device("cuda:0")
    ws = torch.zeros(256, dtype=torch.uint8, device=dev)
    dma.dma_selftest_wait_timeout(ws)
    assert dma.dma_read_status(ws) == -7
    # the context is still usable and a normal call leaves a clean status
    case = wl.small(C2, B=1, Hq=2, Hkv=1, L=256, w=64, backward=False, name="after-timeout")
    inp = wl.make_inputs(case)
    got = gpu_run(case, inp, backward=False)
    assert torch.isfinite(got["O"].float()).all()


# ---- token-compacted forward (DMA_FLAG_COMPACT_KV): same results as the oracle, from the gathered key lists ----------

def _compact_run(case, inp):
    dev = torch.device("cuda:0")
    p = problem_of(case)
    pc = problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV)
    Q, K, V = (inp[k].to(dev) for k in ("Q", "K", "V"))
    bias, expiry, bitmap = dma.dma_mask_build(p, V, inp["W_delta"].to(dev), inp["A"].to(dev))
    ws = torch.empty(dma.dma_query_workspace(pc)[1], dtype=torch.uint8, device=dev)
    O, lse = dma.dma_attn_fwd(pc, Q, K, V, bias, expiry, bitmap, ws=ws)
    torch.cuda.synchronize()
    assert dma.dma_read_status(ws) == 0
    return {"bias": bias, "expiry": expiry, "bitmap": bitmap, "O": O, "lse": lse}


@pytest.mark.parametrize("kw", [
    dict(B=1, Hq=2, Hkv=1, L=384, w=64),            # ragged pair count (3 query tiles), small window
    dict(B=2, Hq=4, Hkv=2, L=1000, w=200),          # ragged tail rows, GQA
    dict(B=1, Hq=2, Hkv=2, L=1536, w=2000),         # w >= L: every causal key is gathered (dense causal attention)
    dict(B=1, Hq=4, Hkv=1, L=2048, w=1),            # w = 1: one key per row
])
def test_compact_forward_small_cases(kw):
    case = wl.small(C2, name="compact-small", backward=False, **kw)
    inp = wl.make_inputs(case)
    got = _compact_run(case, inp)
    dl, e, _ = oracle_mask(case, inp)                     # the oracle's own mask, not the GPU's
    assert np.array_equal(got["expiry"].cpu().numpy(), e)
    ref = oracle.forward(inp["Q"].double().numpy(), inp["K"].double().numpy(), inp["V"].double().numpy(),
                         dl.astype(np.float64), expiry=e, scale=case.d ** -0.5)
    assert_close(got["O"], ref[0], case.dtype, "compact O")
    assert_close(got["lse"], ref[1], case.dtype, "compact lse", lse=True)


@pytest.mark.parametrize("key", ["3", "S", "5"])
def test_compact_forward_full_size_sampled(key):
    case = wl.CONFIGS[key]
    inp = wl.make_inputs(case)
    Samples(case, inp, forward_only=True).check(_compact_run(case, inp), "compact ")


def test_compact_flag_is_rejected_where_unsupported():
    dev = torch.device("cuda:0")
    for case in (wl.small(C1, B=1, Hq=2, Hkv=1, L=256, w=64, d=128, name="compact-fp32"),
                 wl.small(C2, B=1, Hq=2, Hkv=1, L=256, w=64, d=64, name="compact-d64-cuda-cores")):
        inp = wl.make_inputs(case)
        flags = dma.DMA_FLAG_COMPACT_KV | (dma.DMA_FLAG_SIMT if case.dtype == "bf16" else 0)
        with pytest.raises(dma.DmaError) as e:
            gpu_run(case, inp, backward=False, flags=flags)
        assert e.value.status == -4


def test_bf16_d64_runs_on_the_tensor_core_kernels():
    """bf16 with 64 channels runs on the d = 64 instantiations of the tensor-core kernels (both paths): results against the
    oracle within the gate, on strided inputs too, nothing written outside the views."""
    dev = torch.device("cuda:0")
    case = wl.small(C2, B=2, Hq=4, Hkv=2, L=700, w=96, d=64, backward=True, name="d64-native")
    inp = wl.make_inputs(case)
    dl, e, _ = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    for flags in (0, dma.DMA_FLAG_COMPACT_KV):
        compare(case, gpu_run(case, inp, stored=st, flags=flags), ref)
    # strided Q / K / V / O views of wider buffers
    big = {k: torch.randn(case.B, case.L + 9, (case.Hq if k in ("Q", "dO") else case.Hkv) + 1, 64).to(case.torch_dtype).to(dev) for k in ("Q", "K", "V", "dO")}
    view = {k: big[k][:, 3:3 + case.L, 1:] for k in big}
    for k in view:
        view[k].copy_(inp[k].to(dev))
    p = problem_of(case)
    for sdst, t in ((p.q_stride, view["Q"]), (p.k_stride, view["K"]), (p.v_stride, view["V"]), (p.o_stride, view["dO"])):
        sdst[0], sdst[1], sdst[2] = t.stride(0), t.stride(1), t.stride(2)
    bias, expiry, bitmap = dma.dma_mask_build(p, view["V"], inp["W_delta"].to(dev), inp["A"].to(dev))
    Obuf = torch.zeros_like(big["dO"])
    O, lse = dma.dma_attn_fwd(p, view["Q"], view["K"], view["V"], bias, expiry, bitmap, O=Obuf[:, 3:3 + case.L, 1:])
    dQb, dKb, dVb = torch.zeros_like(big["Q"]), torch.zeros_like(big["K"]), torch.zeros_like(big["V"])
    Oin = torch.zeros_like(big["dO"])[:, 3:3 + case.L, 1:]                       # the oracle's stored O in the same strided layout
    Oin.copy_(torch.from_numpy(st["O"]).to(case.torch_dtype).to(dev))
    dQ, dK, dV, dM = dma.dma_attn_bwd(p, view["Q"], view["K"], view["V"], Oin, view["dO"], torch.from_numpy(st["lse"]).to(dev), bias, expiry, bitmap,
                                      dQ=dQb[:, 3:3 + case.L, 1:], dK=dKb[:, 3:3 + case.L, 1:], dV=dVb[:, 3:3 + case.L, 1:])
    torch.cuda.synchronize()
    compare(case, {"O": O, "lse": lse, "dQ": dQ, "dK": dK, "dV": dV, "dM": dM}, ref)
    assert float(Obuf[:, :3].abs().max()) == 0.0 and float(Obuf[:, :, 0].abs().max()) == 0.0
    assert float(dKb[:, :3].abs().max()) == 0.0 and float(dKb[:, :, 0].abs().max()) == 0.0


def test_compact_kernels_on_strided_k_and_v():
    """K and V living inside larger buffers (spare sequence capacity, extra heads between the used ones): the gathers follow
    the descriptor's strides; results equal those on packed copies of the same data."""
    dev = torch.device("cuda:0")
    case = wl.small(C2, B=2, Hq=4, Hkv=2, L=700, w=96, backward=True, name="compact-strided")
    inp = wl.make_inputs(case)
    ref = gpu_run(case, inp, flags=dma.DMA_FLAG_COMPACT_KV)
    B, L, Hkv, d = case.B, case.L, case.Hkv, case.d
    cap, Hbig = L + 52, 2 * Hkv + 1
    bigK = torch.randn(B, cap, Hbig, d).to(case.torch_dtype).to(dev)
    bigV = torch.randn(B, cap, Hbig, d).to(case.torch_dtype).to(dev)
    Kv, Vv = bigK[:, :L, 1:1 + 2 * Hkv:2], bigV[:, :L, 1:1 + 2 * Hkv:2]          # every other head, starting at head 1
    Kv.copy_(inp["K"].to(dev)); Vv.copy_(inp["V"].to(dev))
    p = problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV)
    for sdst, t in ((p.k_stride, Kv), (p.v_stride, Vv)):
        sdst[0], sdst[1], sdst[2] = t.stride(0), t.stride(1), t.stride(2)
    Q, dO = inp["Q"].to(dev), inp["dO"].to(dev)
    O, lse = dma.dma_attn_fwd(p, Q, Kv, Vv, ref["bias"], ref["expiry"], ref["bitmap"])
    dK, dV = torch.zeros_like(bigK), torch.zeros_like(bigV)
    dKv, dVv = dK[:, :L, 1:1 + 2 * Hkv:2], dV[:, :L, 1:1 + 2 * Hkv:2]
    dQ, _, _, dM = dma.dma_attn_bwd(p, Q, Kv, Vv, O, dO, lse, ref["bias"], ref["expiry"], ref["bitmap"], dK=dKv, dV=dVv)
    torch.cuda.synchronize()
    assert torch.equal(O, ref["O"]) and torch.equal(lse, ref["lse"])
    assert_close(dKv, f64(ref["dK"]), case.dtype, "dK (strided)")
    assert_close(dVv, f64(ref["dV"]), case.dtype, "dV (strided)")
    assert_close(dQ, f64(ref["dQ"]), case.dtype, "dQ (strided)")
    assert_close(dM, f64(ref["dM"]), case.dtype, "dM (strided)")
    untouched = torch.ones(Hbig, dtype=torch.bool); untouched[1:1 + 2 * Hkv:2] = False
    assert float(dK[:, :, untouched].abs().max()) == 0.0 and float(dK[:, L:].abs().max()) == 0.0


# ---- token-compacted backward (DMA_FLAG_COMPACT_KV): key tiles follow a lifetime-sorted permutation per query head -----

@pytest.mark.parametrize("case", [c for c in CASES if c.dtype == "bf16" and c.d == 128], ids=lambda c: c.name)
def test_compact_backward_small_cases(case):
    # the same small cases as the tile path (ragged tails and padding entries in the permutation, several query heads
    # adding into one KV head, w = 1 where almost every key is never kept, w >= L where nothing expires, peaked scores)
    inp = wl.make_inputs(case)
    dl, e, _ = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    got = gpu_run(case, inp, stored=stored_forward(case, ref["O"], ref["lse"]), flags=dma.DMA_FLAG_COMPACT_KV)
    assert np.array_equal(got["expiry"].cpu().numpy(), e)
    compare(case, got, ref)


def test_compact_backward_deterministic_option():
    """DMA_FLAG_DETERMINISTIC: the query heads of a group write dK / dV contributions to accumulators of their own, added in
    head order: the same bits from run to run (four heads per KV head here), and the same parity with the oracle."""
    case = wl.small(C2, B=2, Hq=8, Hkv=2, L=1100, w=150, backward=True, name="compact deterministic")
    inp = wl.make_inputs(case)
    dl, e, _ = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    flags = dma.DMA_FLAG_COMPACT_KV | dma.DMA_FLAG_DETERMINISTIC
    runs = [gpu_run(case, inp, stored=st, flags=flags) for _ in range(3)]
    compare(case, runs[0], ref)
    for r in runs[1:]:
        assert torch.equal(r["dK"], runs[0]["dK"]) and torch.equal(r["dV"], runs[0]["dV"])
    plain = gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_COMPACT_KV)
    assert_close(plain["dK"], f64(runs[0]["dK"]), case.dtype, "dK (atomic against ordered sums)")
    assert dma.dma_query_workspace(problem_of(case, flags=flags))[2] > dma.dma_query_workspace(problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV))[2]


@pytest.mark.parametrize("key", ["3", "4w256", "4w2048", "S"])
def test_compact_backward_full_size_sampled(key):
    case = wl.CONFIGS[key]
    inp = wl.make_inputs(case)
    ref = Samples(case, inp)
    ref.check(gpu_run(case, inp, stored=ref.stored, flags=dma.DMA_FLAG_COMPACT_KV), "compact ")


@pytest.mark.parametrize("B,Hq,Hkv,L,d,w", [(1, 1, 1, 7, 64, 3), (1, 2, 1, 9, 128, 9), (1, 3, 1, 64, 64, 20), (1, 1, 1, 65, 128, 1),
                                            (1, 2, 2, 129, 64, 200), (8, 20, 20, 33, 64, 10), (8, 20, 10, 40, 128, 40), (4, 16, 2, 97, 64, 31)])
def test_cuda_core_kernels_at_the_edges_of_their_tiles(B, Hq, Hkv, L, d, w):
    """fp32, 8-row CTAs (small grids) and 32-row CTAs: lengths around the warps' rows and the 64-row streamed tiles; causal against
    the oracle, and every gradient the same bits from run to run."""
    case = wl.small(C1, B=B, Hq=Hq, Hkv=Hkv, L=L, d=d, w=w, seed=L + d, name="edge")
    inp = wl.make_inputs(case)
    dl, e, bmp = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    got = gpu_run(case, inp, stored=st)
    compare(case, got, ref)
    again = gpu_run(case, inp, stored=st)
    assert all(torch.equal(got[k], again[k]) for k in ("O", "lse", "dQ", "dK", "dV", "dM"))


@pytest.mark.parametrize("B,Hq,Hkv,L,d", [(1, 6, 1, 300, 128), (1, 6, 1, 129, 64), (2, 8, 2, 640, 64), (1, 4, 4, 200, 128), (1, 12, 2, 1100, 128)])
def test_tile_backward_with_the_group_dealt_out_to_several_ctas(B, Hq, Hkv, L, d):
    """Short sequences: a KV head's query heads go to several CTAs (2, 3, 4 or 6 of them, or one), whose dK / dV parts are summed from
    slots: against the oracle, and dK, dV, dM the same bits from run to run."""
    case = wl.small(C2, B=B, Hq=Hq, Hkv=Hkv, L=L, d=d, w=L // 3, backward=True, seed=L + Hq, name="split")
    inp = wl.make_inputs(case)
    dl, e, bmp = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    got = gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_TILE_PATH)
    compare(case, got, ref)
    again = gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_TILE_PATH)
    assert all(torch.equal(got[k], again[k]) for k in ("dK", "dV", "dM"))


@pytest.mark.parametrize("Hq,L,w,q_begin", [(80, 1024, 100, 0), (148, 2050, 64, 0), (50, 3000, 700, 0), (80, 2052, 300, 1001)])
def test_gathered_lists_of_several_pairs_per_cta(Hq, L, w, q_begin):
    """Enough heads that a CTA makes the lists of 2, 4 or 8 pairs of query tiles (lengths with and without 16-byte aligned rows, a
    last group that is not full, a chunk that starts inside a pair): against the CUDA-core kernel on the same mask."""
    case = wl.small(C2, B=1, Hq=Hq, Hkv=Hq // 2, L=L, d=64, w=w, seed=L, name="lists")
    inp = {k: v.cuda() for k, v in wl.make_inputs(case).items()}
    p = problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV)
    bias, e, bmp = dma.dma_mask_build(p, inp["V"], inp["W_delta"], inp["A"])
    if q_begin:
        O, lse = dma.dma_attn_fwd_chunk(p, q_begin, inp["Q"][:, q_begin:].contiguous(), inp["K"], inp["V"], bias, e)
    else:
        O, lse = dma.dma_attn_fwd(p, inp["Q"], inp["K"], inp["V"], bias, e, bmp)
    ref_O, ref_lse = dma.dma_attn_fwd(problem_of(case, flags=dma.DMA_FLAG_SIMT), inp["Q"], inp["K"], inp["V"], bias, e, bmp)
    assert_close(O, f64(ref_O[:, q_begin:]), "bf16", "O")
    assert_close(lse, f64(ref_lse[..., q_begin:]), "bf16", "lse", lse=True)


@pytest.mark.parametrize("Hq", [2, 148])
def test_compact_forward_bits_do_not_depend_on_how_the_lists_were_made(Hq):
    """The gathered lists are ascending within their two parts whatever the length's alignment (2048 keys: 16-byte loads, 2049:
    scalar ones) and the pairs per CTA (2 heads: one, 148 heads: eight), so the same rows round the same way: O, lse bit for bit."""
    L, d, w = 2048, 64, 300
    case = wl.small(C2, B=1, Hq=Hq, Hkv=Hq // 2, L=L + 1, d=d, w=w, seed=7, name="list-order")
    inp = {k: v.cuda() for k, v in wl.make_inputs(case).items()}
    p = dma.problem(1, Hq, Hq // 2, L, d, w, flags=dma.DMA_FLAG_COMPACT_KV)
    Q, K, V = (inp[k][:, :L].contiguous() for k in ("Q", "K", "V"))
    bias, e, bmp = dma.dma_mask_build(p, V, inp["W_delta"], inp["A"])
    O, lse = dma.dma_attn_fwd(p, Q, K, V, bias, e, bmp)
    # one pair per call: group 1
    for i in range(0, L, 512):
        Oc, lc = dma.dma_attn_fwd_chunk(p, i, Q[:, i:i + 256].contiguous(), K, V, bias, e)
        assert torch.equal(Oc, O[:, i:i + 256]) and torch.equal(lc, lse[..., i:i + 256]), i
    # one key more, kept by its own row alone
    p1 = problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV)
    bias1, e1 = torch.ones(1, Hq, L + 1, device="cuda"), torch.full((1, Hq, L + 1), L + 1, dtype=torch.int32, device="cuda")
    bias1[..., :L], e1[..., :L] = bias, e
    bmp1 = torch.full((dma.dma_bitmap_words(p1),), -1, dtype=torch.int32, device="cuda")
    O1, lse1 = dma.dma_attn_fwd(p1, inp["Q"], inp["K"], inp["V"], bias1, e1, bmp1)
    assert torch.equal(O1[:, :L], O) and torch.equal(lse1[..., :L], lse)


def test_overflow_of_gathered_lists_made_for_several_pairs():
    """148 heads of 4096 rows: eight pairs of query tiles per CTA. A mask that keeps every key where w promises 64 is reported, both
    where a pair's own list overflows (rows 256 on) and where the keys of the whole group do not fit (rows 2048 on); the next call
    with the same workspace, on a mask within w, is clean."""
    Hq, L, d, w = 148, 4096, 64, 64
    case = wl.small(C2, B=1, Hq=Hq, Hkv=Hq // 2, L=L, d=d, w=w, seed=3, name="list-overflow")
    inp = {k: v.cuda() for k, v in wl.make_inputs(case).items()}
    p = problem_of(case, flags=dma.DMA_FLAG_COMPACT_KV)
    bias, e, _ = dma.dma_mask_build(p, inp["V"], inp["W_delta"], inp["A"])
    ws = torch.empty(dma.dma_query_workspace(p)[1], dtype=torch.uint8, device="cuda")
    forward = lambda q0, rows, ex: dma.dma_attn_fwd_chunk(p, q0, inp["Q"][:, q0:q0 + rows].contiguous(), inp["K"], inp["V"], bias, ex, ws=ws)   # noqa: E731
    want = forward(0, L, e)
    assert dma.dma_read_status(ws) == 0
    dense = torch.full_like(e, L)
    for q0, rows in ((0, L), (0, 2048), (2048, 2048)):
        forward(q0, rows, dense)
        assert dma.dma_read_status(ws) == -8, (q0, rows)
        got = forward(0, L, e)
        assert dma.dma_read_status(ws) == 0
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_fp32_backward_of_more_heads_than_a_grid_has_rows():
    """32 768 query heads that share no KV head: with as many KV heads the dK / dV and dQ parts together are 65 536 heads, one more
    than a grid has rows. Against plain torch in 64 bits; every gradient of every head (8 keys, all kept)."""
    H, L, d = 32768, 8, 64
    g = torch.Generator("cuda").manual_seed(5)
    Q, K, V, dO = (torch.randn(1, L, H, d, generator=g, device="cuda") for _ in range(4))
    p = dma.problem(1, H, H, L, d, L, dtype=torch.float32)
    bias, e, bmp = dma.dma_mask_build(p, V, torch.zeros(H, d, device="cuda"), torch.ones(H, device="cuda"))
    O, lse = dma.dma_attn_fwd(p, Q, K, V, bias, e, bmp)
    got = dma.dma_attn_bwd(p, Q, K, V, O, dO, lse, bias, e, bmp)
    q, k, v, go = (t[0].transpose(0, 1).double() for t in (Q, K, V, dO))                 # [H, L, d]
    hide = torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1)
    pr = torch.softmax((q @ k.mT / d ** 0.5 + bias[0, :, None].double()).masked_fill(hide, float("-inf")), -1)
    ds = pr * (go @ v.mT - (go * (pr @ v)).sum(-1, keepdim=True))
    ref = [ds @ k / d ** 0.5, ds.mT @ q / d ** 0.5, pr.mT @ go]
    for name, a, r in zip(("dQ", "dK", "dV"), got, ref):
        assert_close(a, r.transpose(0, 1)[None].cpu().numpy(), "fp32", name)
    assert_close(got[3], ds.sum(1)[None].cpu().numpy(), "fp32", "dM")


@pytest.mark.parametrize("L,d", [(3000, 64), (3072, 128), (3071, 128)])
def test_tile_backward_of_long_problems_is_the_batch_entries_on_their_own(L, d):
    """Eight batch entries take the backward's instance for long problems, each of them alone the one for short problems: dK, dV, dM are
    the same bits, dQ (atomic sums in fp32) agrees to its rounding to bf16."""
    B, H = 8, 8
    case = wl.small(C2, B=B, Hq=H, Hkv=H, L=L, d=d, w=L // 2, seed=L, name="long-tile-bwd")
    inp = {k: v.cuda() for k, v in wl.make_inputs(case).items()}
    p = problem_of(case, flags=dma.DMA_FLAG_TILE_PATH)
    Q, K, V, dO = (inp[k] for k in ("Q", "K", "V", "dO"))
    bias, e, bmp = dma.dma_mask_build(p, V, inp["W_delta"], inp["A"])
    O, lse = dma.dma_attn_fwd(p, Q, K, V, bias, e, bmp)
    whole = dma.dma_attn_bwd(p, Q, K, V, O, dO, lse, bias, e, bmp)
    p1 = dma.problem(1, H, H, L, d, L // 2, flags=dma.DMA_FLAG_TILE_PATH)
    words = dma.dma_bitmap_words(p1)
    for b in (0, 3, B - 1):
        one = lambda t: t[b:b + 1].contiguous()   # noqa: E731
        part = dma.dma_attn_bwd(p1, one(Q), one(K), one(V), one(O), one(dO), one(lse), one(bias), one(e), bmp.flatten()[b * words:(b + 1) * words].contiguous())
        for name, x, y in zip(("dQ", "dK", "dV", "dM"), whole, part):
            x = x[b:b + 1]
            if name == "dQ":
                # two fp32 sums of the same L / 32 terms in another order: L / 32 roundings of partial sums, bounded by the largest
                # element of the tensor; where they fall on two sides of a rounding boundary the bf16 values are a whole spacing,
                # up to 2^-7 of the element, apart
                x, y = x.float(), y.float()
                assert ((x - y).abs() <= 2.0 ** -7 * torch.maximum(x.abs(), y.abs()) + 2.0 ** -24 * L / 32 * y.abs().max()).all(), b
            else:
                assert torch.equal(x, y), (name, b)
