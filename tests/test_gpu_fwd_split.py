"""GPU parity of the forward whose CTAs own one query tile and deal its key tiles out to both softmax groups (small grids take it)
against the oracle: one key tile (the second group has none), two, odd and even numbers, ragged ends, tiles with few and with many
keys expiring, token-compacted lists and chunks of rows. And against the kernel with two query tiles per CTA, which the same problem takes
when enough batch entries share the call: the same bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import workloads as wl
from helpers import assert_close, f64, gpu_mask, oracle_mask

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


SHAPES = [(1, 1, 0), (5, 2, 0), (128, 128, 0), (129, 40, 0), (256, 256, 0), (300, 30, 0), (640, 500, 0), (897, 64, 0),
          (2050, 100, 0), (2305, 512, 0), (700, 90, 1), (1000, 128, 129), (2500, 300, 250)]


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("L,w,rows", SHAPES)
def test_one_query_tile_per_cta(L, w, rows, d):
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=2, Hkv=1, L=L, w=w, d=d, name=f"one tile L{L} w{w} d{d}")
    inp = wl.make_inputs(case)
    p, bias, expiry, bitmap = gpu_mask(case, inp)
    dl, e, _ = oracle_mask(case, inp)
    assert np.array_equal(expiry.cpu().numpy(), e)
    Q, K, V = (inp[k].to(DEV) for k in ("Q", "K", "V"))
    if rows:
        O, lse = dma.dma_attn_fwd_chunk(p, L - rows, Q[:, L - rows:].contiguous(), K, V, bias, expiry)
    else:
        O, lse = dma.dma_attn_fwd(p, Q, K, V, bias, expiry, bitmap)
    torch.cuda.synchronize()
    kept = np.arange(L - (rows or L), L, dtype=np.int32)
    Or, lr = oracle.forward(*(f64(inp[k]) for k in ("Q", "K", "V")), dl.astype(np.float64), expiry=e, rows=kept)
    assert_close(O, Or, case.dtype, f"{case.name}: O")
    assert_close(lse, lr, case.dtype, f"{case.name}: lse", lse=True)


# (batch entries of two heads: as many as fwd_tiles takes two query tiles per CTA for; rows 0: the whole sequence)
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("L,w,rows,B,flags", [
    (1100, 64, 0, 32, 0), (1152, 1152, 0, 32, 0), (1025, 1, 0, 32, 0), (700, 200, 0, 100, 0),            # tile walk: nine and six query tiles, ragged and whole ends
    (1100, 64, 0, 200, 0), (1152, 1152, 0, 200, 0), (1025, 1, 0, 200, 0), (1250, 90, 0, 32, 0),          # (an odd number of tiles: two per CTA for more heads)
    (2177, 40, 0, 32, dma.DMA_FLAG_TILE_PATH), (3000, 1000, 0, 32, 0), (1500, 1, 0, 64, dma.DMA_FLAG_IGNORE_BITMAP),
    (2050, 1, 0, 32, 0), (2305, 512, 0, 32, 0), (2200, 300, 0, 32, 0),                                   # token-compacted lists
    (1000, 128, 129, 150, 0), (700, 700, 300, 150, 0), (700, 700, 450, 150, 0), (4096, 300, 2048, 74, 0), (2500, 300, 1790, 74, 0)])   # chunks of rows
def test_bits_do_not_depend_on_the_batch(L, w, rows, B, flags, d):
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=2, Hkv=1, L=L, w=w, d=d, name=f"alone and in a batch L{L} w{w} d{d}")
    inp = wl.make_inputs(case)
    inp["Q"] = inp["Q"] * torch.linspace(0.25, 8.0, L).view(1, L, 1, 1).to(inp["Q"].dtype)     # (row references that grow often)
    out = []
    for n in (1, B):
        p = dma.problem(n, 2, 1, L, d, w, flags=flags)
        Q, K, V = (inp[k].to(DEV).repeat(n, 1, 1, 1) for k in ("Q", "K", "V"))
        bias, expiry, bitmap = dma.dma_mask_build(p, V, inp["W_delta"].to(DEV), inp["A"].to(DEV))
        if rows:
            out.append(dma.dma_attn_fwd_chunk(p, L - rows, Q[:, L - rows:].contiguous(), K, V, bias, expiry))
        else:
            out.append(dma.dma_attn_fwd(p, Q, K, V, bias, expiry, bitmap))
    torch.cuda.synchronize()
    for one, many in zip(*out):
        assert all(torch.equal(one[0], x) for x in many)
    dl, e, _ = oracle_mask(case, inp)
    kept = np.arange(L - (rows or L), L, dtype=np.int32)
    Or, lr = oracle.forward(*(f64(inp[k]) for k in ("Q", "K", "V")), dl.astype(np.float64), expiry=e, rows=kept)
    assert_close(out[1][0][:1], Or, case.dtype, f"{case.name}: O")
    assert_close(out[1][1][:1], lr, case.dtype, f"{case.name}: lse", lse=True)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("L,w,rows", SHAPES)
def test_two_query_tiles_on_the_small_shapes(L, w, rows, d):
    """DMA_FLAG_BLOCK_SKIP always takes two query tiles per CTA: odd tile counts, ragged ends, w = 1, w >= L, both walks."""
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=2, Hkv=1, L=L, w=w, d=d, name=f"two tiles L{L} w{w} d{d}")
    inp = wl.make_inputs(case)
    p, bias, expiry, bitmap = gpu_mask(case, inp)
    Q, K, V = (inp[k].to(DEV) for k in ("Q", "K", "V"))
    for path in (0,) if rows else (dma.DMA_FLAG_TILE_PATH, dma.DMA_FLAG_COMPACT_KV):
        out = []
        for flags in (path, path | dma.DMA_FLAG_BLOCK_SKIP):
            p = dma.problem(1, 2, 1, L, d, w, flags=flags)
            if rows:
                out.append(dma.dma_attn_fwd_chunk(p, L - rows, Q[:, L - rows:].contiguous(), K, V, bias, expiry))
            else:
                out.append(dma.dma_attn_fwd(p, Q, K, V, bias, expiry, bitmap))
        torch.cuda.synchronize()
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1]), path


@pytest.mark.parametrize("d", [64, 128])
def test_pairs_whose_tiles_use_different_key_tiles(d):
    """Documents that begin inside a pair of query tiles: one tile skips the key tiles its partner needs and enters the walk late. 400 heads take
    two query tiles per CTA, 64 and two heads one."""
    L, cu = 1100, torch.tensor([0, 77, 384, 520, 700, 1100], dtype=torch.int32, device=DEV)
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=2, Hkv=2, L=L, w=64, d=d, name="late entry")
    inp = wl.make_inputs(case)
    W, A = inp["W_delta"].to(DEV), inp["A"].to(DEV)
    out = {}
    for B, flags in ((1, dma.DMA_FLAG_SIMT), (1, 0), (1, dma.DMA_FLAG_BLOCK_SKIP), (32, 0), (32, 0), (32, 0), (200, 0), (200, 0), (200, 0)):
        p = dma.problem(B, 2, 2, L, d, 64, flags=flags)
        Q, K, V = (inp[k].to(DEV).repeat(B, 1, 1, 1) for k in ("Q", "K", "V"))
        mask = dma.dma_mask_build_varlen(p, V, W, A, cu)
        O, lse = dma.dma_attn_fwd(p, Q, K, V, *mask)
        torch.cuda.synchronize()
        if flags == dma.DMA_FLAG_SIMT:
            assert_close(O, np.asarray(oracle.forward(*(f64(inp[k]) for k in ("Q", "K", "V")), f64(mask[0]), expiry=mask[1].cpu().numpy())[0]), case.dtype, "O")
            out["O"], out["lse"] = O.float(), lse
            continue
        assert float((O.float() - out["O"]).abs().max()) <= 3e-2 and float((lse - out["lse"]).abs().max()) <= 1e-3 * max(1.0, float(out["lse"].abs().max()))
        bits = out.setdefault("bits", (O[0], lse[0]))
        assert all(torch.equal(x, bits[0]) for x in O) and all(torch.equal(x, bits[1]) for x in lse), (B, flags)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,skip", [(1, 0), (1, dma.DMA_FLAG_BLOCK_SKIP), (100, 0)])     # one query tile per CTA, two, two
@pytest.mark.parametrize("path", ["tiles", "lists", "chunk", "noncausal"])
def test_query_tiles_without_keys(path, B, skip, d):
    """A caller's mask (padding) may leave whole query tiles, pairs of them or a head without a key: O is exactly zero there and lse -inf, whatever Q
    holds; the other rows are as ever."""
    L, gone = 1100, [(256, 512), (1024, 1100)]
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=2, Hkv=1, L=L, w=300, d=d, name=f"no keys {path} d{d}")
    inp = wl.make_inputs(case)
    inp["Q"] = inp["Q"] * 8.0
    dl = oracle_mask(case, inp)[0]
    if path == "noncausal":
        e = oracle.select_noncausal(dl, case.w)
        e[:, 1] = 0                                                        # (the second head keeps nothing)
    else:
        e = oracle.select_expiry_varlen(dl, case.w, [0, 256, 512, 1024, L])
        for a, b in gone:
            e[..., a:b] = np.arange(a, b)
    bitmap = torch.from_numpy(oracle.bitmap_from_expiry(e).view(np.int32)).to(DEV).repeat(B, 1, 1, 1)
    flags = {"tiles": dma.DMA_FLAG_TILE_PATH, "lists": dma.DMA_FLAG_COMPACT_KV}.get(path, 0) | skip
    p = dma.problem(B, 2, 1, L, d, case.w, flags=flags, causal=int(path != "noncausal"))
    Q, K, V = (inp[k].to(DEV).repeat(B, 1, 1, 1) for k in ("Q", "K", "V"))
    bias, expiry = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV).repeat(B, 1, 1) for x in (dl, e))
    first = 256 if path == "chunk" else 0
    empty = np.zeros(L, bool)
    if path != "noncausal":
        for a, b in gone:
            empty[a:b] = True
    rows = np.flatnonzero(~empty[first:]).astype(np.int64)
    Or, lr = oracle.forward(*(f64(inp[k]) for k in ("Q", "K", "V")), dl.astype(np.float64), expiry=e, rows=(rows + first).astype(np.int32),
                            causal=path != "noncausal")
    heads = [0] if path == "noncausal" else [0, 1]
    for _ in range(3):
        O, lse = torch.full_like(Q[:, first:], float("nan")), torch.zeros(B, 2, L - first, device=DEV)
        if path == "chunk":
            dma.dma_attn_fwd_chunk(p, first, Q[:, first:].contiguous(), K, V, bias, expiry, O=O, lse=lse)
        else:
            dma.dma_attn_fwd(p, Q, K, V, bias, expiry, bitmap, O=O, lse=lse)
        torch.cuda.synchronize()
        at = torch.from_numpy(np.flatnonzero(empty[first:])).to(DEV)
        assert bool((O[:, at] == 0).all()) and bool(torch.isneginf(lse[:, :, at]).all())
        if path == "noncausal":
            assert bool((O[:, :, 1] == 0).all()) and bool(torch.isneginf(lse[:, 1]).all())
        assert all(torch.equal(x, O[0]) for x in O)
        live = torch.from_numpy(rows).to(DEV)
        assert_close(O[:1, live][:, :, heads], np.asarray(Or)[:, :, heads], case.dtype, f"{case.name}: O")
        assert_close(lse[:1, heads][:, :, live], np.asarray(lr)[:, heads], case.dtype, f"{case.name}: lse", lse=True)
