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


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("L,w,rows", [(1, 1, 0), (5, 2, 0), (128, 128, 0), (129, 40, 0), (256, 256, 0), (300, 30, 0), (640, 500, 0), (897, 64, 0),
                                      (2050, 100, 0), (2305, 512, 0), (700, 90, 1), (1000, 128, 129), (2500, 300, 250)])
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
    (2177, 40, 0, 32, dma.DMA_FLAG_TILE_PATH), (3000, 1000, 0, 32, 0), (1500, 1, 0, 64, dma.DMA_FLAG_IGNORE_BITMAP),
    (2050, 1, 0, 32, 0), (2305, 512, 0, 32, 0), (2200, 300, 0, 32, 0),                                   # token-compacted lists
    (1000, 128, 129, 150, 0), (700, 700, 300, 150, 0), (4096, 300, 2048, 74, 0), (2500, 300, 1790, 74, 0)])   # chunks of rows
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
