"""GPU parity of the forward whose CTAs own one query tile and deal its key tiles out to both softmax groups (small grids take it)
against the oracle: one key tile (the second group has none), two, odd and even numbers, ragged ends, tiles with few and with many
keys expiring, token-compacted lists and chunks of rows."""
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
