"""GPU parity of the token-compacted backward's work items: walks cut into parts for few heads (up to eight CTAs per key tile), tiles whose
keys no row keeps, ragged last tiles, items by length and in the permutation's order, and the uncut walks of DMA_FLAG_DETERMINISTIC."""
import pytest
import torch

from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import workloads as wl
from helpers import gpu_run, oracle_mask, stored_forward
from test_gpu_attention import compare, oracle_all

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,L,d,w", [
    (1, 1, 1, 129, 128, 5),          # two tiles, most keys never kept
    (1, 2, 1, 1345, 64, 1),          # 21 row steps of 64 in the last walk, w = 1
    (1, 1, 1, 2050, 128, 100),       # walks of up to 33 steps in parts of 16
    (1, 2, 1, 2305, 64, 400),
    (2, 1, 1, 3000, 64, 700),        # parts of different lengths
    (1, 1, 1, 4096, 128, 16),
])
def test_walks_in_parts(B, Hq, Hkv, L, d, w):
    case = wl.small(wl.CONFIGS["2"], B=B, Hq=Hq, Hkv=Hkv, L=L, d=d, w=w, backward=True, seed=L + w, name=f"walks L{L} w{w}")
    inp = wl.make_inputs(case)
    dl, e, _ = oracle_mask(case, inp)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    got = gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_COMPACT_KV)
    compare(case, got, ref)
    runs = [gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_COMPACT_KV | dma.DMA_FLAG_DETERMINISTIC) for _ in range(2)]
    compare(case, runs[0], ref)
    assert all(torch.equal(runs[0][k], runs[1][k]) for k in ("dK", "dV", "dM"))
