"""GPU parity of the token-compacted backward's work items: walks cut into parts for few heads (two, three, four and eight CTAs per key
tile), tiles whose keys no row keeps, ragged last tiles, heads whose blocks do not suffice for all their walks, and the uncut walks of
DMA_FLAG_DETERMINISTIC. The items here are ordered by length; four heads of 131072 keys in test_gpu_attention take cut walks in the
permutation's order. What a walk's keys get does not depend on which part ends first."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import workloads as wl
from helpers import assert_close, gpu_run, oracle_mask, stored_forward
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
    for _ in range(4):                       # (two query heads' first parts meet in one sum: a + b = b + a)
        again = gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_COMPACT_KV)
        assert all(torch.equal(got[k], again[k]) for k in ("dK", "dV", "dM"))
    runs = [gpu_run(case, inp, stored=st, flags=dma.DMA_FLAG_COMPACT_KV | dma.DMA_FLAG_DETERMINISTIC) for _ in range(2)]
    compare(case, runs[0], ref)
    assert all(torch.equal(runs[0][k], runs[1][k]) for k in ("dK", "dV", "dM"))


@pytest.mark.parametrize("Hq,Hkv,L,d,w", [
    (2, 2, 16384, 64, 64),           # eight parts
    (1, 1, 9663, 128, 1442),
    (2, 1, 8192, 128, 300),
    (8, 2, 4096, 64, 256),           # four query heads per KV head: dM alone repeats
])
def test_cut_and_whole_walks(Hq, Hkv, L, d, w):
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=Hq, Hkv=Hkv, L=L, d=d, w=w, backward=True, seed=L + w, name=f"cut walks L{L} w{w}")
    inp = wl.make_inputs(case)
    whole = gpu_run(case, inp, flags=dma.DMA_FLAG_DETERMINISTIC)
    runs = [gpu_run(case, inp) for _ in range(4)]
    assert torch.equal(whole["O"], runs[0]["O"])
    for k in ("dK", "dV"):
        assert_close(runs[0][k], whole[k].double().cpu().numpy(), case.dtype, k)
    # fp32 sums of the same terms in another order: 2^-24 sqrt(terms) of their 2-norm, times what cancels between them (dO and O of 64 and
    # 128 channels: terms up to some tens of the sum)
    dm, ref = runs[0]["dM"].double(), whole["dM"].double()
    assert float((dm - ref).norm() / ref.norm()) <= 1e-4
    for r in runs[1:]:
        assert all(torch.equal(runs[0][k], r[k]) for k in ("dM",) + (("dK", "dV") if Hq <= 2 * Hkv else ()))


def test_more_walks_than_blocks():
    """Every key kept to the end, which no window allows: eight of a head's sixteen walks exceed a CTA's share, and 74 heads have four blocks each."""
    B = 37
    case = wl.small(wl.CONFIGS["2"], B=1, Hq=2, Hkv=1, L=2048, d=64, w=16, backward=True, seed=3, name="more walks than blocks")
    inp = wl.make_inputs(case)
    dl, _, _ = oracle_mask(case, inp)
    e = np.full((1, 2, 2048), 2048, np.int32)
    ref = oracle_all(case, inp, dl, e)
    st = stored_forward(case, ref["O"], ref["lse"])
    dev = torch.device("cuda:0")
    put = lambda t: torch.as_tensor(t).to(dev).repeat(B, *[1] * (np.ndim(t) - 1))  # noqa: E731
    Q, K, V, dO = (put(inp[k]) for k in ("Q", "K", "V", "dO"))
    p = dma.problem(B, 2, 1, 2048, 64, 16, flags=dma.DMA_FLAG_COMPACT_KV)
    O, lse, bias, ex = put(torch.from_numpy(st["O"]).to(torch.bfloat16)), put(st["lse"]), put(dl), put(e)
    bmp = put(oracle.bitmap_from_expiry(e).view(np.int32))
    runs = [dma.dma_attn_bwd(p, Q, K, V, O, dO, lse, bias, ex, bmp) for _ in range(2)]
    torch.cuda.synchronize()
    for k, x, y in zip(("dQ", "dK", "dV", "dM"), *runs):
        assert_close(x, np.repeat(ref[k], B, 0), case.dtype, k)
        assert k == "dQ" or (torch.equal(x, y) and all(torch.equal(x[0], z) for z in x)), k
