"""Bit-exact selection on every route of the block sort: heads that one CTA takes whole (blocks of 1024 and of 4096 keys), heads in
blocks of either size that are searched block by block, and those with merge launches, at the edges of threads, warps and blocks; few and many heads,
ties, packed documents, the non-causal mode, square tiles of other sizes and tiles that are not square."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_02124_b200 import binding as dma

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def build(H, L, w, seed, levels=0, causal=1, cu=None, tile=(0, 0)):
    """Mask of H heads with one value head each; `levels` distinct value rows (0: all different)."""
    g = torch.Generator().manual_seed(seed)
    V = torch.randn(1, L, H, 64, generator=g)
    if levels:
        V = V[:, torch.randint(0, levels, (L,), generator=g) % L]
    V, W, A = V.to(torch.bfloat16), torch.randn(H, 64, generator=g) / 8, torch.rand(H, generator=g) + 0.5
    p = dma.problem(1, H, H, L, 64, w, causal=causal, tile_m=tile[0], tile_n=tile[1])
    if cu is None:
        bias, e, bitmap = dma.dma_mask_build(p, V.to(DEV), W.to(DEV), A.to(DEV))
    else:
        bias, e, bitmap = dma.dma_mask_build_varlen(p, V.to(DEV), W.to(DEV), A.to(DEV), torch.tensor(cu, dtype=torch.int32, device=DEV))
    torch.cuda.synchronize()
    _, dl = oracle.delta(V.float().numpy(), W.numpy(), A.numpy(), H)
    return dl, e.cpu().numpy(), bitmap.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("H,L", [(2, n) for n in (4, 31, 127, 128, 129, 255, 257, 1023, 1024, 1025, 2047, 2049, 3071, 3073, 4095, 4097, 5121, 9000)] +
                         [(300, 900), (150, 1100), (150, 2049), (80, 3100), (75, 4096), (75, 4200), (20, 17000)])
def test_block_sizes(H, L):
    for w in (1, max(1, L // 5), L - 1):
        dl, e, bitmap = build(H, L, max(w, 1), seed=L)
        ref = oracle.select_expiry(dl, min(max(w, 1), L))
        assert np.array_equal(e, ref), (H, L, w)
        assert np.array_equal(bitmap, oracle.bitmap_from_expiry(ref)), (H, L, w)


@pytest.mark.parametrize("H,L", [(2, 700), (2, 2500), (2, 5000), (80, 4000)])
def test_ties_documents_and_other_rows(H, L):
    dl, e, bitmap = build(H, L, L // 7, seed=1, levels=23)
    ref = oracle.select_expiry(dl, L // 7)
    assert np.array_equal(e, ref) and np.array_equal(bitmap, oracle.bitmap_from_expiry(ref))
    cu = [0, 1, L // 3, L // 3 + 130, L]
    dl, e, bitmap = build(H, L, 60, seed=2, levels=400, cu=cu)
    ref = oracle.select_expiry_varlen(dl, 60, cu)
    assert np.array_equal(e, ref) and np.array_equal(bitmap, oracle.bitmap_from_expiry(ref))
    dl, e, _ = build(H, L, L // 4, seed=3, levels=50, causal=0)
    assert np.array_equal(e, oracle.select_noncausal(dl, L // 4))


@pytest.mark.parametrize("side", [4096, 8192, 1 << 26, 1 << 27, 1 << 30])
@pytest.mark.parametrize("L,w", [(300, 400), (700, 90), (5000, 800), (9000, 9000)])
def test_tiles_longer_than_the_sequence(L, w, side):
    """Also where 32 sides, a word's worth of tiles, are more than 32 bits hold."""
    dl, e, bitmap = build(2, L, w, seed=L, tile=(side, side))
    ref = oracle.select_expiry(dl, min(w, L))
    assert np.array_equal(e, ref)
    assert np.array_equal(bitmap, oracle.bitmap_from_expiry(ref, side, side))


@pytest.mark.parametrize("tile", [(64, 64), (96, 96), (160, 160), (32, 32), (48, 48), (128, 64), (64, 128)])
@pytest.mark.parametrize("L", [900, 4000, 5000])
def test_tiles(L, tile):
    dl, e, bitmap = build(2, L, L // 6, seed=L, tile=tile)
    ref = oracle.select_expiry(dl, L // 6)
    assert np.array_equal(e, ref)
    assert np.array_equal(bitmap, oracle.bitmap_from_expiry(ref, *tile)), tile


@pytest.mark.parametrize("H,L", [(2, 4097), (2, 12000), (2, 32768), (2, 32769), (80, 4097), (80, 9000)])
def test_heads_searched_block_by_block(H, L):
    """Equal weights across blocks, documents that begin at, one behind and inside a block, a last block of one key, windows that are never reached; up to the longest
    head whose blocks are searched and one key beyond."""
    for w in (3, L // 3, L - 1):
        dl, e, bitmap = build(H, L, w, seed=L + w, levels=300)
        ref = oracle.select_expiry(dl, w)
        assert np.array_equal(e, ref) and np.array_equal(bitmap, oracle.bitmap_from_expiry(ref)), w
    cu = sorted({0, 1024, 1025, 4096, L - 1, L})
    for w in (2, 700):
        dl, e, bitmap = build(H, L, w, seed=L, levels=300, cu=cu)
        ref = oracle.select_expiry_varlen(dl, w, cu)
        assert np.array_equal(e, ref) and np.array_equal(bitmap, oracle.bitmap_from_expiry(ref)), w
    dl, e, _ = build(H, L, L // 4, seed=3, levels=300, causal=0)
    assert np.array_equal(e, oracle.select_noncausal(dl, L // 4))


@pytest.mark.parametrize("H,L", [(10, 32768), (12, 28700), (20, 16385), (36, 12200), (48, 17000), (60, 8190)])
def test_heads_searched_in_blocks_of_4096_keys(H, L):
    """Two to eight blocks, whole and ragged, a last block of one key: all three modes (documents of 48 heads are merged), equal weights across blocks, documents that begin at, one
    behind and inside a block."""
    test_heads_searched_block_by_block(H, L)
    cu = sorted({0, 4095, 4096, 4097, L // 2, L})                                # (long documents: walks that end in another block than the key's)
    dl, e, bitmap = build(H, L, 1500, seed=L + 1, levels=2000, cu=cu)
    ref = oracle.select_expiry_varlen(dl, 1500, cu)
    assert np.array_equal(e, ref) and np.array_equal(bitmap, oracle.bitmap_from_expiry(ref))
