"""Workspace sizes, host side: what the entry points ask for and accept. No GPU: a call whose arguments pass is told apart by its
next check, which finds no device."""
import ctypes

import pytest
import torch

from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import build as dma_build

no_device = pytest.mark.skipif(torch.cuda.is_available(), reason="tells accepted calls by the missing device")
ERR_WORKSPACE, ERR_CUDA = -5, -6


@pytest.fixture(scope="module")
def lib():
    dma_build.build()
    return dma.lib()


def backward(lib, p, ws_bytes):
    a = ctypes.c_void_p(4096)
    return lib.dma_attn_bwd(ctypes.byref(p), *([a] * 13), a, ctypes.c_size_t(ws_bytes), ctypes.c_void_p(0))


def backward_bytes(B, Hq, Hkv, L, d, slots):
    """Header, D (whole 64 rows), the dQ accumulator of whole query tiles, `slots` copies of the dK and dV accumulators."""
    return 256 + 4 * (-(-B * Hq * L // 64) * 64 + B * Hq * -(-L // 128) * 128 * d + 2 * slots * B * L * Hkv * d)


@no_device
@pytest.mark.parametrize("B,Hq,Hkv,L,n", [
    (2, 16, 4, 1000, 4),                       # 64 key tiles for 148 SMs
    (1, 32, 8, 2048, 2), (1, 16, 4, 4096, 2),  # 128 tiles, long walks
    (8, 16, 4, 512, 2), (32, 16, 4, 128, 1),   # 128 tiles, short walks: another CTA costs what it takes over
    (16, 16, 4, 512, 1), (1, 32, 16, 2048, 1),  # 256 tiles
    (1, 16, 1, 2048, 16), (1, 16, 1, 8192, 4), (1, 6, 2, 1500, 3), (1, 8, 8, 512, 1)])
def test_tile_backward_split(lib, B, Hq, Hkv, L, n):
    """The number of CTAs that share a KV head's query heads, seen through the slots that the call needs."""
    p = dma.problem(B, Hq, Hkv, L, 128, L, flags=dma.DMA_FLAG_TILE_PATH)
    need = backward_bytes(B, Hq, Hkv, L, 128, n if n > 1 else 0)
    assert backward(lib, p, need) == ERR_CUDA
    assert backward(lib, p, need - 1) == ERR_WORKSPACE


def mask_backward(lib, p, ws_bytes):
    a = ctypes.c_void_p(4096)
    return lib.dma_mask_bwd(ctypes.byref(p), *([a] * 8), a, ctypes.c_size_t(ws_bytes), ctypes.c_void_p(0))


@no_device
@pytest.mark.parametrize("B,Hq,Hkv,L,d,rows", [
    (1, 16, 4, 4096, 128, 32), (1, 16, 4, 4736, 128, 32),     # at most 74 CTAs of 64 rows: twice as many still run at once
    (1, 16, 4, 4737, 128, 64), (1, 16, 4, 8192, 128, 64), (1, 8, 8, 8192, 64, 64), (2, 8, 4, 3000, 128, 64),
    (1, 16, 4, 16384, 128, 64), (1, 32, 8, 8192, 128, 32)])   # 1024 channels: 64 rows do not fit
def test_full_weight_backward_rows(lib, B, Hq, Hkv, L, d, rows):
    """Rows per CTA of the mask backward with full sampling weights, seen through the partial sums that the call needs."""
    p = dma.problem(B, Hq, Hkv, L, d, 64, flags=dma.DMA_FLAG_FULL_DELTA)
    need = B * -(-L // rows) * Hq * (Hkv * d + 1) * 4
    assert mask_backward(lib, p, need) == ERR_CUDA
    assert mask_backward(lib, p, need - 1) == ERR_WORKSPACE


# ---- a workspace taken for the longest sequence and the largest batch serves the others --------------------------------------
LENGTHS = sorted({1, 7, 100, 127, 128, 129, 255, 300, 513, 900, 1000, 1151, 1152, 1153, 1279, 1280, 1281, 1500, 2047, 2048, 2049, 2500,
                  3000, 4095, 4096, 4097, 4607, 4608, 4609, 4736, 4737, 6000, 8063, 8064, 8191, 8192, 8193, 9408, 9409, 9472, 16383, 16384,
                  16385, 20000, 32768})
BATCHES = [1, 2, 3, 4, 5, 8, 16, 37, 64]
HEADS = [(32, 8), (16, 2), (16, 4), (16, 1), (12, 4), (6, 2), (32, 32), (8, 8), (14, 2), (1, 1)]


def never_falls(size, make):
    """size(make(B, L)) over all pairs: not below that of any shorter sequence or smaller batch."""
    table = [[size(make(B, L)) for L in LENGTHS] for B in BATCHES]
    for row in table:
        assert row == sorted(row), [(L, n) for L, n, m in zip(LENGTHS, row, row[1:] + [row[-1]]) if n > m]
    for i, L in enumerate(LENGTHS):
        col = [row[i] for row in table]
        assert col == sorted(col), (L, list(zip(BATCHES, col)))


@pytest.mark.parametrize("flags", [0, dma.DMA_FLAG_TILE_PATH, dma.DMA_FLAG_COMPACT_KV, dma.DMA_FLAG_COMPACT_KV | dma.DMA_FLAG_DETERMINISTIC])
@pytest.mark.parametrize("Hq,Hkv", HEADS)
def test_attention_and_mask_workspaces_never_fall(lib, Hq, Hkv, flags):
    for d in (64, 128):
        for w in (1, 256, 1280, 4096):
            for causal in ((1, 0) if flags == 0 else (1,)):
                for i in range(3):
                    never_falls(lambda p: dma.dma_query_workspace(p)[i], lambda B, L: dma.problem(B, Hq, Hkv, L, d, w, causal=causal, flags=flags))


@no_device
@pytest.mark.parametrize("B,Hq,Hkv,L,d,w", [(1, 32, 8, 8192, 128, 4096), (1, 16, 2, 8192, 64, 2048), (4, 16, 4, 1000, 64, 256), (2, 32, 8, 16384, 128, 2048)])
def test_backward_accepts_a_workspace_of_a_longer_sequence(lib, B, Hq, Hkv, L, d, w):
    ws = dma.dma_query_workspace(dma.problem(B, Hq, Hkv, L, d, w))[2]
    for n in (n for n in LENGTHS if n <= L):
        for b in range(1, B + 1):
            assert backward(lib, dma.problem(b, Hq, Hkv, n, d, w), ws) == ERR_CUDA, (b, n)


@pytest.mark.parametrize("Hq,Hkv", HEADS)
@pytest.mark.parametrize("w", [1, 100, 600, 1152, 1200, 1280, 2048, 5000, 16384])
def test_decode_workspace_never_falls(lib, Hq, Hkv, w):
    never_falls(dma.dma_decode_workspace, lambda B, N: dma.problem(B, Hq, Hkv, N, 128, w))


@no_device
@pytest.mark.parametrize("B,Hq,w", [(1, 32, 1280), (1, 32, 1200), (2, 32, 600), (1, 1, 2048), (3, 8, 1024), (1, 40, 512)])
def test_decoding_calls_accept_the_last_step_s_workspace(lib, B, Hq, w):
    a, z = ctypes.c_void_p(4096), ctypes.c_void_p(0)
    ws = ctypes.c_size_t(dma.dma_decode_workspace(dma.problem(B, Hq, Hq, 16384, 128, w)))
    for N in (n for n in LENGTHS if n <= 16384):
        p, ld = ctypes.byref(dma.problem(B, Hq, Hq, N, 128, w)), ctypes.c_int64(16384)
        assert lib.dma_decode(p, a, a, a, a, ld, a, a, z, a, ws, z) == ERR_CUDA, N
        assert lib.dma_decode_step(p, a, a, a, a, ld, a, a, a, a, ws, z) == ERR_CUDA, N
        assert lib.dma_decode_state_init(p, a, ld, a, a, ws, z) == ERR_CUDA, N
    for b in range(1, B):                                    # (fewer rows may take shorter splits, hence more of them)
        p = ctypes.byref(dma.problem(b, Hq, Hq, 4096, 128, w))
        assert lib.dma_decode_step(p, a, a, a, a, ld, a, a, a, a, ws, z) == ERR_CUDA, b


@no_device
@pytest.mark.parametrize("B,Hq,w", [(1, 32, 1280), (1, 32, 2048), (2, 8, 1000), (1, 1, 65536), (1, 2, 1 << 20)])
def test_decoding_calls_accept_the_first_step_s_workspace(lib, B, Hq, w):
    a, z = ctypes.c_void_p(4096), ctypes.c_void_p(0)
    ws = ctypes.c_size_t(dma.dma_decode_workspace(dma.problem(B, Hq, Hq, 1, 128, w)))
    for N in (n for n in LENGTHS if n <= 65536):
        p, ld = ctypes.byref(dma.problem(B, Hq, Hq, N, 128, w)), ctypes.c_int64(65536)
        assert lib.dma_decode(p, a, a, a, a, ld, a, a, z, a, ws, z) == ERR_CUDA, N
        assert lib.dma_decode_step(p, a, a, a, a, ld, a, a, a, a, ws, z) == ERR_CUDA, N


@pytest.mark.parametrize("w", [2 ** 31 - 1, 2 ** 31 - 200, 2 ** 24])
def test_decode_workspace_of_a_window_without_bound(lib, w):
    """`Keep all`: the window does not count beyond the cached keys. (Kept indices and, per 128 of them, a partial row of d + 2 floats.)"""
    for N in (1, 1000, 65536, 200000):
        rows, keep = 32, N
        assert 0 < dma.dma_decode_workspace(dma.problem(1, 32, 8, N, 128, w)) <= 200000 + rows * (keep * 4 + (keep // 128 + 1) * 130 * 4), (w, N)


@pytest.mark.parametrize("flags", [0, dma.DMA_FLAG_FULL_DELTA])
@pytest.mark.parametrize("Hq,Hkv", HEADS)
def test_mask_backward_workspace_never_falls(lib, Hq, Hkv, flags):
    for d in (64, 128):
        never_falls(dma.dma_mask_bwd_workspace, lambda B, L: dma.problem(B, Hq, Hkv, L, d, 64, flags=flags))


@no_device
@pytest.mark.parametrize("flags", [0, dma.DMA_FLAG_FULL_DELTA])
@pytest.mark.parametrize("B,Hq,Hkv,L", [(1, 16, 4, 16384), (3, 16, 4, 4737), (64, 8, 8, 1000)])
def test_mask_backward_accepts_a_workspace_of_a_longer_sequence(lib, B, Hq, Hkv, L, flags):
    ws = dma.dma_mask_bwd_workspace(dma.problem(B, Hq, Hkv, L, 64, 64, flags=flags))
    for n in (n for n in LENGTHS if n <= L):
        for b in range(1, B + 1):
            assert mask_backward(lib, dma.problem(b, Hq, Hkv, n, 64, 64, flags=flags), ws) == ERR_CUDA, (b, n)
