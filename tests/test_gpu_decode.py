"""GPU parity of the decoding step (dma_delta_range + dma_decode) against the oracle: selected key sets bit-exact,
outputs within the element type's tolerance."""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_02124_b200 import binding as dma
from paper_2508_02124_b200 import workloads as wl
from helpers import assert_close, bits_equal, oracle_mask

pytestmark = pytest.mark.gpu


def run_case(case, cap_extra=0, seed=21, tie_heads=False):
    """The case's K, V (and W_delta, A) form the cache; the query of every head is a fresh N(0,1) vector."""
    inp = wl.make_inputs(case)
    dev = torch.device("cuda:0")
    B, N, Hq, Hkv, d = case.B, case.L, case.Hq, case.Hkv, case.d
    g = torch.Generator().manual_seed(seed)
    q = torch.randn(B, Hq, d, generator=g).to(case.torch_dtype)
    cap = N + cap_extra
    Kc = torch.zeros(B, cap, Hkv, d, dtype=case.torch_dtype); Kc[:, :N] = inp["K"]
    Vc = torch.zeros(B, cap, Hkv, d, dtype=case.torch_dtype); Vc[:, :N] = inp["V"]
    A = inp["A"].clone()
    if tie_heads:
        A[0] = 0.0                                   # delta == 1 for every key of head 0: the w lowest indices win
    p = dma.problem(B, Hq, Hkv, N, d, case.w, dtype=case.torch_dtype)
    p.k_stride[0], p.k_stride[1], p.k_stride[2] = cap * Hkv * d, Hkv * d, d
    p.v_stride[0], p.v_stride[1], p.v_stride[2] = cap * Hkv * d, Hkv * d, d
    Kd, Vd = Kc.to(dev), Vc.to(dev)
    delta = torch.full((B, Hq, cap), -1.0, device=dev)
    # the cache is filled in two appends, as a prefill followed by decoding steps would do
    half = N // 2
    dma.dma_delta_range(p, Vd, inp["W_delta"].to(dev), A.to(dev), delta, 0, half)
    dma.dma_delta_range(p, Vd, inp["W_delta"].to(dev), A.to(dev), delta, half, N)
    o, lse, idx = dma.dma_decode(p, q.to(dev), Kd, Vd, delta, want_idx=True)
    torch.cuda.synchronize()
    # oracle: delta in the pinned fp32 arithmetic, then the definition
    z, dl = oracle.delta(inp["V"].float().numpy(), inp["W_delta"].numpy(), A.numpy(), Hq)
    assert bits_equal(delta[:, :, :N], dl), "delta cache differs from the pinned arithmetic"
    assert (delta[:, :, N:] == -1.0).all(), "entries beyond the appended range were touched"
    ro, rl, ridx = oracle.decode(q.double().numpy(), inp["K"].double().numpy(), inp["V"].double().numpy(), dl, case.w)
    assert np.array_equal(idx.cpu().numpy(), ridx), "selected key sets differ"
    assert_close(o, ro, case.dtype, f"{case.name}: o")
    assert_close(lse, rl, case.dtype, f"{case.name}: lse", lse=True)


@pytest.mark.parametrize("kw", [
    dict(B=1, Hq=2, Hkv=2, L=256, d=64, w=64, dtype="fp32"),
    dict(B=2, Hq=4, Hkv=2, L=1000, d=64, w=100, dtype="bf16"),
    dict(B=2, Hq=8, Hkv=2, L=3001, d=128, w=512, dtype="bf16"),       # ragged: two splits, the second partly empty
    dict(B=1, Hq=4, Hkv=4, L=5000, d=128, w=1, dtype="fp32"),         # a single key
    dict(B=1, Hq=4, Hkv=1, L=700, d=128, w=4096, dtype="bf16"),       # w >= N: dense attention over the cache
    dict(B=1, Hq=2, Hkv=1, L=9500, d=128, w=9000, dtype="bf16"),      # 71 splits of a row: combined in three turns
    dict(B=1, Hq=1, Hkv=1, L=13000, d=64, w=12500, dtype="fp32"),     # 98 splits
    dict(B=2, Hq=4, Hkv=2, L=20000, d=64, w=17000, dtype="bf16"),     # 34 splits of 512 keys
])
def test_small_cases(kw):
    run_case(wl.small(wl.CONFIGS["2"], name="decode-small", backward=False, **kw), cap_extra=37)


def test_ties_go_to_the_lower_index():
    run_case(wl.small(wl.CONFIGS["2"], name="decode-ties", backward=False, B=1, Hq=2, Hkv=1, L=4500, d=128, w=300), tie_heads=True)


def test_long_cache_config5_shapes():
    # the paper's decode setting on the long-context shapes: 65 536 cached keys, w = 4096, 32 / 8 heads
    run_case(wl.CONFIGS["5"], cap_extra=128)


@pytest.mark.parametrize("N,w", [(1, 1), (33, 7), (4096, 512), (4097, 4096), (16384, 2048), (16385, 1), (32768, 8192), (32769, 100),
                                 (65537, 4096), (262144, 1000), (262177, 20000)])
@pytest.mark.parametrize("kind", ["random", "tied", "few", "ramp", "outlier"])
def test_selection_at_the_edges_of_the_register_and_cluster_sizes(N, w, kind):
    """The kept indices (ascending) against a stable sort, at the row lengths where the selection kernel changes shape, for rows
    whose threshold takes one pass, several passes over ever narrower ranges (few distinct values, one value far above the
    others) or a cut among equal keys."""
    g = torch.Generator().manual_seed(N + w)
    BH = 3
    z = torch.randn(1, BH, N, generator=g)
    delta = {"random": lambda: torch.exp(torch.nn.functional.softplus(z)), "tied": lambda: torch.full((1, BH, N), 1.5),
             "few": lambda: 1.0 + torch.randint(0, 4, (1, BH, N), generator=g) / 7.0,
             "ramp": lambda: torch.exp(3.0 * torch.arange(N) / N).expand(1, BH, N).contiguous(),
             "outlier": lambda: torch.where(torch.rand(1, BH, N, generator=g) < 2.0 / N, 1e38, 1.0 + 1e-3 * torch.rand(1, BH, N, generator=g))}[kind]()
    p = dma.problem(1, BH, 1, N, 64, w)
    K = torch.randn(1, N, 1, 64, generator=g).bfloat16().cuda()
    q = torch.zeros(1, BH, 64, dtype=torch.bfloat16, device="cuda")
    _, _, idx = dma.dma_decode(p, q, K, K, delta.cuda(), want_idx=True)
    want = torch.sort(torch.sort(delta, dim=-1, descending=True, stable=True)[1][..., :min(w, N)], dim=-1)[0]
    assert torch.equal(idx.cpu().long(), want)
    state = dma.dma_decode_state_init(p, delta.cuda(), dma.dma_decode_state(p, "cuda"))
    assert dma.decode_state_sets(state, w) == [r.tolist() for r in want[0]]


@pytest.mark.parametrize("N,w", [(33, 7), (16384, 2048), (40000, 100), (262177, 20000)])
@pytest.mark.parametrize("share", [0.0001, 0.5])
def test_selection_with_infinite_weights(N, w, share):
    """exp overflows to infinity in earnest (a large gate): such keys come first, the lower index among them, whether fewer or more
    than w. (A row with fewer still ranks the finite ones, over a range of bit patterns that ends at infinity.)"""
    g = torch.Generator().manual_seed(N)
    BH = 2
    delta = torch.exp(torch.randn(1, BH, N, generator=g))
    delta[torch.rand(1, BH, N, generator=g) < share] = float("inf")
    delta[..., N // 2] = float("inf")
    p = dma.problem(1, BH, 1, N, 64, w)
    K = torch.zeros(1, N, 1, 64, dtype=torch.bfloat16, device="cuda")
    q = torch.zeros(1, BH, 64, dtype=torch.bfloat16, device="cuda")
    _, _, idx = dma.dma_decode(p, q, K, K, delta.cuda(), want_idx=True)
    want = torch.sort(torch.sort(delta, dim=-1, descending=True, stable=True)[1][..., :w], dim=-1)[0]
    assert torch.equal(idx.cpu().long(), want)
    state = dma.dma_decode_state_init(p, delta.cuda(), dma.dma_decode_state(p, "cuda"))
    assert dma.decode_state_sets(state, w) == [r.tolist() for r in want[0]]


@pytest.mark.parametrize("N", [4096, 8193, 33000, 65537, 131072])
@pytest.mark.parametrize("kind", ["random", "tied", "few", "ramp", "outlier", "infinite"])
def test_selection_of_many_rows(N, kind):
    """Rows that are streamed once between a sampled bracket: the kept indices (ascending) and the carried state's sets against a stable sort, for a
    threshold at either end of the row, brackets that hold too many keys (equal ones) and rows whose bracket lies in one place."""
    BH = 304
    g = torch.Generator("cuda").manual_seed(N)
    z = torch.randn(1, BH, N, generator=g, device="cuda")
    delta = {"random": lambda: torch.exp(torch.nn.functional.softplus(z)), "tied": lambda: torch.full_like(z, 1.5),
             "few": lambda: 1.0 + torch.floor(z.abs() * 2) / 7.0, "ramp": lambda: torch.exp(3.0 * torch.arange(N, device="cuda") / N + 1e-4 * z),
             "outlier": lambda: torch.where(z.abs() > 4.2, 1e38, 1.0 + 1e-3 * torch.sigmoid(z)),
             "infinite": lambda: torch.where(z > 1.5, float("inf"), torch.exp(z))}[kind]()
    order = torch.sort(delta, dim=-1, descending=True, stable=True)[1]
    K = torch.zeros(1, N, 1, 64, dtype=torch.bfloat16, device="cuda")
    q = torch.zeros(1, BH, 64, dtype=torch.bfloat16, device="cuda")
    for w in (1, N // 16, N // 4, N - 1):
        want = torch.sort(order[..., :w], dim=-1)[0]
        p = dma.problem(1, BH, 1, N, 64, w)
        _, _, idx = dma.dma_decode(p, q, K, K, delta, want_idx=True)
        assert torch.equal(idx.long(), want), w
        state = dma.dma_decode_state_init(p, delta, dma.dma_decode_state(p, "cuda"))
        rows = state.view(torch.int32).view(BH, -1)
        assert (rows[:, 0] == w).all() and torch.equal(rows[:, 8:8 + w].long(), want[0]), w
        assert torch.equal(torch.gather(rows[:, 8:8 + w], 1, rows[:, 1:2].long())[:, 0].long(), order[0, :, w - 1]), w    # the weakest kept key


@pytest.mark.parametrize("N", [4097, 20000, 32768, 50001, 131072])
@pytest.mark.parametrize("kind", ["misled down", "misled up", "two", "saturated", "low", "repeat", "clusters", "neighbours"])
def test_selection_where_weights_crowd(N, kind):
    """Streamed rows whose bracket misses (the sampled keys are unlike the others), lies across two heavy values or at an end of the row that many keys share, or holds more keys
    than are gathered, of few or of many bit patterns."""
    BH = 304 if N < 60000 else 160
    g = torch.Generator("cuda").manual_seed(N)
    z = torch.rand(1, BH, N, generator=g, device="cuda")
    S = 8192 if N > 65536 else 4096
    i = torch.arange(S, dtype=torch.int64)
    sampled = (i * N // S + ((((i * 2654435761) & 0xFFFFFFFF) >> 16) * (N // S) >> 16)).cuda()
    if kind.startswith("misled"):
        delta = 2.0 + z
        delta[..., sampled] = delta[..., sampled] + (8.0 if kind == "misled up" else -1.5)
    elif kind == "clusters":                                       # 40 values, neighbours in bit patterns
        delta = (torch.tensor(1.5, device="cuda").view(torch.int32) + (z * 40).int()).view(torch.float32)
    elif kind == "neighbours":                                     # every bit pattern of a short range, among outliers
        delta = (torch.tensor(1.5, device="cuda").view(torch.int32) + (z * 3000).int()).view(torch.float32)
        delta[..., ::997] = 1e30
    else:
        delta = {"two": lambda: torch.where(z < 0.25, 3.0, 2.0), "saturated": lambda: torch.where(z < 0.3, 1.6e38, 1.0 + z),
                 "low": lambda: torch.where(z < 0.3, 1.0 + z, 1e-38), "repeat": lambda: 1.0 + z[..., :64].repeat(1, 1, N // 64 + 1)[..., :N]}[kind]()
    delta = delta.contiguous()
    order = torch.sort(delta, dim=-1, descending=True, stable=True)[1]
    K = torch.zeros(1, N, 1, 64, dtype=torch.bfloat16, device="cuda")
    q = torch.zeros(1, BH, 64, dtype=torch.bfloat16, device="cuda")
    for w in (3, N // 16, N // 4 - 5, N // 4 + N // 50, N // 2, N - 2):
        want = torch.sort(order[..., :w], dim=-1)[0]
        p = dma.problem(1, BH, 1, N, 64, w)
        _, _, idx = dma.dma_decode(p, q, K, K, delta, want_idx=True)
        assert torch.equal(idx.long(), want), w
        rows = dma.dma_decode_state_init(p, delta, dma.dma_decode_state(p, "cuda")).view(torch.int32).view(BH, -1)
        assert (rows[:, 0] == w).all() and torch.equal(rows[:, 8:8 + w].long(), want[0]), w
        assert torch.equal(torch.gather(rows[:, 8:8 + w], 1, rows[:, 1:2].long())[:, 0].long(), order[0, :, w - 1]), w    # the weakest kept key
        key = (delta.view(torch.int32)[0].gather(1, order[0, :, w - 1:w])[:, 0].long() << 32) | (0xFFFFFFFF - order[0, :, w - 1])
        assert torch.equal((rows[:, 3].long() << 32) | (rows[:, 2].long() & 0xFFFFFFFF), key), w


@pytest.mark.parametrize("Hq,Hkv,d,dtype", [(1, 1, 64, "fp32"), (3, 3, 128, "bf16"), (6, 2, 64, "bf16"), (32, 8, 128, "bf16"), (33, 11, 128, "fp32")])
def test_delta_of_a_few_keys(Hq, Hkv, d, dtype):
    """Ranges of 1 to 9 keys (up to 8 take a kernel of their own) have the bits of the whole range; heads that do not fill a CTA, groups of any size."""
    g = torch.Generator().manual_seed(d + Hq)
    B, N, td = 2, 40, {"bf16": torch.bfloat16, "fp32": torch.float32}[dtype]
    V = torch.randn(B, N, Hkv, d, generator=g).to(td).cuda()
    W, A = (torch.randn(Hq, d, generator=g) / d ** 0.5).cuda(), (torch.rand(Hq, generator=g) + 0.5).cuda()
    p = dma.problem(B, Hq, Hkv, N, d, 8, dtype=td)
    whole, part = torch.zeros(B, Hq, N, device="cuda"), torch.full((B, Hq, N), -1.0, device="cuda")
    dma.dma_delta_range(p, V, W, A, whole, 0, N)
    at = 0
    for n in (1, 2, 7, 8, 9, 1):
        dma.dma_delta_range(p, V, W, A, part, at, at + n)
        at += n
    assert bits_equal(part[..., :at], whole[..., :at].cpu().numpy()) and (part[..., at:] == -1.0).all()
