// Tensor-core forward (Sec. 4.2, Alg. 1) for bf16, d = 128 or 64, on sm_100a: TMA-staged Q/K/V tiles, tcgen05 MMAs with
// accumulators in tensor memory, online softmax in registers, bitmap-driven tile skipping.
//
// One CTA owns two consecutive 128-row query tiles of one (batch, head) and walks the union of their active key
// tiles. Bias and mask are folded into the score GEMM: S_w = Q_w K^T gets a ninth k-step whose operands the stager
// warps build per (key tile, query tile) - it adds bias / scale, -BIG for keys that expired before the tile's rows
// and a step function per key that expires inside them - so that the softmax warps read finished scores from tensor
// memory and touch no shared memory per element. Diagonal tiles, and tiles in which more than 13 keys expire inside
// the query tile's rows, take the general path with the explicit test j <= i < expiry[j].
// Warp roles (12 warps):
//   warps 4-7 / 8-11 softmax group 0 / 1: thread r owns query row r of its tile (TMEM lane r): row max, lazy rescale of
//                    O, p = 2^(x c - stab), row sum, P (bf16) written back to tensor memory over S, final normalisation
//   warp 0           producer: builds the tile schedule from the bitmap, then issues the TMA loads of K and V per
//                    active key tile (inactive tiles are never loaded); K and V stages are released separately
//   warp 1           MMA issuer (whole warp, warp-uniform values, one elected lane issues): S_w = Q_w K^T (+ ninth
//                    k-step), O_w += P_w V, ping-ponging between the two query tiles
//   warps 2, 3       stagers for query tile 0 / 1: ninth k-step operands, expiry vector, fast / general flag
// Tensor memory (512 columns): S0 [0,128) S1 [128,256) O0 [256,384) O1 [384,512); P_w aliases columns [0,64) of S_w.
// kD = 64 (its own instantiations): Q, K and V tiles are one 16 KB half tile each (the second half of every buffer stays
// unused), S = Q K^T has four k-steps and the ninth, O_w takes 64 columns.
// The log-sum-exp replaces Alg. 1's (l, m) pair.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <type_traits>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace dma {
namespace {

using namespace ptx;

constexpr int kStages = 2;
constexpr int kMaxSched = 1024;               // key tiles per CTA schedule (L <= 131072)
constexpr int kThreads = 384;
constexpr int kLaunchRegs = 168;             // registers per thread the kernel must be compiled to: its setmaxnreg requests
                                            // (8 warps up by 40, 4 warps down by 80) balance only for this count, and an
                                            // unbalanced request waits forever
constexpr uint32_t kTileBytes = 128 * 128 * 2;   // one 128 x 128 bf16 tile = two 16 KB swizzled half tiles
constexpr int kMaskSlots = 13;                 // keys expiring inside a tile's rows that the ninth k-step can mask
constexpr float kSmallStab = 1048576.0f;        // 2^20: below it the stabiliser is fl(m_ref c), see the softmax groups
constexpr float kRescaleThreshold = 8.0f;     // log2 units: P stays below 2^8, O is rescaled only on larger jumps

struct SharedStorage {
    alignas(1024) uint8_t q[2][kTileBytes];
    alignas(1024) uint8_t k[kStages][kTileBytes];
    alignas(1024) uint8_t v[kStages][kTileBytes];
    // Ninth k-step of S = Q K^T, per query tile: A rows [1, 1, 1, t_0(r) .. t_12(r)], B rows [b_hi, b_mid, b_lo, -BIG [j = j_0] ..],
    // unswizzled K-major core matrices (row r, element e at (r/8) 256 + (e/8) 128 + (r%8) 16 + (e%8) 2 bytes). The
    // product adds bias / scale to the score, -BIG for keys that expired before the tile's rows, and -BIG from row
    // expiry[j_k] on for the up to 13 keys j_k that expire inside the tile's rows (t_k(r) = 1 from that row on).
    // Token-compacted mode: the A rows are constant and elements 8-15 of every row zero, so the same 16 KB hold, in blocks of
    // 2 KB (128 rows x 16 bytes): ones | B of stage 0, tile 0 | stage 0, tile 1 | stage 1, tile 0 | stage 1, tile 1 | zeros
    // (the descriptors' second core matrix is the block of zeros), and the stager runs a whole slice ahead of the S products.
    alignas(128) uint8_t aext[2][4096];
    alignas(128) uint8_t bext[2][4096];
    alignas(16) int len[kStages][128];        // expiry[j] (0 beyond L): row i keeps key j iff j <= i < expiry[j]
    alignas(16) int jidx[kStages][128];       // token-compacted mode: the key index of each gathered column
    int thr[2][16];                           // stager scratch: row thresholds of the keys that expire inside the tile
    uint32_t fast[kStages][2];                // bit 0: the extra k-step carries the whole mask of this (key tile, query tile);
                                              // token-compacted mode: bit q (0-3) = 32-column chunk q needs the per-element test;
                                              // bits 8-15: 16-key blocks that hold a key some row of the query tile may keep
    uint32_t sched[kMaxSched];                // key tile | use by tile 0 << 30 | use by tile 1 << 31
    uint64_t q_full, k_full[kStages], v_full[kStages], k_empty[kStages], v_empty[kStages];
    uint64_t s_full[2], p_half[2], p_ready[2], o_done[2], merge, ref_set[2][4];
    uint32_t tmem_base;
    int n_iters;
    int abort_flag;
    // One query tile per CTA (kSplit): a group's flags, `fast`, and what its per-element test reads are in two slots that its entries take
    // in turn. Token-compacted: group 1's len and jidx. Tile mode: a byte per column, expiry[j] relative to the query tile's first row, cut
    // to [0, 128]: row r of the tile keeps the key iff r is below it (and, in the diagonal tile, not below the column).
    union {
        struct { alignas(16) int len1[2][128], jidx1[2][128]; };
        alignas(16) uint8_t last[2][2][128];
    };
};
static_assert(sizeof(SharedStorage) + 1024 <= 232448, "shared memory of a CTA");
static_assert(kStages == 2 && offsetof(SharedStorage, bext) == offsetof(SharedStorage, aext) + 2 * 4096,
              "token-compacted mode takes aext and bext as six blocks of 2 KB in a row: ones, two stages of two tiles, zeros");

struct FwdParams {
    const float* bias;
    const int32_t* expiry;
    const uint32_t* bitmap;
    __nv_bfloat16* O;
    float* lse;
    int32_t* status;
    int B, Hq, G, L, Tr, Tc, Wd, ignore_bitmap;
    float scale_log2;                          // softmax scale * log2(e)
    float inv_scale;                           // 1 / softmax scale
    float rescale_gap;                         // growth of a row max (score units) beyond which O is rescaled
    // token-compacted mode: per (batch, head, pair of query tiles) the list of keys that some row of the
    // pair keeps (see compact_lists_kernel), padded with -1 to a multiple of 128 (ccap entries per list), and its length
    const int* cidx;
    const int* ccnt;
    const __nv_bfloat16* Kg;                   // K and V base pointers for the row gathers (strides below)
    const __nv_bfloat16* Vg;
    int ccap, Hkv;
    int causal;                                // 0: key j is visible to every row (token-compacted mode only)
    int Lq, q_off, Trq;                        // chunk of query rows (token-compacted mode only): Q, O, lse hold rows q_off .. q_off + Lq - 1; Trq = its 128-row tiles
    int64_t os_b, os_l, os_h;
    int64_t ks_b, ks_l, ks_h, vs_b, vs_l, vs_h;
};


__device__ __forceinline__ uint32_t use_bit(uint32_t entry, int w) { return (entry >> (30 + w)) & 1u; }

// Warp roles. The four service warps come FIRST: among ready warps the schedulers favour the older (lower-numbered) ones,
// and a stager that gets an issue slot only when both softmax warps of its scheduler stall was measured to need ~3600
// cycles for the few hundred instructions of one key tile.
constexpr int kWarpProducer = 0, kWarpIssuer = 1, kWarpStager0 = 2, kWarpStager1 = 3, kFirstSoftmaxWarp = 4;

// kCompact: instead of walking the active 128-key tiles of the bitmap, the CTA walks its gathered key list (keys that
// at least one of its 256 query rows keeps, at most w + 256 of them). Warps 0 and 3 fetch the K and V rows with 16-byte
// asynchronous copies into the swizzled tile layout (TMA row gathers of four rows were measured at ~70 cycles per
// request: too slow), warp 2 builds the B rows of the ninth k-step (bias, and -BIG for columns no row of the tile keeps; the A
// rows are constant) and flags the 32-column chunks that still need the per-element test.
// kBlockSkip: MMA-block skipping inside executed tiles (DMA_FLAG_BLOCK_SKIP), a separate instantiation so that the
// default kernel carries none of its code (the kernel is sensitive to the size of its service warps' loops).
// kSplit: the CTA owns ONE query tile and its two softmax groups take the key tiles (slices) in turn, entry t of the schedule by
// group t & 1. A CTA's walk is then half as long, for grids that leave SMs idle (fwd_tiles). Both groups' products go to one
// accumulator in the order of the schedule, and the row references and row sums are handed from entry to entry: O and lse have the bits
// of the kernel with two query tiles, so that they do not depend on how many heads share the call.
template <bool kCompact, bool kBlockSkip, int kD, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
           const __grid_constant__ CUtensorMap tmV, const FwdParams P) {
    static_assert(kD == 128 || kD == 64, "head dimensions of the tensor-core kernels");
    static_assert(!(kSplit && kBlockSkip), "no blocks are skipped where the groups share a query tile");
    constexpr int kHalves = kD / 64;                         // 64-channel (128-byte) swizzled half tiles per operand tile
    constexpr uint32_t kLoadBytes = kHalves * (kTileBytes / 2);
    extern __shared__ uint8_t smem_raw[];
    SharedStorage& S = *reinterpret_cast<SharedStorage*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    pdl_enter();
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);      // warp-uniform to the compiler: role branches stay uniform
    const int bh = blockIdx.x, b = bh / P.Hq, h = bh % P.Hq, hk = h / P.G;
    const int npairs = (P.Trq + 1) / 2;
    const int unit = (kSplit ? P.Trq : npairs) - 1 - (int)blockIdx.y;  // pair of query tiles (kSplit: query tile), heaviest first
    const int pair = kSplit ? unit >> 1 : unit;
    const int qt0 = kSplit ? unit : 2 * pair, qt1 = kSplit ? unit : 2 * pair + 1;   // query tiles inside the chunk (the whole sequence unless P.q_off / P.Lq say otherwise)
    const bool has1 = !kSplit && qt1 < P.Trq;
    const int lpair = (kCompact && !P.causal) ? 0 : pair;   // non-causal: all rows of a head keep the same keys, one list serves every pair
    volatile int* abort_flag = &S.abort_flag;

    if (tid == 0) {
        mbar_init(&S.q_full, 1);
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&S.k_full[s], kCompact ? 33 : 3);   // K: TMA bytes + the two stager warps | 32 gathering lanes + the stager warp
            mbar_init(&S.v_full[s], kCompact ? 32 : 1);
            mbar_init(&S.k_empty[s], 1);
            mbar_init(&S.v_empty[s], 1);
        }
        for (int w = 0; w < 2; ++w) {
            mbar_init(&S.s_full[w], 1);
            mbar_init(&S.p_half[w], 4);          // one arrival per softmax warp
            mbar_init(&S.p_ready[w], 4);
            mbar_init(&S.o_done[w], 1);
        }
        mbar_init(&S.merge, kSplit ? 8 : 4);      // (unused with two query tiles; with another count than its neighbours' that instance was 1.5 % slower)
        for (int q = 0; q < 8; ++q) mbar_init(&S.ref_set[q >> 2][q & 3], 1);
        S.abort_flag = 0;
        S.n_iters = 0;
        fence_barrier_init();
    }
    // Token-compacted mode: a gather warp fetches the first slice's keys beside the list's length, before the CTA's barrier. (Behind it, 16 heads of 4096 keys 64.1
    // against 63.1 us, last 2048 rows of 16384 keys 101.0 / 99.0, 16 heads of 65536 2180 / 2080; with the rows' copies ahead of the barrier too it is no faster.)
    const bool isK = warp == kWarpProducer;
    int2 jrow[kCompact ? 16 : 1];
    int listed = 0, n_plain = 0;
    const int* list = nullptr;
    const int rsub = (lane >> 3) * 2;              // lanes 8 g .. 8 g + 7 take the rows 8 m + 2 g and 8 m + 2 g + 1
    // Slices without padding, rows less than 4 GB apart (all but a list's last slice): three instructions per row. What the gather warps issue, the softmax
    // warps of the same scheduler wait for: with seven, and a load per row, a slice's exponentials beside a gather took up to 470 clk more. Forward, us,
    // before / now: 16 heads of 4096 keys 67.5 / 63.6, last 2048 rows of 16384 108.6 / 99.5, 32 heads of 16384 643 / 600, 16 of 65536 2400 / 2150.
    auto gather = [&](int it) {
        const int st = it % kStages;
        const int64_t row_stride = isK ? P.ks_l : P.vs_l;
        const __nv_bfloat16* src = (isK ? P.Kg + b * P.ks_b + hk * P.ks_h : P.Vg + b * P.vs_b + hk * P.vs_h) + (lane & 7) * 8;
        const uint32_t sw0 = (uint32_t)(((lane & 7) ^ rsub) << 4), sw1 = (uint32_t)(((lane & 7) ^ (rsub + 1)) << 4) + 128;
        const uint32_t step = (uint32_t)row_stride * 2u;
        uint8_t* dst = (isK ? S.k[st] : S.v[st]) + rsub * 128;
        if (it < n_plain) {
            const uint32_t d0 = smem_u32(dst) + sw0, d1 = smem_u32(dst) + sw1;
            const char* base = reinterpret_cast<const char*>(src);
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                const char* r0 = base + (uint64_t)(uint32_t)jrow[kCompact ? m : 0].x * step;
                const char* r1 = base + (uint64_t)(uint32_t)jrow[kCompact ? m : 0].y * step;
                cp_async16_at(d0 + m * 1024, r0);
                if constexpr (kD == 128) cp_async16_at(d0 + m * 1024 + kTileBytes / 2, r0 + 128);
                cp_async16_at(d1 + m * 1024, r1);
                if constexpr (kD == 128) cp_async16_at(d1 + m * 1024 + kTileBytes / 2, r1 + 128);
            }
        } else {
            // (a list's last slice: its keys are read again. Out of jrow, which unrolls this branch, the kernel is slower: 16 heads of 4096 keys 63.1 -> 65.6 us, of 3000 (w = 90) 28.3 -> 29.4)
#pragma unroll 4
            for (int q = 0; q < 32; ++q) {
                const int j = list[it * 128 + 8 * (q >> 1) + (q & 1)];
                const __nv_bfloat16* row = src + (int64_t)max(j, 0) * row_stride;
                uint8_t* d = dst + (q >> 1) * 1024 + ((q & 1) ? sw1 : sw0);          // row r, chunk c ^ (r & 7)
                cp_async16(d, row, j >= 0 ? 16 : 0);
                if constexpr (kD == 128) cp_async16(d + kTileBytes / 2, row + 64, j >= 0 ? 16 : 0);
            }
        }
    };
    if constexpr (kCompact) {
        if (warp == kWarpProducer || warp == kWarpStager1) {
            list = P.cidx + ((size_t)bh * npairs + lpair) * P.ccap + rsub;
            listed = P.ccnt[(size_t)bh * npairs + lpair];              // (beyond the capacity: there may be padding anywhere)
#pragma unroll
            for (int m = 0; m < 16; ++m) jrow[m] = *reinterpret_cast<const int2*>(list + 8 * m);
            const int64_t row_stride = isK ? P.ks_l : P.vs_l;
            n_plain = listed <= P.ccap && row_stride > 0 && row_stride < (1ll << 31) ? listed / 128 : 0;
        }
    }
    if (warp == kWarpIssuer) {
        tmem_alloc(&S.tmem_base, 512);
        tmem_relinquish();
    }
    // tile mode: the workspace header is cleared here (a wait that times out writes the status a second later at the earliest)
    if (!kCompact && blockIdx.x == 0 && blockIdx.y == 0 && tid < kWsHeaderBytes / 4) P.status[tid] = 0;
    if (warp == kWarpProducer) {
        // schedule: ascending key tiles that at least one of the two query tiles uses
        if (lane == 0) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); }
        int n = 0;
        if constexpr (kCompact) {
            // every 128-key slice of the gathered list, used by both query tiles
            if (listed > P.ccap && lane == 0) atomicExch(P.status, (int32_t)DMA_ERR_MASK_OVERFLOW);
            n = min((min(listed, P.ccap) + 127) / 128, kMaxSched);
            for (int t = lane; t < n; t += 32) S.sched[t] = (uint32_t)t | (kSplit ? 1u << (30 + (t & 1)) : (1u << 30) | (has1 ? (1u << 31) : 0u));
        } else {
            const int kt_last = min(has1 ? qt1 : qt0, P.Tc - 1);
            for (int base = 0; base <= kt_last; base += 32) {
                const int kt = base + lane;
                uint32_t u0 = 0, u1 = 0;
                if (kt <= kt_last) {
                    u0 = kt <= qt0 && (P.ignore_bitmap || bitmap_test(P.bitmap, P.Tr, P.Wd, bh, qt0, kt));
                    u1 = has1 && kt <= qt1 && (P.ignore_bitmap || bitmap_test(P.bitmap, P.Tr, P.Wd, bh, qt1, kt));
                }
                const uint32_t act = __ballot_sync(0xffffffffu, u0 | u1);
                const int at = n + __popc(act & ((1u << lane) - 1));
                if (u0 | u1) S.sched[at] = (uint32_t)kt | (kSplit ? 1u << (30 + (at & 1)) : (u0 << 30) | (u1 << 31));
                n += __popc(act);
            }
        }
        if (lane == 0) S.n_iters = n;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    const int n_iters = S.n_iters;

    if (warp >= kFirstSoftmaxWarp) {
        // =========================================== softmax groups ===========================================
        setmaxnreg_inc<208>();
        const int w = (warp - kFirstSoftmaxWarp) >> 2;
        const int r = tid & 127;
        const int qt = w ? qt1 : qt0;
        const int il = qt * 128 + r;                        // row inside Q, O, lse
        const int i = P.q_off + il;                         // its position in the sequence
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_base + w * 128;
        const uint32_t tO = tmem + lane_base + 256 + (kSplit ? 0 : w * 128);
        const uint32_t rows4 = (uint32_t)r * 0x01010101u;
        float m_ref = -INFINITY, r_ref = 0.0f, l = 0.0f;
        float f_last = 1.0f, s_last = 0.0f;                 // kSplit: the group's last entry, its factor and its row sum, not yet handed over
        // kSplit, in the second query tile's buffer: per group and row the reference maximum after the group's last entry and the row sum up
        // to its entry before that one; in the end f_last and s_last
        float2 (*handed)[128] = reinterpret_cast<float2 (*)[128]>(S.q[1]);
        int n_used = 0;
        bool ok = true;
        for (int it = 0; it < n_iters && ok; ++it) {
            const uint32_t entry = S.sched[it];
            if (!use_bit(entry, w)) continue;
            const int st = kSplit ? n_used & 1 : it % kStages, j0 = (int)(entry & 0xFFFFF) * 128;
            ok = mbar_wait_warp(&S.s_full[w], n_used & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            // The stagers' flag is read only now. The S product was issued after k_full[st] completed, so the flag of THIS
            // iteration is in place. (Waiting on k_full[st] here instead is wrong: a tile that skipped earlier key tiles
            // has not followed that barrier's phases, and a parity wait on a barrier it is a whole phase ahead of returns
            // at once, before the stager has written the flag.)
            const uint32_t tile_flags = S.fast[st][w];
            const bool fast_tile = kCompact || (tile_flags & 1u) != 0;      // token-compacted mode: the low bits are a chunk mask instead
            // The accumulator holds q.k + bias / scale (+ -BIG where the ninth k-step masks). On the fast path that
            // is the whole masked score; otherwise (diagonal tile, or more than 13 keys expiring inside the tile's
            // rows) the validity test j <= i < expiry[j] is applied here. x = log2e * scale * score, -inf if masked.
            float x[128];
            {
                uint32_t raw[128];                 // the four loads are in flight together, one wait
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld32p(tS + c * 32, &raw[c * 32]);
                tc_wait_ld();
#pragma unroll
                for (int u = 0; u < 128; ++u) x[u] = __uint_as_float(raw[u]);
            }
            float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
            if (kCompact && (kSplit || (tile_flags & 15u))) {
                // gathered columns: bias and the keys that are gone for the whole tile are already in the score; the
                // per-element test is needed only in the 32-column chunks the stager flagged (a key expiring or
                // entering inside the tile's rows). Most slices have none, and one test for all four chunks skips the four branches: 250 clk of a slice's
                // 4400, 32 heads of 16384 keys 683 -> 640 us, 16 of 65536 2625 -> 2360. (One query tile per CTA: 50.6 -> 53.5, so not there.)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if ((tile_flags >> q) & 1u) {
                        const int* le = kSplit && w ? S.len1[st] : S.len[st];
                        const int* ji = kSplit && w ? S.jidx1[st] : S.jidx[st];
#pragma unroll
                        for (int c = 32 * q; c < 32 * q + 32; c += 4) {
                            const int4 ee = *reinterpret_cast<const int4*>(&le[c]);
                            const int4 jj = *reinterpret_cast<const int4*>(&ji[c]);
                            const int ev[4] = {ee.x, ee.y, ee.z, ee.w}, jv[4] = {jj.x, jj.y, jj.z, jj.w};
#pragma unroll
                            for (int u = 0; u < 4; ++u) x[c + u] = (jv[u] <= i && i < ev[u]) ? x[c + u] : -INFINITY;
                        }
                    }
                }
            }
            if (fast_tile) {
#pragma unroll
                for (int c = 0; c < 128; c += 4) {
                    mxa[(c >> 2) & 1] = max3(mxa[(c >> 2) & 1], x[c], x[c + 1]);
                    mxa[2 + ((c >> 2) & 1)] = max3(mxa[2 + ((c >> 2) & 1)], x[c + 2], x[c + 3]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) mxa[u] = mxa[u] < -1e20f ? -INFINITY : mxa[u];
            } else if constexpr (kSplit) {
                // four columns per word, bit 7 of a byte: r < last, and in the diagonal tile column <= r
                const bool diag = (int)(entry & 0xFFFFF) == qt;
                const uint32_t step = diag ? 0x04040404u : 0u, seen0 = diag ? 0x80808080u + rows4 - 0x03020100u : 0x80808080u;
#pragma unroll
                for (int h4 = 0; h4 < 8; ++h4) {
                    const uint4 t4 = *reinterpret_cast<const uint4*>(&S.last[st][w][16 * h4]);
                    const uint32_t tw[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const int c = 16 * h4 + 4 * g;
                        const uint32_t keep = (tw[g] + (0x7F7F7F7Fu - rows4)) & (seen0 - (uint32_t)(4 * h4 + g) * step);
#pragma unroll
                        for (int u = 0; u < 4; ++u) x[c + u] = (keep & (0x80u << (8 * u))) ? x[c + u] : -INFINITY;
                        mxa[g & 1] = max3(mxa[g & 1], x[c], x[c + 1]);
                        mxa[2 + (g & 1)] = max3(mxa[2 + (g & 1)], x[c + 2], x[c + 3]);
                    }
                }
            } else {
#pragma unroll
                for (int c = 0; c < 128; c += 4) {
                    const int4 ee = *reinterpret_cast<const int4*>(&S.len[st][c]);
                    const int ev[4] = {ee.x, ee.y, ee.z, ee.w};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const bool valid = j0 + c + u <= i && i < ev[u];
                        x[c + u] = valid ? x[c + u] : -INFINITY;
                        mxa[u] = fmaxf(mxa[u], x[c + u]);
                    }
                }
            }
            // The running max m_ref stays in score units and the exponent is formed as (x - m_ref) * c: the difference
            // is exact for the entries that matter, whatever the magnitude of the bias.
            const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3]));
            float m_new = fmaxf(m_ref, mx);
            bool grown = false;
            float before = -INFINITY;
            if constexpr (kSplit) {
                // Entry it - 1's reference comes from the other group (the warp with the same rows), this entry's is published before the
                // exponentials. (With a reference of its own per group P was rounded at other places: O 1.7e-3 away, dA, a sum that
                // cancels, by up to 1e-2.) The row sum travels with it two entries late, when its terms are known.
                float2 from = make_float2(-INFINITY, 0.0f);                 // (row sum up to entry it - 3)
                if (it > 0) {
                    ok = mbar_wait_warp(&S.ref_set[w ^ 1][warp & 3], ((it - 1) >> 1) & 1, abort_flag);
                    if (!ok) break;
                    from = handed[w ^ 1][r];
                }
                before = from.x;
                m_new = fmaxf(before, mx);
                grown = it > 0 && __any_sync(0xffffffffu, m_new > before + P.rescale_gap);
                if (it > 0 && !grown) m_new = before;
                // (the other group has read the values before it published its own last ones)
                handed[w][r] = make_float2(m_new, __fadd_rn(__fmul_rn(from.y, f_last), s_last));
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.ref_set[w][warp & 3]);
                f_last = 1.0f;
            }
            auto stab_resid = [&](float m) {           // m c - stab(m); 0 for m = -inf
                const float mm = (m == -INFINITY) ? 0.0f : m;
                const float Mm = mm * P.scale_log2;
                return fabsf(Mm) < kSmallStab ? fmaf(mm, P.scale_log2, -Mm) : 0.0f;
            };
            if (kSplit ? !grown : n_used == 0) {
                m_ref = m_new;
                if constexpr (!kSplit) r_ref = stab_resid(m_ref);
            } else if (kSplit || __any_sync(0xffffffffu, m_new > m_ref + P.rescale_gap)) {
                // O_w *= 2^(stab(m_ref) - stab(m_new)): the previous P V product must have landed first (kSplit: that of entry it - 1, after which
                // nothing is added until this entry's P is released)
                ok = kSplit ? mbar_wait_warp(&S.o_done[w ^ 1], ((it - 1) >> 1) & 1, abort_flag) : mbar_wait_warp(&S.o_done[w], (n_used - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if constexpr (kSplit) {
                    m_ref = before;
                    r_ref = stab_resid(before);
                }
                const float r_new = stab_resid(m_new);
                const float f = (m_new == -INFINITY) ? 1.0f : (m_ref == -INFINITY) ? 0.0f : ex2(fmaf(m_ref - m_new, P.scale_log2, r_new - r_ref));
#pragma unroll
                for (int c = 0; c < kD / 32; ++c) {
                    uint32_t o[32];
                    tmem_ld32(tO + c * 32, o);
                    tc_wait_ld();
#pragma unroll
                    for (int u = 0; u < 32; ++u) o[u] = __float_as_uint(__uint_as_float(o[u]) * f);
                    tmem_st32(tO + c * 32, o);
                }
                tc_wait_st();
                if constexpr (kSplit) f_last = f;
                else l *= f;
                m_ref = m_new;
                r_ref = r_new;
            }
            // p = 2^(x c - stab(m_ref)). The stabiliser is a function of the row's m_ref alone: fl(m_ref c) while that
            // is below 2^20 in magnitude (then x c - stab is one FMA per element and fl() is off by < 0.07), else the
            // exact product m_ref c, reached by taking the exact difference x - m_ref first (bias magnitudes up to the
            // fp32 range stay safe). r_ref = m_ref c - stab(m_ref) travels with m_ref.
            const float m_use = (m_ref == -INFINITY) ? 0.0f : m_ref;
            const float M = m_use * P.scale_log2, nM = -M;
            const float resid = kSplit ? stab_resid(m_ref) : r_ref;
            const bool small = __all_sync(0xffffffffu, fabsf(M) < kSmallStab);
            // Pairs of columns: one packed FMA for two arguments, one packed add for two terms of the row sum. The loop is bound by issue slots as much as by the
            // exponentials; two FMAs and two adds per pair instead: 16 heads of 4096 keys 72.2 against 69.2 us, 32 heads of 8192 keys at d = 64 189 against 179.
            float sa[4] = {0.f, 0.f, 0.f, 0.f};
            float2 sum2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            const float2 c2 = make_float2(P.scale_log2, P.scale_log2), nM2 = make_float2(nM, nM);
            if (small) {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t pk[32];
#pragma unroll
                    for (int c = 0; c < 64; c += 2) {
                        const float2 y = fma2(make_float2(x[half * 64 + c], x[half * 64 + c + 1]), c2, nM2);
                        const float2 p = make_float2(ex2(y.x), ex2(y.y));
                        sum2[(c >> 1) & 1] = add2(sum2[(c >> 1) & 1], p);
                        pk[c >> 1] = pack_bf16(p.x, p.y);
                    }
                    tmem_st32(tS + half * 32, pk);
                    if (half == 0) {          // keys 0-63 of P are complete: their half of P V can start now
                        tc_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&S.p_half[w]);
                    }
                }
            } else {
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t pk[32];
#pragma unroll
                    for (int c = 0; c < 64; c += 2) {
                        const float2 p = make_float2(ex2(fmaf(x[half * 64 + c] - m_use, P.scale_log2, resid)),
                                                     ex2(fmaf(x[half * 64 + c + 1] - m_use, P.scale_log2, resid)));
                        // (tile mode keeps a sum of its own here: with the packed one the compiler's other loop is 4 % slower, 155 -> 161 us at 32 heads
                        // of 4096; token-compacted the other way round, 98 -> 103 for the last 2048 rows of 16384 keys)
                        if constexpr (kCompact) sum2[(c >> 1) & 1] = add2(sum2[(c >> 1) & 1], p);
                        else sa[(c >> 1) & 3] += p.x + p.y;
                        pk[c >> 1] = pack_bf16(p.x, p.y);
                    }
                    tmem_st32(tS + half * 32, pk);
                    if (half == 0) {
                        tc_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&S.p_half[w]);
                    }
                }
            }
            sa[0] += sum2[0].x + sum2[0].y;
            sa[1] += sum2[1].x + sum2[1].y;
            const float sum = (sa[0] + sa[1]) + (sa[2] + sa[3]);
            if constexpr (kSplit) s_last = sum;
            else l += sum;
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.p_ready[w]);      // one arrival per warp: 128 serialised arrivals cost ~400 cycles
            ++n_used;
        }
        // epilogue: O_w / l -> bf16 rows, log-sum-exp in natural log. kSplit: each group writes half of the channels
        const bool exists = w == 0 || has1 || kSplit;
        if constexpr (kSplit) {
            handed[2 + w][r] = make_float2(f_last, s_last);
            __syncwarp();
            if (ok && lane == 0) mbar_arrive(&S.merge);
            if (ok) ok = mbar_wait_warp(&S.merge, 0, abort_flag);
            const int a = (n_iters - 1) & 1;                     // the group of the last entry
            if (ok && n_iters > 0) {
                m_ref = handed[a][r].x;
                l = handed[a][r].y;
                const float m_use = m_ref == -INFINITY ? 0.0f : m_ref, M = m_use * P.scale_log2;
                r_ref = fabsf(M) < kSmallStab ? fmaf(m_use, P.scale_log2, -M) : 0.0f;
                if (n_iters > 1) l = __fadd_rn(__fmul_rn(l, handed[2 + (a ^ 1)][r].x), handed[2 + (a ^ 1)][r].y);
                l = __fadd_rn(__fmul_rn(l, handed[2 + a][r].x), handed[2 + a][r].y);
            }
            // (the entry before the last one first: a wait for a phase that is two ahead would not wait)
            if (ok && n_iters > 1) ok = mbar_wait_warp(&S.o_done[a ^ 1], ((n_iters - 2) >> 1) & 1, abort_flag);
            if (ok && n_iters > 0) ok = mbar_wait_warp(&S.o_done[a], ((n_iters - 1) >> 1) & 1, abort_flag);
            // (no entry at all: nothing above has waited for the load of Q, whose buffer is written next)
            if (ok && n_iters == 0) ok = mbar_wait_warp(&S.q_full, 0, abort_flag);
        } else if (ok && exists && n_used > 0) {
            ok = mbar_wait_warp(&S.o_done[w], (n_used - 1) & 1, abort_flag);
        }
        if (ok && exists) {
            tc_fence_after();
            const float inv = l > 0.0f ? 1.0f / l : 0.0f;
            if constexpr (kSplit) n_used = n_iters;
            if constexpr (kSplit) {
                // Each group writes half of the channels. A thread holds a row: a warp turns its 32 rows around in the Q buffer, which the last S product
                // has left (16-byte chunks swizzled by the row), so that neighbouring lanes write neighbouring 16 bytes of a row instead of 32 rows
                // per instruction. 8 heads of 4096 keys (w = 2048) 50.9 -> 49.3 us. (With two query tiles the two groups' ends overlap, and 66.6 -> 70.4 at 16 heads of 4096.)
                uint8_t* turn = S.q[0] + (warp & 3) * 4096 + (kD == 128 ? w * (kTileBytes / 2) : 0);
                constexpr int kLanes = kD == 128 ? 8 : 4, kRowsPer = 32 / kLanes;      // lanes per row, rows per instruction
                const int ch0 = kD == 128 ? 0 : 4 * w;
#pragma unroll
                for (int c = 0; c < kD / 64; ++c) {
                    uint32_t o[32];
                    if (n_used > 0) {
                        tmem_ld32(tO + w * (kD / 2) + c * 32, o);
                        tc_wait_ld();
                    } else {
#pragma unroll
                        for (int u = 0; u < 32; ++u) o[u] = 0;
                    }
#pragma unroll
                    for (int u = 0; u < 32; u += 8) {
                        uint4 pkt;
                        pkt.x = pack_bf16(__uint_as_float(o[u]) * inv, __uint_as_float(o[u + 1]) * inv);
                        pkt.y = pack_bf16(__uint_as_float(o[u + 2]) * inv, __uint_as_float(o[u + 3]) * inv);
                        pkt.z = pack_bf16(__uint_as_float(o[u + 4]) * inv, __uint_as_float(o[u + 5]) * inv);
                        pkt.w = pack_bf16(__uint_as_float(o[u + 6]) * inv, __uint_as_float(o[u + 7]) * inv);
                        *reinterpret_cast<uint4*>(turn + lane * 128 + (((ch0 + c * 4 + (u >> 3)) ^ (lane & 7)) << 4)) = pkt;
                    }
                }
                __syncwarp();
                const int ch = ch0 + lane % kLanes, rsub = lane / kLanes, row0 = qt * 128 + (warp & 3) * 32 + rsub;
                __nv_bfloat16* orow = P.O + b * P.os_b + (int64_t)row0 * P.os_l + h * P.os_h + (kD == 128 ? w * 64 : 0) + ch * 8;
#pragma unroll
                for (int t = 0; t < kLanes; ++t) {
                    const int rr = t * kRowsPer + rsub;
                    const uint4 v = *reinterpret_cast<const uint4*>(turn + rr * 128 + ((ch ^ (rr & 7)) << 4));
                    if (row0 + t * kRowsPer < P.Lq) *reinterpret_cast<uint4*>(orow + (int64_t)(t * kRowsPer) * P.os_l) = v;
                }
            } else {
            __nv_bfloat16* orow = P.O + b * P.os_b + (int64_t)il * P.os_l + h * P.os_h;
            constexpr int kUnroll = kCompact ? 1 : kD / 32;                // (rolled: 8 bytes of spills less, 32 heads of 16384 keys 690 -> 666 us)
#pragma unroll kUnroll
            for (int c = 0; c < kD / 32; ++c) {
                uint32_t o[32];
                if (n_used > 0) {
                    tmem_ld32(tO + c * 32, o);
                    tc_wait_ld();
                } else {
#pragma unroll
                    for (int u = 0; u < 32; ++u) o[u] = 0;
                }
                if (il < P.Lq) {
#pragma unroll
                    for (int u = 0; u < 32; u += 8) {
                        uint4 pkt;
                        pkt.x = pack_bf16(__uint_as_float(o[u]) * inv, __uint_as_float(o[u + 1]) * inv);
                        pkt.y = pack_bf16(__uint_as_float(o[u + 2]) * inv, __uint_as_float(o[u + 3]) * inv);
                        pkt.z = pack_bf16(__uint_as_float(o[u + 4]) * inv, __uint_as_float(o[u + 5]) * inv);
                        pkt.w = pack_bf16(__uint_as_float(o[u + 6]) * inv, __uint_as_float(o[u + 7]) * inv);
                        *reinterpret_cast<uint4*>(orow + c * 32 + u) = pkt;
                    }
                }
            }
            }
            if (il < P.Lq && (!kSplit || w == 0)) P.lse[(size_t)bh * P.Lq + il] = l > 0.0f ? 0.6931471805599453f * ((m_ref * P.scale_log2 - r_ref) + log2f(l)) : -INFINITY;
        }
    } else {
        setmaxnreg_dec<88>();   // 4 warps x 80 registers released = 8 warps x 40 acquired above
        if (kCompact && (warp == kWarpProducer || warp == kWarpStager1)) {
            // ================================ token-compacted mode: gather warps ================================
            // Warp 0 fetches the K rows of each 128-key slice of the gathered list, warp 3 the V rows: 16-byte
            // asynchronous copies into the 128-byte-swizzled tile layout (8 lanes per 128-byte half row, 4 rows per
            // instruction; padding entries (-1) are zero-filled). Each lane's copies report to the stage's barrier.
            if (isK && lane == 0) {
                mbar_arrive_expect_tx(&S.q_full, has1 ? 2 * kLoadBytes : kLoadBytes);
                for (int w = 0; w < (has1 ? 2 : 1); ++w)
                    for (int hf = 0; hf < kHalves; ++hf)
                        tma_load_4d(&S.q[w][hf * (kTileBytes / 2)], &tmQ, &S.q_full, hf * 64, (qt0 + w) * 128, h, b);
            }
            bool ok = true;
            for (int it = 0; it < n_iters && ok; ++it) {
                const int st = it % kStages;
                uint64_t* empty = isK ? &S.k_empty[st] : &S.v_empty[st];
                uint64_t* full = isK ? &S.k_full[st] : &S.v_full[st];
                if (it >= kStages) ok = mbar_wait_warp(empty, ((it / kStages) - 1) & 1, abort_flag);
                if (!ok) break;
                gather(it);
                cp_async_arrive(full);
                if (it + 1 < n_iters) {
#pragma unroll
                    for (int m = 0; m < 16; ++m) jrow[m] = *reinterpret_cast<const int2*>(list + (it + 1) * 128 + 8 * m);
                }
            }
            for (int it = max(0, n_iters - kStages); it < n_iters && ok; ++it)
                ok = mbar_wait_warp(isK ? &S.k_empty[it % kStages] : &S.v_empty[it % kStages], (it / kStages) & 1, abort_flag);
        } else if (kCompact && warp == kWarpStager0) {
            // ================================ token-compacted mode: stager ================================
            // Per 128-key slice and query tile: the B rows of the ninth k-step (bias / scale as three bf16 terms, or
            // -BIG for a column that no row of the tile keeps; the A rows are constant ones), the key index and expiry
            // vectors, and the mask of 32-column chunks that hold a key expiring or entering inside the tile's rows (only
            // those need the per-element test). Two dependent levels of global loads, each issued a tile ahead.
            constexpr uint32_t kOne = 0x3F80u, kNegBig = 0xF14Au;     // bf16 1.0 and about -1e30
            uint8_t* ext = &S.aext[0][0];
            for (int r = lane; r < 128; r += 32) {
                *reinterpret_cast<uint4*>(ext + r * 16) = make_uint4(kOne | (kOne << 16), kOne, 0u, 0u);
                *reinterpret_cast<uint4*>(ext + 5 * 2048 + r * 16) = make_uint4(0u, 0u, 0u, 0u);
            }
            const int* list = P.cidx + ((size_t)bh * npairs + lpair) * P.ccap;
            auto vals = [&](const int (&jv)[4], float (&bv)[4], int (&ev)[4]) {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    bv[t] = jv[t] >= 0 ? P.bias[(size_t)bh * P.L + jv[t]] : 0.0f;
                    ev[t] = jv[t] >= 0 ? P.expiry[(size_t)bh * P.L + jv[t]] : 0;
                }
            };
            int jv[4] = {-1, -1, -1, -1}, jn[4] = {-1, -1, -1, -1}, ev[4] = {0, 0, 0, 0};
            float bv[4] = {0.f, 0.f, 0.f, 0.f};
            if (n_iters > 0) {
#pragma unroll
                for (int t = 0; t < 4; ++t) jv[t] = list[lane + 32 * t];
                vals(jv, bv, ev);
            }
            if (n_iters > 1) {
#pragma unroll
                for (int t = 0; t < 4; ++t) jn[t] = list[128 + lane + 32 * t];
            }
            bool ok = true;
            for (int it = 0; it < n_iters && ok; ++it) {
                const int st = it % kStages;
                float bn[4] = {0.f, 0.f, 0.f, 0.f};
                int en[4] = {0, 0, 0, 0}, jnn[4] = {-1, -1, -1, -1};
                if (it + 1 < n_iters) vals(jn, bn, en);
                if (it + 2 < n_iters) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) jnn[t] = list[(it + 2) * 128 + lane + 32 * t];
                }
                // rows and flags are formed in registers before the waits
                uint32_t b0[2][4], b1[4], flags[2] = {0u, 0u}, live[2] = {0u, 0u};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float bsc = bv[t] * P.inv_scale;
                    const __nv_bfloat16 hi = __float2bfloat16_rn(bsc);
                    const float r1 = bsc - __bfloat162float(hi);
                    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
                    const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
                    const uint32_t w0 = (uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(mid) << 16);
                    b1[t] = (uint32_t)__bfloat16_as_ushort(lo);
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        const int i0 = P.q_off + (w ? qt1 : qt0) * 128;
                        const int first = P.causal ? jv[t] : 0;             // first row that can see the key
                        const bool dead = jv[t] < 0 || ev[t] <= i0 || first > i0 + 127;
                        const bool mixed = !dead && (ev[t] < i0 + 128 || first > i0);
                        b0[w][t] = dead ? kNegBig : w0;
                        flags[w] |= __ballot_sync(0xffffffffu, mixed) ? (1u << t) : 0u;
                        if constexpr (kBlockSkip) {
                            const uint32_t alive = __ballot_sync(0xffffffffu, !dead);
                            live[w] |= ((alive & 0xFFFFu) ? 1u : 0u) << (2 * t) | ((alive >> 16) ? 1u : 0u) << (2 * t + 1);
                        }
                    }
                }
                // What this slot holds was last read by the softmax groups before they released P of slice it - kStages,
                // hence before its P V, and by that slice's S products, which were issued before that P V. kSplit: the group's
                // slot was last read for its entry before the last one, and the last one's S product was issued after that P V
                const int slot = kSplit ? (it >> 1) & 1 : st;
                if (it >= kStages) ok = kSplit ? mbar_wait_warp(&S.s_full[it & 1], ((it >> 1) - 1) & 1, abort_flag)
                                               : mbar_wait_warp(&S.v_empty[st], ((it / kStages) - 1) & 1, abort_flag);
                if (!ok) break;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = lane + 32 * t;
                    (kSplit && (it & 1) ? S.jidx1 : S.jidx)[slot][c] = jv[t] >= 0 ? (P.causal ? jv[t] : 0) : 0x7fffffff;  // first row of the key; padding: never <= a row index
                    (kSplit && (it & 1) ? S.len1 : S.len)[slot][c] = ev[t];
#pragma unroll
                    for (int w = 0; w < 2; ++w) {
                        if (kSplit && w != (it & 1)) continue;
                        *reinterpret_cast<uint4*>(ext + (1 + slot * 2 + w) * 2048 + c * 16) =
                            make_uint4(b0[w][t], b0[w][t] == kNegBig ? 0u : b1[t], 0u, 0u);
                    }
                    jv[t] = jn[t]; bv[t] = bn[t]; ev[t] = en[t]; jn[t] = jnn[t];
                }
                if (lane < 2 && (!kSplit || lane == (it & 1))) S.fast[slot][lane] = (lane ? flags[1] : flags[0]) | ((kBlockSkip ? (lane ? live[1] : live[0]) : 0xFFu) << 8);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.k_full[st]);
            }
        } else if (warp == kWarpProducer) {
            // =========================================== producer ===========================================
            if (lane == 0) {
                mbar_arrive_expect_tx(&S.q_full, has1 ? 2 * kLoadBytes : kLoadBytes);
                for (int w = 0; w < (has1 ? 2 : 1); ++w)
                    for (int hf = 0; hf < kHalves; ++hf)
                        tma_load_4d(&S.q[w][hf * (kTileBytes / 2)], &tmQ, &S.q_full, hf * 64, (qt0 + w) * 128, h, b);
            }
            // K and V of a stage are released separately (K once its S = Q K^T products are done, V after P V), so
            // the next K tile is in flight about two key tiles ahead of its use
            bool ok = true;
            for (int it = 0; it < n_iters && ok; ++it) {
                const int st = it % kStages, j0 = (int)(S.sched[it] & 0xFFFFF) * 128;
                if (it >= kStages) ok = mbar_wait_warp(&S.k_empty[st], ((it / kStages) - 1) & 1, abort_flag);
                if (!ok) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&S.k_full[st], kLoadBytes);
                    tma_load_4d(&S.k[st][0], &tmK, &S.k_full[st], 0, j0, hk, b);
                    if constexpr (kD == 128) tma_load_4d(&S.k[st][kTileBytes / 2], &tmK, &S.k_full[st], 64, j0, hk, b);
                }
                if (it >= kStages) ok = mbar_wait_warp(&S.v_empty[st], ((it / kStages) - 1) & 1, abort_flag);
                if (!ok) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&S.v_full[st], kLoadBytes);
                    tma_load_4d(&S.v[st][0], &tmV, &S.v_full[st], 0, j0, hk, b);
                    if constexpr (kD == 128) tma_load_4d(&S.v[st][kTileBytes / 2], &tmV, &S.v_full[st], 64, j0, hk, b);
                }
            }
            // tail: the last stages' release arrivals must land before the CTA's shared memory is given up
            for (int it = max(0, n_iters - kStages); it < n_iters && ok; ++it)
                ok = mbar_wait_warp(&S.k_empty[it % kStages], (it / kStages) & 1, abort_flag) &&
                     mbar_wait_warp(&S.v_empty[it % kStages], (it / kStages) & 1, abort_flag);
        } else if (warp == kWarpStager0 || warp == kWarpStager1) {
            // =========================================== stagers ===========================================
            // Warp 2 + w serves query tile w: per key tile it builds the ninth k-step operands described at
            // SharedStorage (warp 2 also stages the expiry vector for the general softmax path). The global loads run
            // one tile ahead and the rows are formed in registers before the wait for the blocks to be free, so that
            // only the stores are left between the previous S product and the next one.
            const int w = warp - kWarpStager0;
            const int i0 = (w ? qt1 : qt0) * 128;
            // key indices of a tile's columns, then their bias and expiry, loaded one tile before they are needed
            auto fetch_idx = [&](int it, int (&jv)[4]) {
                const int j0 = (int)(S.sched[it] & 0xFFFFF) * 128;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    jv[t] = j0 + lane + 32 * t;
                }
            };
            auto fetch_vals = [&](const int (&jv)[4], float (&bv)[4], int (&ev)[4]) {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const bool real = jv[t] >= 0 && jv[t] < P.L;
                    bv[t] = real ? P.bias[(size_t)bh * P.L + jv[t]] : 0.0f;
                    ev[t] = real ? P.expiry[(size_t)bh * P.L + jv[t]] : 0;
                }
            };
            constexpr uint32_t kOne = 0x3F80u, kNegBig = 0xF14Au;     // bf16 1.0 and about -1e30
            float bv[4] = {0.f, 0.f, 0.f, 0.f};
            int ev[4] = {0, 0, 0, 0}, jv[4] = {0, 0, 0, 0}, jn[4] = {0, 0, 0, 0};
            if (n_iters > 0) { fetch_idx(0, jv); fetch_vals(jv, bv, ev); }
            if (n_iters > 1) fetch_idx(1, jn);
            bool ok = true;
            for (int it = 0; it < n_iters && ok; ++it) {
                const int st = it % kStages;
                const uint32_t entry = S.sched[it];
                const bool use = use_bit(entry, w);
                float bn[4] = {0.f, 0.f, 0.f, 0.f};
                int en[4] = {0, 0, 0, 0}, jnn[4] = {0, 0, 0, 0};
                if (it + 1 < n_iters) fetch_vals(jn, bn, en);
                if (it + 2 < n_iters) fetch_idx(it + 2, jnn);
                uint32_t b0[4], b1[4], aw[4][7];
                int hot[4];
                bool fast = false;
                uint32_t live8 = 0xFFu;
                if (use) {
                    // general path needed: the tile holds keys that enter inside the query tile's rows (the diagonal tile)
                    const bool diag = (int)(entry & 0xFFFFF) == (w ? qt1 : qt0);
                    uint32_t bal[4];
                    bool mixed[4], dead[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        dead[t] = ev[t] <= i0;
                        mixed[t] = !dead[t] && ev[t] < i0 + 128;
                        bal[t] = __ballot_sync(0xffffffffu, mixed[t]);
                    }
                    if constexpr (kBlockSkip) {
                        live8 = 0u;
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const uint32_t alive = __ballot_sync(0xffffffffu, !dead[t]);     // keys 32 t .. 32 t + 31
                            live8 |= ((alive & 0xFFFFu) ? 1u : 0u) << (2 * t) | ((alive >> 16) ? 1u : 0u) << (2 * t + 1);
                        }
                    }
                    const int cnt = __popc(bal[0]) + __popc(bal[1]) + __popc(bal[2]) + __popc(bal[3]);
                    fast = !diag && cnt <= kMaskSlots;
                    if (lane < kMaskSlots) S.thr[w][lane] = 1 << 20;
                    __syncwarp();
                    int before = 0;
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int slot = before + __popc(bal[t] & ((1u << lane) - 1));
                        before += __popc(bal[t]);
                        hot[t] = (fast && mixed[t]) ? 3 + slot : -1;          // element that holds this key's -BIG
                        if (hot[t] >= 0) S.thr[w][slot] = ev[t] - i0;
                    }
                    __syncwarp();
                    // B rows (keys): bias / scale as three bf16 terms (24 significant bits, as many as the fp32 bias
                    // has), or -BIG for a key that is gone for the whole tile
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const float bs = bv[t] * P.inv_scale;
                        const __nv_bfloat16 hi = __float2bfloat16_rn(bs);
                        const float r1 = bs - __bfloat162float(hi);
                        const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
                        const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
                        b0[t] = dead[t] ? kNegBig : ((uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(mid) << 16));
                        b1[t] = (dead[t] ? 0u : (uint32_t)__bfloat16_as_ushort(lo)) | (hot[t] == 3 ? (kNegBig << 16) : 0u);
                    }
                    // A rows (queries): ones for the bias terms, then one step function per expiring key
                    int th[kMaskSlots];
#pragma unroll
                    for (int k = 0; k < kMaskSlots; ++k) th[k] = S.thr[w][k];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int r = lane + 32 * t;
                        aw[t][0] = kOne | (r >= th[0] ? (kOne << 16) : 0u);
#pragma unroll
                        for (int m = 2; m < 8; ++m)
                            aw[t][m - 1] = (r >= th[2 * m - 3] ? kOne : 0u) | (r >= th[2 * m - 2] ? (kOne << 16) : 0u);
                    }
                }
                const int slot = kSplit ? (it >> 1) & 1 : st;
                if constexpr (kSplit) {
                    // The group's operand blocks were last read by its last S product, and the slot by the group before it released P of the
                    // entry before that one, hence before that S product was issued. k_full takes one arrival per entry: not before its last phase is over.
                    if (it >= kStages) ok = mbar_wait_warp(&S.k_empty[st], ((it / kStages) - 1) & 1, abort_flag);
                } else {
                    // fast[st] / len[st] were last read by the softmax groups before they released P of tile it - kStages
                    // (hence before its P V); the operand blocks were last read by the S products of tile it - 1
                    if (it >= kStages) ok = mbar_wait_warp(&S.v_empty[st], ((it / kStages) - 1) & 1, abort_flag);
                    if (ok && it >= 1) ok = mbar_wait_warp(&S.k_empty[(it - 1) % kStages], ((it - 1) / kStages) & 1, abort_flag);
                }
                if (!ok) break;
                if (!kSplit && w == 0) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        S.len[st][lane + 32 * t] = ev[t];
                    }
                }
                if (use) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int c = lane + 32 * t;
                        if constexpr (kSplit) S.last[slot][w][c] = (uint8_t)min(max(ev[t] - i0, 0), 128);     // (columns beyond L: expiry 0)
                        uint32_t wd[8];
                        wd[0] = b0[t];
                        wd[1] = b1[t];
#pragma unroll
                        for (int m = 2; m < 8; ++m) wd[m] = (hot[t] >> 1) == m ? (kNegBig << ((hot[t] & 1) * 16)) : 0u;
                        uint8_t* brow = S.bext[w] + (c >> 3) * 256 + (c & 7) * 16;
                        *reinterpret_cast<uint4*>(brow) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                        *reinterpret_cast<uint4*>(brow + 128) = make_uint4(wd[4], wd[5], wd[6], wd[7]);
                        uint8_t* arow = S.aext[w] + (c >> 3) * 256 + (c & 7) * 16;
                        *reinterpret_cast<uint4*>(arow) = make_uint4(kOne | (kOne << 16), aw[t][0], aw[t][1], aw[t][2]);
                        *reinterpret_cast<uint4*>(arow + 128) = make_uint4(aw[t][3], aw[t][4], aw[t][5], aw[t][6]);
                    }
                    if (lane == 0) S.fast[slot][w] = (fast ? 1u : 0u) | (live8 << 8);
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    bv[t] = bn[t];
                    ev[t] = en[t];
                    jv[t] = jn[t];
                    jn[t] = jnn[t];
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.k_full[st]);
            }
        } else if (warp == kWarpIssuer) {
            // =========================================== MMA issuer ===========================================
            // The whole warp walks the schedule with warp-uniform values (descriptors, stage and tile indices stay in
            // the uniform datapath); one elected lane issues the tcgen05 instructions.
            constexpr uint32_t idesc_s = idesc_bf16(128, 128, 0, 0);     // Q (K-major) x K (K-major)
            constexpr uint32_t idesc_pv = idesc_bf16(128, kD, 0, 1);     // P (TMEM)    x V (MN-major)
            // operand descriptors are formed once; a stage, query tile or k-step only moves the 16-byte address field
            const uint64_t dQ0 = smem_desc_sw128(smem_u32(S.q[0]), 16, 1024), dK0 = smem_desc_sw128(smem_u32(S.k[0]), 16, 1024);
            const uint64_t dV0 = smem_desc_sw128(smem_u32(S.v[0]), kTileBytes / 2, 1024);
            const uint64_t dA0 = smem_desc_plain(smem_u32(S.aext[0]), 128, 256), dB0 = smem_desc_plain(smem_u32(S.bext[0]), 128, 256);
            // token-compacted mode: the second core matrix of every operand is the block of zeros, five blocks behind the ones
            const uint64_t dOnes = smem_desc_plain(smem_u32(S.aext[0]), 5 * 2048, 128);
            const uint64_t dRows = smem_desc_plain(smem_u32(S.aext[0]) + 2048, 4 * 2048, 128);      // stage 0, tile 0
            constexpr uint64_t kNextBlock = (uint64_t)(2048 >> 4) - ((uint64_t)(2048 >> 4) << 16);  // one block on, one less to the zeros
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
            const int n_iters_u = __shfl_sync(0xffffffffu, n_iters, 0);
            // MMA-block skipping (the finer granularity inside an active tile): the stager marks the 16-key blocks of the key
            // tile in which some key may be kept by the query tile's rows, and P V multiplies the marked blocks only (P is
            // exactly zero in the others, so the result does not change). The S product is always multiplied in full: leaving
            // out a dead 64-key half was built and measured (the issuer then needs the marks BEFORE the issue, a shared-memory
            // load on the critical path: 1.98 -> 2.55 ms at L = 16384), so it stayed out.
            uint32_t live[2] = {0xFFu, 0xFFu};          // marks of the key tile whose S product was issued last, per query tile
            bool o_started[2] = {false, false};         // the O accumulator has been written (first product: no accumulate)
            auto issue_s = [&](int w, int st, int slot) {
                const uint64_t dq = dQ0 + (uint64_t)(kSplit ? 0 : w * (kTileBytes >> 4)), dk = dK0 + (uint64_t)(st * (kTileBytes >> 4));
                const uint32_t d_tmem = tmem_u + w * 128;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kD / 16; ++kk) {
                        const uint32_t off = ((kk >> 2) * (kTileBytes / 2) + (kk & 3) * 32) >> 4;
                        mma_ss(d_tmem, dq + off, dk + off, idesc_s, kk > 0);
                    }
                    if constexpr (kCompact) mma_ss(d_tmem, dOnes, dRows + kNextBlock * (uint64_t)(slot * 2 + w), idesc_s, 1u);
                    else mma_ss(d_tmem, dA0 + (uint64_t)(w * (4096 >> 4)), dB0 + (uint64_t)(w * (4096 >> 4)), idesc_s, 1u);
                    tc_commit(&S.s_full[w]);
                }
                __syncwarp();
                // the block marks of this key tile, for its P V product later on: read AFTER the issue (a shared-memory load
                // costs hundreds of cycles while the MMAs stream their operands, and the S products are on the critical path)
                if constexpr (kBlockSkip) live[w] = *reinterpret_cast<volatile uint32_t*>(&S.fast[slot][w]) >> 8;     // (every lane reads the same word; first used at the P V issue)
            };
            const uint32_t both = (1u << 30) | (has1 ? (1u << 31) : 0u);     // token-compacted mode: every slice serves both tiles
            int n_p[2] = {0, 0};
            bool ok = mbar_wait_warp(&S.q_full, 0, abort_flag);
            if constexpr (kSplit) {
                // entry it: group and stage it & 1, the group's entry number it >> 1. Both groups start at once; the next S product of a group
                // is issued right behind its P V, so that the other group's softmax runs beside both
                auto start = [&](int it) {
                    const int w = it & 1;
                    ok = mbar_wait_warp(&S.k_full[w], (it >> 1) & 1, abort_flag);
                    if constexpr (kCompact) fence_proxy_async();
                    if (!ok) return;
                    tc_fence_after();
                    issue_s(w, w, (it >> 1) & 1);
                    if (elect_one()) tc_commit(&S.k_empty[w]);
                    __syncwarp();
                };
                if (ok && n_iters_u > 0) start(0);
                if (ok && n_iters_u > 1) start(1);
                for (int it = 0; it < n_iters_u && ok; ++it) {
                    const int w = it & 1, ph = (it >> 1) & 1;
                    const uint64_t dv = dV0 + (uint64_t)(w * (kTileBytes >> 4));
                    const uint32_t d_tmem = tmem_u + 256, a_tmem = tmem_u + w * 128;
                    ok = mbar_wait_warp(&S.v_full[w], ph, abort_flag);
                    if constexpr (kCompact) fence_proxy_async();
                    if (ok) ok = mbar_wait_warp(&S.p_half[w], ph, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_ts(d_tmem, a_tmem + kk * 8, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, kk > 0 || it > 0 ? 1u : 0u);
                    }
                    __syncwarp();
                    ok = mbar_wait_warp(&S.p_ready[w], ph, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 4; kk < 8; ++kk) mma_ts(d_tmem, a_tmem + kk * 8, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, 1u);
                        tc_commit(&S.o_done[w]);
                        tc_commit(&S.v_empty[w]);
                    }
                    __syncwarp();
                    if (it + 2 < n_iters_u) start(it + 2);
                }
            } else if (ok && n_iters_u > 0) {
                ok = mbar_wait_warp(&S.k_full[0], 0, abort_flag);
                if (ok) {
                    if constexpr (kCompact) fence_proxy_async();
                    tc_fence_after();
                    const uint32_t e0 = __shfl_sync(0xffffffffu, S.sched[0], 0);
#pragma unroll
                    for (int w = 0; w < 2; ++w)
                        if (ok && use_bit(e0, w)) {
                            // token-compacted mode: the second tile starts half a slice after the first. Started together, the
                            // two softmax groups stay in step: they contend for the issue slots and then wait for the MMAs
                            // together (L = 16384, w = 2048: 694 -> 680 us; 700 before the stager ran ahead)
                            if (kCompact && w == 1) ok = mbar_wait_warp(&S.p_half[0], 0, abort_flag);
                            if (ok) issue_s(w, 0, 0);
                        }
                    if (elect_one()) tc_commit(&S.k_empty[0]);
                    __syncwarp();
                }
            }
            for (int it = 0; !kSplit && it < n_iters_u && ok; ++it) {
                const int st = it % kStages, nst = (it + 1) % kStages;
                const uint32_t entry = kCompact ? both : __shfl_sync(0xffffffffu, S.sched[it], 0);
                const uint32_t next = it + 1 >= n_iters_u ? 0u : kCompact ? both : __shfl_sync(0xffffffffu, S.sched[it + 1], 0);
                ok = mbar_wait_warp(&S.v_full[st], (it / kStages) & 1, abort_flag);
                if constexpr (kCompact) fence_proxy_async();     // the gathered tiles were written through the generic proxy
                bool k_ready = false;
#pragma unroll
                for (int w = 0; w < 2; ++w) {          // unrolled: n_p[] stays in registers
                    if (ok && use_bit(entry, w)) {
                        // P V in two halves of 64 keys: the first runs while the softmax group still forms the second
                        const uint64_t dv = dV0 + (uint64_t)(st * (kTileBytes >> 4));
                        const uint32_t d_tmem = tmem_u + 256 + w * 128, a_tmem = tmem_u + w * 128;
                        // blocks to multiply; an accumulator that has never been written takes block 0 in any case (P is zero there)
                        const uint32_t l8 = !kBlockSkip ? 0xFFu : (!o_started[w] && live[w] == 0u) ? 1u : live[w];
                        const uint32_t acc0 = o_started[w] ? 1u : 0u;
                        ok = mbar_wait_warp(&S.p_half[w], n_p[w] & 1, abort_flag);
                        if (ok) {
                            tc_fence_after();
                            if (elect_one()) {
                                if (l8 == 0xFFu) {                                   // the common case: every block
#pragma unroll
                                    for (int kk = 0; kk < 4; ++kk)
                                        mma_ts(d_tmem, a_tmem + kk * 8, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, kk > 0 ? 1u : acc0);
                                } else {
                                    uint32_t acc = acc0;
#pragma unroll
                                    for (int kk = 0; kk < 4; ++kk) {
                                        if ((l8 >> kk) & 1u) {
                                            mma_ts(d_tmem, a_tmem + kk * 8, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, acc);
                                            acc = 1u;
                                        }
                                    }
                                }
                            }
                            __syncwarp();
                            ok = mbar_wait_warp(&S.p_ready[w], n_p[w] & 1, abort_flag);
                        }
                        if (ok) {
                            tc_fence_after();
                            if (elect_one()) {
                                if (l8 == 0xFFu) {
#pragma unroll
                                    for (int kk = 4; kk < 8; ++kk)
                                        mma_ts(d_tmem, a_tmem + kk * 8, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, 1u);
                                } else {
                                    uint32_t acc = (acc0 || (l8 & 0x0Fu)) ? 1u : 0u;
#pragma unroll
                                    for (int kk = 4; kk < 8; ++kk) {
                                        if ((l8 >> kk) & 1u) {
                                            mma_ts(d_tmem, a_tmem + kk * 8, dv + (uint64_t)((kk * 2048) >> 4), idesc_pv, acc);
                                            acc = 1u;
                                        }
                                    }
                                }
                                tc_commit(&S.o_done[w]);
                            }
                            __syncwarp();
                            o_started[w] = o_started[w] || l8 != 0u;
                            ++n_p[w];
                        }
                    }
                    if (ok && use_bit(next, w)) {
                        if (!k_ready) {
                            ok = mbar_wait_warp(&S.k_full[nst], ((it + 1) / kStages) & 1, abort_flag);
                            if constexpr (kCompact) fence_proxy_async();
                            if (ok) tc_fence_after();
                            k_ready = true;
                        }
                        if (ok) issue_s(w, nst, nst);
                    }
                }
                if (ok) {
                    if (elect_one()) {
                        tc_commit(&S.v_empty[st]);
                        if (it + 1 < n_iters_u) tc_commit(&S.k_empty[nst]);
                    }
                    __syncwarp();
                }
            }
        }
    }
    // teardown: every role falls through to here, also after a timed-out wait
    tc_fence_before();
    __syncthreads();
    if (warp == kWarpIssuer) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    if (tid == 0 && S.abort_flag) atomicExch(P.status, (int32_t)DMA_ERR_DEVICE_TIMEOUT);
}

}  // namespace

EncodeTiledFn get_encode_tiled() {
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

int make_tmap_bf16(CUtensorMap* m, const void* base, int B, int L, int H, int d, const int64_t strides[3], int rows) {
    EncodeTiledFn enc = get_encode_tiled();
    if (!enc) return DMA_ERR_CUDA;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)L, (cuuint64_t)H, (cuuint64_t)B};
    cuuint64_t str[3] = {(cuuint64_t)strides[1] * 2, (cuuint64_t)strides[2] * 2, (cuuint64_t)strides[0] * 2};   // bytes, dims 1..3
    cuuint32_t box[4] = {64, (cuuint32_t)rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, str, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? DMA_OK : DMA_ERR_CUDA;
}

// Token-compacted mode, per (batch, head, pair of query tiles): the list of keys j that some row i of the
// pair's 256 rows keeps, i.e. j <= i < expiry[j] for some i in [i0, i0 + 255]  <=>  j <= i0 + 255 and expiry[j] > max(i0, j).
// At most w + 256 keys qualify. The list is in two parts, each ascending: first the keys that ALL 256 rows keep
// (j <= i0 and expiry[j] >= i0 + 256), then the keys that enter or expire inside the pair's rows. The split leaves the keys
// that need the per-element test (a few hundred per pair) in the last slices instead of a few in every slice. The order inside
// a part decides how O rounds, so it is the same however the list was made: for any length and group.
// A CTA makes the lists of `group` consecutive pairs of one head. Every list on its own would read all keys before its rows, in
// two passes (count, write), which at 65536 keys was 781 us, an eighth of the prefill. With group > 1 the CTA first collects the
// keys that some row of the group keeps (at most the list's capacity and the group's rows: shared memory), and its lists are
// made from those: the head is read once per 256 group rows. group = 1: the lists are made straight from the head.
// Every warp owns a contiguous part of what it reads, 128 keys at a time (four coalesced loads per lane in flight), and writes
// from the sum of the earlier parts' counts. Padded with -1 to the next multiple of 128.
constexpr int kListGroup = 8;               // most pairs per CTA
constexpr int kWideListKeys = 8192;
constexpr int kListSmem = 100 * 1024;       // the most dynamic shared memory a CTA takes: two fit on an SM

template <int kListWarps>
__global__ void __launch_bounds__(32 * kListWarps) compact_lists_kernel(const int32_t* __restrict__ expiry, int* __restrict__ cidx,
                                                                     int* __restrict__ ccnt, int L, int npairs, int cap, int causal,
                                                                     int q_off, int32_t* __restrict__ status, int group, int ccap) {
    extern __shared__ int2 cand[];                       // group > 1: (key, expiry) of the keys some row of the group keeps
    __shared__ int wcount[2][kListWarps];
    const int ngroups = (npairs + group - 1) / group;
    const int bh = blockIdx.x / ngroups, pair0 = blockIdx.x % ngroups * group;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t below = (1u << lane) - 1u;
    pdl_enter(expiry, cidx, ccnt, status);
    if (blockIdx.x == 0 && tid < kWsHeaderBytes / 4) status[tid] = 0;       // the stage's first kernel: it clears the workspace header
    if (!causal && pair0 != 0) return;                   // non-causal: the head's one list is that of its first pair
    const int32_t* e = expiry + (size_t)bh * L;
    const int pairs = causal ? min(group, npairs - pair0) : 1;
    const int lo = q_off + pair0 * 256, jend = causal ? min(L, lo + pairs * 256) : L;
    // four keys of the head per lane, from base on: (key, expiry), expiry 0 (never kept) beyond `end`
    auto load4 = [&](int base, int end, int (&j)[4], int (&ej)[4]) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            j[u] = base + 32 * u + lane;
            ej[u] = j[u] < end ? e[j[u]] : 0;
        }
    };
    int ncand = jend;
    bool over = false;
    if (group > 1) {
        const int seg = ((jend + kListWarps - 1) / kListWarps + 127) / 128 * 128, j0 = warp * seg, j1 = min(jend, j0 + seg);
        int c = 0;
#pragma unroll 4
        for (int base = j0; base < j1; base += 128) {
            int j[4], ej[4];
            load4(base, j1, j, ej);
#pragma unroll
            for (int u = 0; u < 4; ++u) c += ej[u] > max(lo, causal ? j[u] : 0);
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) wcount[0][warp] = c;
        __syncthreads();
        int at = 0, all = 0;
#pragma unroll
        for (int q = 0; q < kListWarps; ++q) {
            at += q < warp ? wcount[0][q] : 0;
            all += wcount[0][q];
        }
#pragma unroll 4
        for (int base = j0; base < j1; base += 128) {
            int j[4], ej[4];
            load4(base, j1, j, ej);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = ej[u] > max(lo, causal ? j[u] : 0);
                const uint32_t bal = __ballot_sync(0xffffffffu, in);
                const int p = at + __popc(bal & below);
                if (in && p < ccap) cand[p] = make_int2(j[u], ej[u]);
                at += __popc(bal);
            }
        }
        over = all > ccap;                               // then the group's first row alone keeps more than a list holds
        ncand = min(all, ccap);
        __syncthreads();
    }
    // the lists: kListWarps / group warps per pair
    const int per = kListWarps / group, part = warp % per, pair = pair0 + warp / per;
    const bool exists = warp / per < pairs;
    const int i0 = q_off + pair * 256, list = bh * npairs + pair;
    const int end = group > 1 ? ncand : causal ? min(L, i0 + 256) : L;
    const int seg = ((end + per - 1) / per + 127) / 128 * 128, k0 = part * seg, k1 = exists ? min(end, k0 + seg) : 0;
    auto fetch = [&](int base, int (&j)[4], int (&ej)[4]) {
        if (group > 1) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = base + 32 * u + lane;
                const int2 v = k < k1 ? cand[k] : make_int2(0, 0);
                j[u] = v.x;
                ej[u] = v.y;
            }
        } else {
            load4(base, k1, j, ej);
        }
    };
    // 0: not in the list, 1: kept by every row of the pair, 2: kept by some
    auto kind = [&](int j, int ej) {
        const int first = causal ? j : 0;
        if (ej <= max(i0, first) || first > i0 + 255) return 0;
        return (first <= i0 && ej >= i0 + 256) ? 1 : 2;
    };
    int c1 = 0, c2 = 0;
#pragma unroll 4
    for (int base = k0; base < k1; base += 128) {
        int j[4], ej[4];
        fetch(base, j, ej);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = kind(j[u], ej[u]);
            c1 += k == 1;
            c2 += k == 2;
        }
    }
    c1 = __reduce_add_sync(0xffffffffu, c1);
    c2 = __reduce_add_sync(0xffffffffu, c2);
    if (group > 1) __syncthreads();                      // wcount was read above
    if (lane == 0) { wcount[0][warp] = c1; wcount[1][warp] = c2; }
    __syncthreads();
    if (!exists) return;
    int p1 = 0, p2 = 0, n1 = 0, n2 = 0;
    for (int q = 0; q < per; ++q) {
        const int a = wcount[0][warp - part + q], b = wcount[1][warp - part + q];
        p1 += q < part ? a : 0;
        p2 += q < part ? b : 0;
        n1 += a;
        n2 += b;
    }
    p2 += n1;                                            // the second part starts behind the first
    int* out = cidx + (size_t)list * cap;
#pragma unroll 4
    for (int base = k0; base < k1; base += 128) {
        int j[4], ej[4];
        fetch(base, j, ej);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = kind(j[u], ej[u]);
            const uint32_t b1 = __ballot_sync(0xffffffffu, k == 1), b2 = __ballot_sync(0xffffffffu, k == 2);
            const int at = k == 1 ? p1 + __popc(b1 & below) : p2 + __popc(b2 & below);
            if (k != 0 && at < cap) out[at] = j[u];
            p1 += __popc(b1);
            p2 += __popc(b2);
        }
    }
    // more kept keys than the list holds (a mask that keeps more than w keys in some row): the count says so and the forward
    // kernel reports it
    const int n = min(n1 + n2, cap), fill = over ? cap : (n + 127) / 128 * 128;
    for (int t = n + part * 32 + lane; t < fill && t < cap; t += per * 32) out[t] = -1;
    if (part == 0 && lane == 0) ccnt[list] = over ? cap + 1 : n1 + n2;
}

static int compact_cap(const Prob& P) { return ((P.w + 256 + 127) / 128) * 128; }
static size_t compact_lists(const Prob& P) { return (size_t)P.B * P.Hq * ((P.Tr + 1) / 2); }

size_t tc_fwd_ws_bytes(const Prob& P) {
    if (!(P.flags & DMA_FLAG_COMPACT_KV)) return kWsHeaderBytes;
    const size_t cnt_bytes = ((compact_lists(P) * sizeof(int) + 255) / 256) * 256;
    return kWsHeaderBytes + cnt_bytes + compact_lists(P) * compact_cap(P) * sizeof(int);
}

// Query tiles per CTA: two, or one whose key tiles are dealt out to the two softmax groups where that shortens the call. Both grids
// are estimated in steps of a CTA (a key tile and two score tiles): its steps and a fixed cost, the CTAs started heaviest first on the SMs. Tile mode: the SMs' share of the work, four
// in five key tiles before the rows taken to be active, and part of the longest CTA behind it, more of it where the caller asks for tiles because the kept keys cluster (packed documents: walks of
// all lengths). Token-compacted, where the CTAs are of about the same length: half way between the SMs' share and whole waves. (A one-tile CTA's slices: 0.55 of the other's with all SMs
// gathering.) Fitted to 710 shapes of 1 to 256 heads and 128 to 32768 keys, each timed with both, and held against 360 others: 0.1 % (token-compacted) and 0.4 % (tiles) from the better one in the
// mean, where the rule of slower kernels before, without the longest CTA and the half-empty last pair, was 0.8 and 0.6 %, on documents 3 %; worst 256 heads of 1054 keys with 64 channels, 10 %,
// and 64 of 306, 9 %. Forward, us, two tiles / one: 16 heads of 5231 keys 138 / 147, 8 of 10069 206 / 237, 128 of 170 14.8 / 17.4, 8 of 5250 (w = 1312) 49.7 / 59.0, but
// 16 of 3880 (64 channels) 94 / 78, documents in 8 heads of 16245 keys 199 / 147, in 32 of 2144 41 / 36, the last 693 of 23017 rows, 32 heads 178 / 149. The results are the same bits.
// DMA_FLAG_BLOCK_SKIP is for two tiles: its marks are read where one group walks every entry.
static int fwd_tiles(const Prob& P) {
    if (P.flags & DMA_FLAG_BLOCK_SKIP) return 2;
    constexpr double kSms = 148.0;
    const int Trq = (P.Lq + 127) / 128, npairs = (Trq + 1) / 2, odd = Trq & 1;
    const double heads = (double)P.B * P.Hq;
    if (P.flags & DMA_FLAG_COMPACT_KV) {
        // a pair's list: w + 256 keys, or the keys before its last row where they are fewer (`rising` pairs; non-causal: the head's w)
        const double full = std::min((int64_t)P.w + (P.causal ? 256 : 0), (int64_t)P.L) / 128.0, before = P.q_off / 128.0;
        const double rising = P.causal && P.w > P.q_off ? std::min(npairs, (P.w - P.q_off) / 256) : 0;
        const double lists = rising * before + rising * (rising + 1) + (npairs - rising) * full;
        const double longest = rising < npairs ? full : std::min(full, before + 2.0 * npairs);
        auto cost = [&](double ctas, double work, double cta) { return 0.5 * std::max(cta, work / kSms) + 0.5 * std::ceil(ctas / kSms) * cta; };
        const double one = cost(heads * Trq, heads * (0.55 * (2 * lists - odd * full) + 3.5 * Trq), 0.55 * longest + 3.5);
        return one < cost(heads * npairs, heads * (lists + 4.0 * npairs), longest + 4.0) ? 1 : 2;
    }
    const bool clustered = (P.flags & DMA_FLAG_TILE_PATH) && !(P.flags & DMA_FLAG_IGNORE_BITMAP);
    const double tail = clustered ? 0.4 : 0.2;
    auto cost = [&](double work, double cta) { return std::max(cta, work / kSms + tail * cta); };       // walks grow with the row: the last tile's is the longest
    const double fixed = clustered ? 1.0 : 1.5;
    const double one = (clustered ? 1.1 : 1.15) * cost(heads * (0.2 * Trq * (Trq + 1.0) + Trq), Trq / 2.0 + 1.0);
    return one < cost(heads * (0.8 * (npairs * (npairs + 1.0) - odd) + fixed * npairs), Trq + fixed) ? 1 : 2;
}

int launch_tc_fwd(const Prob& P, const void* Q, const void* K, const void* V, const float* bias,
                  const int32_t* expiry, const uint32_t* bitmap, void* O, float* lse, void* ws, cudaStream_t st) {
    const bool compact = (P.flags & DMA_FLAG_COMPACT_KV) != 0;
    if (P.Tc > kMaxSched) return DMA_ERR_UNSUPPORTED;
    const bool block_skip = (P.flags & DMA_FLAG_BLOCK_SKIP) != 0;
    const bool split = fwd_tiles(P) == 1;
    auto pick = [&](auto d_tag) {
        constexpr int kD = decltype(d_tag)::value;
        if (split) return compact ? fwd_kernel<true, false, kD, true> : fwd_kernel<false, false, kD, true>;
        return compact ? (block_skip ? fwd_kernel<true, true, kD, false> : fwd_kernel<true, false, kD, false>)
                       : (block_skip ? fwd_kernel<false, true, kD, false> : fwd_kernel<false, false, kD, false>);
    };
    auto kern = P.d == 128 ? pick(std::integral_constant<int, 128>{}) : pick(std::integral_constant<int, 64>{});
    {
        cudaFuncAttributes fa;       // (before anything is enqueued)
        if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || fa.numRegs != kLaunchRegs) return DMA_ERR_CUDA;
    }
    CUtensorMap tmQ, tmK, tmV;
    int rc;
    const int Trq = (P.Lq + 127) / 128, npairs = (Trq + 1) / 2;
    if ((P.Lq != P.L || P.q_off != 0) && !compact) return DMA_ERR_UNSUPPORTED;
    if ((rc = make_tmap_bf16(&tmQ, Q, P.B, P.Lq, P.Hq, P.d, P.qs, 128))) return rc;
    FwdParams fp;
    fp.cidx = nullptr; fp.ccnt = nullptr; fp.ccap = 0; fp.Hkv = P.Hkv; fp.causal = P.causal;
    fp.Lq = P.Lq; fp.q_off = P.q_off; fp.Trq = Trq;
    if (!P.causal && !compact) return DMA_ERR_UNSUPPORTED;
    if (compact) {
        if (compact_cap(P) / 128 > kMaxSched) return DMA_ERR_UNSUPPORTED;
        const size_t nl = (size_t)P.B * P.Hq * npairs;
        int* ccnt = reinterpret_cast<int*>((char*)ws + kWsHeaderBytes);
        int* cidx = reinterpret_cast<int*>((char*)ws + kWsHeaderBytes + ((nl * sizeof(int) + 255) / 256) * 256);
        // pairs per CTA: as many as leave every SM a CTA and whose candidates fit twice into an SM's shared memory. List kernel, us,
        // one pair / this rule: 32 heads of 65536 keys 539 / 141, of 16384 keys 49 / 25 (a scalar two-pass scan per pair: 781, 69)
        const int cap = compact_cap(P);
        int group = 1;
        while (group < kListGroup && P.causal && npairs >= 2 * group && (int64_t)P.B * P.Hq * ((npairs + 2 * group - 1) / (2 * group)) >= 148 &&
               (size_t)(cap + 2 * group * 256) * sizeof(int2) <= (size_t)kListSmem) group *= 2;
        const size_t smem = group > 1 ? (size_t)(cap + group * 256) * sizeof(int2) : 0;
        // one pair per CTA: a long head takes twice the warps (us, forward, 8 / 16 / 32 warps: 500 rows of 20000 keys, 8 heads 57.0 / 53.5 / 56.2,
        // 2048 of 16384, 32 heads 119.9 / 118.1 / 127.1, but 16 heads of 4096 73.8 / 74.3 / 79.0)
        const bool wide = group == 1 && P.L >= kWideListKeys;
        auto lists = wide ? compact_lists_kernel<2 * kListGroup> : compact_lists_kernel<kListGroup>;
        const int threads = wide ? 64 * kListGroup : 32 * kListGroup;
        // (the limit is state of the function, which other threads' calls share: always the same value)
        if (smem && cudaFuncSetAttribute(lists, cudaFuncAttributeMaxDynamicSharedMemorySize, kListSmem) != cudaSuccess) return DMA_ERR_CUDA;
        if ((rc = launch_overlapped(lists, dim3((unsigned)(P.B * P.Hq * ((npairs + group - 1) / group))), dim3(threads), smem, st, 1,
                                    expiry, cidx, ccnt, P.L, npairs, cap, P.causal, P.q_off, (int32_t*)ws, group, cap + group * 256)))
            return rc;                 // the forward kernel must not run on lists that nobody wrote
        fp.cidx = cidx; fp.ccnt = ccnt; fp.ccap = compact_cap(P);
    }
    fp.Kg = (const __nv_bfloat16*)K; fp.Vg = (const __nv_bfloat16*)V;
    if ((rc = make_tmap_bf16(&tmK, K, P.B, P.L, P.Hkv, P.d, P.ks, 128))) return rc;
    if ((rc = make_tmap_bf16(&tmV, V, P.B, P.L, P.Hkv, P.d, P.vs, 128))) return rc;
    fp.bias = bias; fp.expiry = expiry; fp.bitmap = bitmap; fp.O = (__nv_bfloat16*)O; fp.lse = lse;
    fp.status = (int32_t*)ws;
    fp.B = P.B; fp.Hq = P.Hq; fp.G = P.G; fp.L = P.L; fp.Tr = P.Tr; fp.Tc = P.Tc; fp.Wd = P.Wd;
    fp.ignore_bitmap = (P.flags & DMA_FLAG_IGNORE_BITMAP) ? 1 : 0;
    fp.scale_log2 = P.scale * 1.4426950408889634f;
    fp.inv_scale = 1.0f / P.scale;
    fp.rescale_gap = kRescaleThreshold / fp.scale_log2;
    fp.os_b = P.os[0]; fp.os_l = P.os[1]; fp.os_h = P.os[2];
    fp.ks_b = P.ks[0]; fp.ks_l = P.ks[1]; fp.ks_h = P.ks[2]; fp.vs_b = P.vs[0]; fp.vs_l = P.vs[1]; fp.vs_h = P.vs[2];
    const size_t smem = sizeof(SharedStorage) + 1024;
    dim3 grid(P.B * P.Hq, split ? Trq : npairs);
    timing_mark(0, false, st);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return DMA_ERR_CUDA;
    rc = launch_overlapped(kern, grid, dim3(kThreads), smem, st, 1, tmQ, tmK, tmV, fp);
    timing_mark(0, true, st);
    return rc;
}

}  // namespace dma
