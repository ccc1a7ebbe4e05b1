// Tensor-core backward (Sec. 4.3, Alg. 2) for bf16, d = 128 or 64, on sm_100a.
//
// One CTA owns one 128-key tile of one KV head and, as in Alg. 2's outer loop, keeps dK, dV (fp32, tensor memory)
// and dM (registers) for it while walking the query heads of the group and their active query tiles in steps of
// 64 query rows. Everything is computed transposed, keys on the 128 TMEM lanes, so that dM is a per-thread row sum
// and P^T, dS^T feed the dV / dK GEMMs straight from tensor memory:
//   S^T  = K Q^T - lse_i / scale     dP^T = V dO^T - D_i      (smem x smem -> TMEM, 64 columns each; the per-row terms
//                                                              come from a ninth k-step: ones (x) three bf16 terms)
//   P^T  = exp2(c S^T + log2e bias_j) where j <= i < expiry[j], else 0;   dS^T = P^T o dP^T
//   dV  += P^T dO           dK  += dS^T Q                      (TMEM x smem  -> TMEM, 128 columns each)
//   dQ^T = K^T dS^T                                            (smem x smem  -> TMEM, 64 columns), staged in shared memory
//                                                              and added to the fp32 dQ accumulator by bulk reduce-adds
// The dQ accumulator is blocked: 16 rows x 32 channels of one head are 2 KB of consecutive floats, so that a staged
// quarter step leaves as ONE contiguous bulk reduce-add (as a tile of a [B, L, Hq, d] tensor map the same 2 KB were 16
// strided 128-byte rows, and issuing that request took the drain warp ~350 cycles: the drain was as long as the step).
// Shared-memory bandwidth is the scarce resource (operand reads of the smem x smem MMAs alone take ~1400 of a step's
// ~2250 cycles), so the compute warps read nothing from shared memory per element.
// Warp roles (16 warps): warps 0-7 compute (thread = key; warps w and w+4 share the 32 TMEM lanes of quadrant w%4 and
// split the 64 query columns of a step), warps 8-11 dQ drain (thread = channel), warp 12 TMA producer + schedule,
// warps 13 and 14 MMA issuers (S^T, dP^T | dV, dK, dQ^T; whole warps with warp-uniform values, one elected lane
// issues), warp 15 stages the ninth k-step operand of each step's query rows.
// TMEM columns: dK [0,128) dV [128,256) S^T [256,320) dP^T [320,384) P^T [384,416) dS^T [416,448) dQ^T [448,512).
// kD = 64 (its own instantiations): K, V, Q and dO tiles are one swizzled half tile each, S^T and dP^T have four k-steps
// and the ninth, dK and dV take 64 columns. What that frees is spent on the two chains that bound a step at d = 128:
//   - P^T and dS^T are double-buffered (tensor-memory columns [64,128) and the unused half of the V buffer for the
//     shared-memory copy of dS^T), so the compute warps store step n+1 while the MMAs of step n still read step n's;
//   - dQ^T = K^T dS^T keeps M = 128 with the K tile loaded a second time into the unused half of its buffer: lanes
//     64-127 repeat lanes 0-63, so all four drain warps work, two per 32 channels, each on half of the step's rows.
#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace dma {
namespace {

using namespace ptx;

constexpr int kStages = 3;
constexpr int kMaxSteps = 8192;              // 64-row steps of one CTA: G * ceil(L / 128) * 2 (L = 131072 with four query heads per KV head)
constexpr int kThreads = 512;
constexpr uint32_t kKVBytes = 128 * 128 * 2;   // K or V tile: two 16 KB halves (channels 0-63 | 64-127)
constexpr uint32_t kQBytes = 64 * 128 * 2;     // Q or dO step tile (64 rows): two 8 KB halves
constexpr int cDK = 0, cDV = 128, cS = 256, cDP = 320, cP = 384, cDS = 416, cDQ = 448;
constexpr int cP1 = 64, cDS1 = 96;             // second P^T / dS^T buffer (d = 64 only: beside the 64 columns of dK)

struct SharedStorage {
    alignas(1024) uint8_t k[kKVBytes];
    alignas(1024) uint8_t v[kKVBytes];
    alignas(1024) uint8_t q[kStages][kQBytes];
    alignas(1024) uint8_t g[kStages][kQBytes];       // dO
    alignas(1024) uint8_t ds[128 * 128];             // dS^T as bf16: [128 keys][64 queries], 128-byte swizzled rows
    alignas(1024) float dq_stage[4][2][16][32];      // dQ per drain warp (32 channels), two buffers of 16 query rows: sources of the TMA reduce-adds
    // Ninth k-step of S^T = K Q^T and dP^T = V dO^T (unswizzled K-major core matrices of 8 rows x 16 bytes): it adds
    // -lse_i / scale to S^T and -D_i to dP^T, each as three bf16 terms, so that the compute warps read finished values
    // from tensor memory and need no per-column vector. `ones` = [zero | rows (1,1,1,0..) | zero] blocks of 128 rows:
    // A operand with the ones in elements 0-2 (block 1, then block 2) or in elements 8-10 (block 0, then block 1).
    // `qext[stage]` = B operand, 64 query rows: elements 0-2 = -lse / scale, elements 8-10 = -D.
    alignas(128) uint8_t ones[3][2048];
    alignas(128) uint8_t qext[kStages][2048];
    uint16_t sched[kMaxSteps];                       // head-in-group << 11 | query tile << 1 | half
    uint64_t kv_full, qd_full[kStages], qd_empty[kStages];
    uint64_t sdp_full, sdp_free, pds_ready[2], pds_free[2], dq_full, dq_free;
    uint32_t tmem_base;
    int n_steps;
    int abort_flag;
    int part, block;                                 // token-compacted mode: the walk's part, and where its dK and dV go (WalkBlocks; -1: to the accumulators)
    int cut;                                         // what the first part notes for the last kernel: WalkBlocks::where but for the row (0: nothing)
};

// Token-compacted mode: the sums of walks that are cut into parts. What a key gets must not depend on which part ends first where it did
// not depend on order without cuts: dM, and dK and dV with one or two query heads per KV head (a sum of two addends onto a zero has one
// value). The first `direct` parts of a walk add their dK and dV to the accumulators, two with one query head, one with two, all of them with
// more, whose sums vary in any case. The others have a block each, `cap` of them per (batch, query head), and every part but the
// first has a place for its dM; the last kernel adds these in the order of the parts.
struct WalkBlocks {
    float* kv;                  // [B, Hq, cap] x dK [128 keys][d] | dV [128][d], unscaled
    float* m;                   // [B, Hq, key tile, part - 1] x two halves of the query columns [2][128]
    int* where;                 // [B, Hq, L], zeros before: row of the key in its tile | parts - 1 << 7 | first block << 10 | key tile << 19. NULL: no walk is cut
    int cap, direct;
};

struct BwdParams {
    const float* lse;
    const float* Dv;
    const float* bias;
    const int32_t* expiry;
    const uint32_t* bitmap;
    int sched_group;            // (batch, head) entries per scheduling group, a divisor of gridDim.x
    float* dQacc;               // fp32, zeroed, blocked: [B, Hq, Lblk, d / 32] blocks of 16 rows x 32 channels = 2 KB, each laid out
                                // as the drain warps stage it: channel c owns 64 bytes (its 16 rows), and the 16-byte chunk of
                                // rows 4q .. 4q + 3 sits at chunk q ^ ((c >> 1) & 3) (a thread = a channel then stores four
                                // 16-byte chunks without bank conflicts, instead of 16 scalars)
    int Lblk;                   // 16-row blocks per head: 8 * Tr (rows padded to whole 128-row tiles)
    __nv_bfloat16* dK;
    __nv_bfloat16* dV;
    float* dM;
    int32_t* status;
    int B, Hq, Hkv, G, L, Tr, Tc, Wd, ignore_bitmap;
    float scale, scale_log2, inv_scale;
    // token-compacted mode: per (batch, query head) a permutation of the keys (padded with L to a multiple of 128) that
    // groups keys of similar lifetime; a CTA owns 128 consecutive entries of one query head's permutation
    const int* perm;
    const int2* items;         // what each CTA does: [B, Hq, gridDim.y]
    WalkBlocks blocks;
    int causal;                // 0: key j is visible to every row (token-compacted mode only): its first row is 0 instead of j
    const __nv_bfloat16* Kg;    // K, V base pointers for the row gathers (ks_*, vs_* strides)
    const __nv_bfloat16* Vg;
    float* dKacc;               // fp32 [B, L, Hkv, 128] accumulators (several query heads add into one KV head's rows)
    float* dVacc;
    int64_t acc_slot;           // 0: the group's heads add into one accumulator with atomics; else: elements between the
                                // slots [slot][B, L, Hkv, d] (one per query head of the group, or per split of the group in tile
                                // mode), written with plain stores and summed in slot order afterwards
    int nsplit;                 // tile mode: CTAs that share a KV head's query heads, G / nsplit each (1: dK, dV are written directly)
    int64_t ks_b, ks_l, ks_h, vs_b, vs_l, vs_h;
};


// Token-compacted mode: one CTA's work, a key tile of the head's permutation and a part of its walk over the query tiles q0 .. q1:
//   x = key tile | part << 10 | parts << 13 | block << 17 (-1: nothing)     y = q0 | q1 << 16
// block: of the parts that have none the first that has
constexpr int kMostParts = 8;
constexpr int kWalkBlocks = 296;               // blocks of a call in all (39 MB at d = 128): parts are about an SM's share of the work, 148 / 0.8 of them in all
// 64-row steps of a walk (the sequence's last tile may have one only)
__device__ __forceinline__ int walk_steps(int q0, int q1, int L) { return min(2 * (q1 - q0 + 1) - (q1 * 128 + 64 >= L ? 1 : 0), kMaxSteps); }

// x as three bf16 terms (hi, mid, lo: 24 significant bits) in elements 0-2 of a 16-byte core-matrix row
__device__ __forceinline__ uint4 split3(float x) {
    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
    return make_uint4((uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(mid) << 16), (uint32_t)__bfloat16_as_ushort(lo), 0u, 0u);
}

// kCompact: token-compacted mode. The CTA's 128 keys are 128 consecutive entries of one QUERY head's lifetime-sorted
// key permutation instead of 128 consecutive keys of a KV head: keys that live equally long are kept by about the
// same query rows, so the walk over query tiles [first key's tile, last expiry's tile] wastes little. K and V rows
// are gathered once with 16-byte asynchronous copies; dK and dV are added to fp32 accumulators (the query heads of a
// group meet there), dM, the sum of two halves of the query columns, to zeros.
// kLong: tile mode without a split of the query heads and without the overlapped launch, for problems that last long (bwd_long).
template <bool kCompact, int kD, bool kLong = false>
__global__ void __launch_bounds__(kThreads, 1)
bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
           const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG, const BwdParams P) {
    static_assert(kD == 128 || kD == 64, "head dimensions of the tensor-core kernels");
    constexpr int kHalves = kD / 64;                 // 64-channel (128-byte) swizzled half tiles per operand tile
    constexpr bool kDouble = kD == 64;               // P^T / dS^T in two buffers used in turn (see the file header)
    extern __shared__ uint8_t smem_raw[];
    SharedStorage& S = *reinterpret_cast<SharedStorage*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    static_assert(!(kCompact && kLong), "kLong is a tile mode");
    if constexpr (!kLong) pdl_enter();
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);      // warp-uniform to the compiler: role branches stay uniform
    // tile mode: blockIdx.x = (batch, KV head, split of its query heads); token-compacted mode: (batch, query head), whose group index is fixed
    // CTAs start in the order of lin: heads of one scheduling group (P.sched_group of them) innermost, then key tiles (key
    // tile 0 has the most query tiles: heaviest first), then the groups
    const int lin = blockIdx.y * gridDim.x + blockIdx.x, per_group = P.sched_group * (int)gridDim.y;
    const int bx = (lin / per_group) * P.sched_group + (lin % per_group) % P.sched_group;
    const int nsplit = kCompact || kLong ? 1 : P.nsplit, sp = kCompact || kLong ? 0 : bx % nsplit;
    const int b = kCompact ? bx / P.Hq : bx / (nsplit * P.Hkv);
    const int hq_c = bx % P.Hq;                        // token-compacted mode only
    const int hk = kCompact ? hq_c / P.G : bx / nsplit % P.Hkv;
    const int at = (lin % per_group) / P.sched_group;
    const int2 item = kCompact ? P.items[(size_t)bx * gridDim.y + at] : make_int2(at, 0);
    if (kCompact && item.x < 0) return;                // no more items for this head
    const int kt = kCompact ? item.x & 0x3FF : at;
    const int j0 = kt * 128;
    const int* my_perm = kCompact ? P.perm + ((size_t)bx * P.Tc + kt) * 128 : nullptr;
    volatile int* abort_flag = &S.abort_flag;

    if (tid == 0) {
        mbar_init(&S.kv_full, kCompact ? 8 : 1);        // one arrival per gathering warp | TMA bytes
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&S.qd_full[s], 2);      // TMA bytes + the staged vectors
            mbar_init(&S.qd_empty[s], 1);
        }
        mbar_init(&S.sdp_full, 1);
        mbar_init(&S.sdp_free, 8);        // one arrival per compute warp (256 serialised arrivals would cost hundreds of cycles)
        for (int u = 0; u < 2; ++u) {
            mbar_init(&S.pds_ready[u], 8);
            mbar_init(&S.pds_free[u], 1);
        }
        mbar_init(&S.dq_full, 1);
        mbar_init(&S.dq_free, 4);         // one arrival per drain warp
        S.abort_flag = 0;
        S.n_steps = 0;
        if constexpr (kCompact) {
            const int part = (item.x >> 10) & 7, later = ((item.x >> 13) & 0xF) - 1, block = item.x >> 17;
            S.part = part;
            S.block = part >= P.blocks.direct ? block : -1;
            S.cut = part == 0 && later > 0 ? later << 7 | block << 10 | kt << 19 : 0;
        }
        fence_barrier_init();
        if constexpr (!kCompact) {                     // K and V need no schedule: they are under way while it is built
            mbar_arrive_expect_tx(&S.kv_full, (kD == 128 ? 4 : 3) * (kKVBytes / 2));
            for (int hf = 0; hf < 2; ++hf) {           // d = 64: both halves of the K buffer hold the same 64 channels
                tma_load_4d(&S.k[hf * (kKVBytes / 2)], &tmK, &S.kv_full, kD == 128 ? hf * 64 : 0, j0, hk, b);
                if (hf < kHalves) tma_load_4d(&S.v[hf * (kKVBytes / 2)], &tmV, &S.kv_full, hf * 64, j0, hk, b);
            }
        }
    }
    if (kCompact && warp < 8) {
        // The compute warps gather the CTA's 128 K and V rows into the swizzled tile layout, 16 rows each (8 lanes per 128-byte half row, 4
        // rows per instruction; padding entries are zero-filled), while the schedule is built. (One warp after the schedule: the first
        // product was issued 10500 clk after the CTA's start, now 4200 to 4900 in the median.)
        const int rsub = lane >> 3, c = lane & 7;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = warp * 16 + 4 * q + rsub, j = my_perm[r];
            const int64_t jr = min(j, P.L - 1);
            const int64_t krow = b * P.ks_b + jr * P.ks_l + hk * P.ks_h + c * 8, vrow = b * P.vs_b + jr * P.vs_l + hk * P.vs_h + c * 8;
            const uint32_t off = r * 128 + ((c ^ (r & 7)) << 4);
            const int nb = j < P.L ? 16 : 0;
            cp_async16(S.k + off, P.Kg + krow, nb);
            cp_async16(S.k + off + kKVBytes / 2, P.Kg + krow + (kD == 128 ? 64 : 0), nb);     // d = 64: the same 64 channels once more
            cp_async16(S.v + off, P.Vg + vrow, nb);
            if constexpr (kD == 128) cp_async16(S.v + off + kKVBytes / 2, P.Vg + vrow + 64, nb);
        }
    }
    if (warp == 13) {
        tmem_alloc(&S.tmem_base, 512);
        tmem_relinquish();
    }
    if (warp == 12) {
        // schedule: for each query head of the group, the active query tiles (ascending), two 64-row steps each
        if (lane == 0) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); prefetch_tmap(&tmG); }
        int n = 0;
        if constexpr (kCompact) {
            // Query tiles from the first key's tile to the tile of the last row that keeps one of the keys, or a part of that walk. The walk
            // goes BACKWARDS, from the last row that keeps one of the keys to the first key's row: the CTAs
            // of neighbouring entries of the permutation share their expiry band, i.e. the END of their walks, and start
            // about together, so walking down from there they pass the same query rows (the Q / dO tiles they load, the
            // dQ accumulator rows they add to) at about the same time, while those are in L2; walking up, each from its
            // own first key, they passed a row at times spread over the life of the whole group.
            const int g = hq_c % P.G, q0 = item.y & 0xFFFF, q1 = item.y >> 16, part = (item.x >> 10) & 7, parts = (item.x >> 13) & 0xF;
            const int all = walk_steps(q0, q1, P.L), p0 = all * part / parts, p1 = all * (part + 1) / parts;
            n = p1 - p0;
            for (int qt = q0 + lane; qt <= q1; qt += 32) {
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int pos = all - 1 - (2 * (qt - q0) + hf);
                    if (pos >= p0 && pos < p1) S.sched[pos - p0] = (uint16_t)((g << 11) | (qt << 1) | hf);
                }
            }
        } else {
        const int gper = P.G / nsplit;                     // this CTA's query heads of the group
        for (int g = sp * gper; g < (sp + 1) * gper; ++g) {
            const int bh = b * P.Hq + hk * P.G + g;
            for (int base = kt; base < P.Tr; base += 32) {
                const int qt = base + lane;
                const bool act = qt < P.Tr && (P.ignore_bitmap || bitmap_test(P.bitmap, P.Tr, P.Wd, bh, qt, kt));
                const int halves = act ? ((qt * 128 + 64 < P.L) ? 2 : 1) : 0;
                // exclusive prefix sum of `halves` over the warp
                int incl = halves;
                for (int o = 1; o < 32; o <<= 1) {
                    int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                const int pos = n + incl - halves;
                for (int hf = 0; hf < halves; ++hf)
                    if (pos + hf < kMaxSteps) S.sched[pos + hf] = (uint16_t)((g << 11) | (qt << 1) | hf);
                n += __shfl_sync(0xffffffffu, incl, 31);
            }
        }
        }
        if (lane == 0) S.n_steps = min(n, kMaxSteps);
    }
    if (warp == 15) {
        // constant A operand of the ninth k-step: zero block | rows (1, 1, 1, 0, ...) | zero block
        for (int r = lane; r < 128; r += 32) {
            *reinterpret_cast<uint4*>(S.ones[0] + r * 16) = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(S.ones[1] + r * 16) = make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
            *reinterpret_cast<uint4*>(S.ones[2] + r * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    const int n_steps = S.n_steps;

    if (warp < 8) {
        // ============================ compute group: thread = key j, 32 of the step's 64 query columns ============================
        const int quad = warp & 3, hsel = warp >> 2;
        const int r = quad * 32 + lane;                     // key within the tile = TMEM lane
        const int j = kCompact ? my_perm[r] : j0 + r;           // token-compacted mode: padding entries hold L
        const int jf = (kCompact && !P.causal) ? 0 : j;         // first row that can see the key
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        float bj = 0.0f;
        float2 dm2 = make_float2(0.0f, 0.0f);
        int len = 0, cur_g = -1;
        bool ok = true;
        if constexpr (kCompact) {
            cp_async_wait_all();       // (behind the barrier, so that the first Q and dO are requested meanwhile: 16 heads of 4096 keys, backward, 161.0 -> 157.6 us)
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.kv_full);
        }
        for (int n = 0; n < n_steps && ok; ++n) {
            const uint32_t e = S.sched[n];
            const int g = (int)(e >> 11), i0 = (int)((e >> 1) & 0x3FF) * 128 + (int)(e & 1) * 64;
            const int st = n % kStages;
            if (g != cur_g) {
                const int bh = b * P.Hq + hk * P.G + g;
                if (cur_g >= 0 && j < P.L) atomicAdd(&P.dM[(size_t)(bh - (g - cur_g)) * P.L + j], dm2.x + dm2.y);
                dm2 = make_float2(0.0f, 0.0f);
                bj = j < P.L ? P.bias[(size_t)bh * P.L + j] * 1.4426950408889634f : 0.0f;
                len = j < P.L ? max(0, P.expiry[(size_t)bh * P.L + j] - jf) : 0;
                cur_g = g;
            }
            // (S^T and dP^T were issued after the step's Q / dO stage was full: nothing else of that stage is read here)
            ok = mbar_wait_warp(&S.sdp_full, n & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint32_t sr[32], pr[32];
            tmem_ld32(tmem + lane_base + cS + hsel * 32, sr);
            tmem_ld32(tmem + lane_base + cDP + hsel * 32, pr);
            tc_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.sdp_free);
            // valid columns of this thread within its 32: col in [lo, lo + width)
            const int c0 = hsel * 32;
            const int lo = max(0, jf - i0 - c0);
            const int width = max(0, min(32, jf - i0 - c0 + len) - lo);
            // Almost every (key, 32-row group) pair is all-or-nothing: then the mask is one additive term per thread
            // (0 or -inf) and the per-element test is skipped. Warps with a partly kept key take the general loop.
            const bool uniform = __all_sync(0xffffffffu, width == 0 || (lo == 0 && width == 32));
            uint32_t pp[16], dd[16];
            const float2 sc2 = make_float2(P.scale_log2, P.scale_log2);
            if (uniform) {
                const float be = width ? bj : -INFINITY;
                const float2 bj2 = make_float2(be, be);
#pragma unroll
                for (int c = 0; c < 32; c += 4) {
                    const float2 x0 = fma2(make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), sc2, bj2);
                    const float2 x1 = fma2(make_float2(__uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3])), sc2, bj2);
                    const float2 t0 = make_float2(__uint_as_float(pr[c]), __uint_as_float(pr[c + 1]));
                    const float2 t1 = make_float2(__uint_as_float(pr[c + 2]), __uint_as_float(pr[c + 3]));
                    const float2 p0 = make_float2(ex2(x0.x), ex2(x0.y)), p1 = make_float2(ex2(x1.x), ex2(x1.y));
                    const float2 d0 = mul2(p0, t0), d1 = mul2(p1, t1);
                    dm2 = add2(dm2, add2(d0, d1));
                    pp[(c >> 1)] = pack_bf16(p0.x, p0.y);
                    pp[(c >> 1) + 1] = pack_bf16(p1.x, p1.y);
                    dd[(c >> 1)] = pack_bf16(d0.x, d0.y);
                    dd[(c >> 1) + 1] = pack_bf16(d1.x, d1.y);
                }
            } else {
                const float2 bj2 = make_float2(bj, bj);
#pragma unroll
                for (int c = 0; c < 32; c += 4) {
                    const float2 x0 = fma2(make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), sc2, bj2);
                    const float2 x1 = fma2(make_float2(__uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3])), sc2, bj2);
                    const float2 t0 = make_float2(__uint_as_float(pr[c]), __uint_as_float(pr[c + 1]));
                    const float2 t1 = make_float2(__uint_as_float(pr[c + 2]), __uint_as_float(pr[c + 3]));
                    float p[4] = {ex2(x0.x), ex2(x0.y), ex2(x1.x), ex2(x1.y)};
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const bool valid = (unsigned)(c + u - lo) < (unsigned)width;
                        p[u] = valid ? p[u] : 0.0f;
                    }
                    const float2 d0 = mul2(make_float2(p[0], p[1]), t0), d1 = mul2(make_float2(p[2], p[3]), t1);
                    dm2 = add2(dm2, add2(d0, d1));
                    pp[(c >> 1)] = pack_bf16(p[0], p[1]);
                    pp[(c >> 1) + 1] = pack_bf16(p[2], p[3]);
                    dd[(c >> 1)] = pack_bf16(d0.x, d0.y);
                    dd[(c >> 1) + 1] = pack_bf16(d1.x, d1.y);
                }
            }
            // the dV / dK / dQ GEMMs that last used this P^T / dS^T buffer (TMEM and smem) must have finished reading it:
            // those of the previous step, or with two buffers those of the step before it
            const int pb = kDouble ? (n & 1) : 0;
            if (kDouble) { if (n > 1) ok = mbar_wait_warp(&S.pds_free[pb], ((n >> 1) - 1) & 1, abort_flag); }
            else if (n > 0) ok = mbar_wait_warp(&S.pds_free[0], (n - 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            tmem_st16(tmem + lane_base + (pb ? cP1 : cP) + hsel * 16, pp);
            tmem_st16(tmem + lane_base + (pb ? cDS1 : cDS) + hsel * 16, dd);
            {   // dS^T row r -> shared memory: 16-byte chunk q of the row sits at q XOR (row % 8) (128-byte swizzle)
                uint8_t* row = (pb ? S.v + kKVBytes / 2 : S.ds) + r * 128;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    *reinterpret_cast<uint4*>(row + (((hsel * 4 + q) ^ (r & 7)) << 4)) = make_uint4(dd[4 * q], dd[4 * q + 1], dd[4 * q + 2], dd[4 * q + 3]);
            }
            fence_proxy_async();
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.pds_ready[pb]);
        }
        const int block = kCompact ? S.block : -1, part = kCompact ? S.part : 0, cut = kCompact ? S.cut : 0;
        if (cut && hsel == 0 && j < P.L) P.blocks.where[(size_t)bx * P.L + j] = r | cut;
        if (part) P.blocks.m[(((size_t)bx * P.Tc + kt) * (kMostParts - 1) + part - 1) * 256 + hsel * 128 + r] = dm2.x + dm2.y;
        else if (cur_g >= 0 && j < P.L) atomicAdd(&P.dM[(size_t)(b * P.Hq + hk * P.G + cur_g) * P.L + j], dm2.x + dm2.y);
        // epilogue: dK (scaled) and dV rows to global memory; warps w and w+4 each write one half of the channels
        if (ok && n_steps > 0)
            ok = kDouble ? mbar_wait_warp(&S.pds_free[(n_steps - 1) & 1], ((n_steps - 1) >> 1) & 1, abort_flag)
                         : mbar_wait_warp(&S.pds_free[0], (n_steps - 1) & 1, abort_flag);
        if (ok) {
            tc_fence_after();
            // A thread holds 32 channels of its key's row. The warp turns each such block of 32 rows around in shared memory (the Q stages, which
            // the last MMAs have left; 16-byte chunks swizzled by the row), so that eight lanes write 128 consecutive bytes of a row, and the
            // block after it is on its way from tensor memory meanwhile. What is left is the stores and reductions themselves, 14 to 32 bytes per clock:
            // 6000 clk for fp32 parts (10000 without the turn), 8400 for reductions, 5400 for bf16 rows.
            uint8_t* turn = S.q[0] + warp * 4096;
            static_assert(sizeof(S.q) >= 8 * 4096, "a block of 32 x 32 floats per compute warp");
            const int rsub = lane >> 3, ch = lane & 7;
            int jr[8];                                             // keys of the rows this lane writes a part of
#pragma unroll
            for (int t = 0; t < 8; ++t) jr[t] = __shfl_sync(0xffffffffu, j, 4 * t + rsub);
            uint32_t o[32];
            auto fetch = [&](int blk) { tmem_ld32(tmem + lane_base + (blk < kHalves ? cDK : cDV) + (hsel * kHalves + blk % kHalves) * 32, o); };
#pragma unroll
            for (int u = 0; u < 32; ++u) o[u] = 0u;
            if (n_steps > 0) fetch(0);
#pragma unroll 1
            for (int blk = 0; blk < 2 * kHalves; ++blk) {
                const bool isK = blk < kHalves;
                const int col = (hsel * kHalves + blk % kHalves) * 32 + ch * 4;
                if (n_steps > 0) tc_wait_ld_dep(o);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    *reinterpret_cast<uint4*>(turn + lane * 128 + ((q ^ (lane & 7)) << 4)) = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
                if (n_steps > 0 && blk + 1 < 2 * kHalves) fetch(blk + 1);
                __syncwarp();
                float4 x[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int row = 4 * t + rsub;
                    x[t] = *reinterpret_cast<const float4*>(turn + row * 128 + ((ch ^ (row & 7)) << 4));
                }
                if (kCompact && block >= 0) {
                    float* dst = P.blocks.kv + (((size_t)bx * P.blocks.cap + block) * 2 + (isK ? 0 : 1)) * (128 * kD) + quad * (32 * kD) + col;
#pragma unroll
                    for (int t = 0; t < 8; ++t) *reinterpret_cast<float4*>(dst + (4 * t + rsub) * kD) = x[t];
                } else if (kCompact || nsplit > 1) {
                    // Unscaled sums in fp32. Token-compacted: the group's query heads add into the same rows, or (slots) this (key, query head) pair is
                    // written by this CTA alone. Tile mode: this split's part, zeros where it had nothing to add.
                    float* acc = (isK ? P.dKacc : P.dVacc) + (size_t)(kCompact ? hq_c % P.G : sp) * (size_t)P.acc_slot +
                                 ((size_t)b * P.L * P.Hkv + hk) * kD + col;
                    const bool red = kCompact && P.acc_slot == 0;
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        float* row = acc + (int64_t)jr[t] * (P.Hkv * kD);
                        if (jr[t] < P.L && (!kCompact || n_steps > 0)) {
                            if (red) red_add_v4(row, x[t].x, x[t].y, x[t].z, x[t].w);
                            else *reinterpret_cast<float4*>(row) = x[t];
                        }
                    }
                } else {
                    const float mul = isK ? P.scale : 1.0f;
                    __nv_bfloat16* out = (isK ? P.dK + b * P.ks_b + hk * P.ks_h : P.dV + b * P.vs_b + hk * P.vs_h) + col;
                    const int64_t out_l = isK ? P.ks_l : P.vs_l;
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if (jr[t] < P.L)
                            *reinterpret_cast<uint2*>(out + jr[t] * out_l) = make_uint2(pack_bf16(x[t].x * mul, x[t].y * mul), pack_bf16(x[t].z * mul, x[t].w * mul));
                }
                __syncwarp();                                      // (the block has been read)
            }
        }
    } else if (warp < 12) {
        // ============================ dQ drain group: thread = channel c, columns = query rows ============================
        // Each warp owns 32 channels and its own pair of staging buffers (16 query rows each, used in turn), so the
        // warps never wait for each other: a buffer is rewritten once the reduce-add issued from it two groups ago has
        // finished reading it.
        // d = 64: lanes 64-127 of dQ^T repeat lanes 0-63 (the K tile sits in both halves of its buffer), so warps 2 and 3
        // own the same channels as warps 0 and 1 and take the second half of the step's rows.
        const int dw = warp & 3;
        constexpr int kQuarters = kD == 64 ? 2 : 4;                     // quarter steps per warp
        const int ch = kD == 64 ? (dw & 1) : dw, qr0 = kD == 64 ? (dw >> 1) * 2 : 0;
        const uint32_t lane_base = (uint32_t)(dw * 32) << 16;
        bool ok = true;
        for (int n = 0; n < n_steps && ok; ++n) {
            const uint32_t e = S.sched[n];
            const int g = (int)(e >> 11), i0 = (int)((e >> 1) & 0x3FF) * 128 + (int)(e & 1) * 64;
            ok = mbar_wait_warp(&S.dq_full, n & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            uint32_t v[kQuarters * 16];
#pragma unroll
            for (int c = 0; c < kQuarters / 2; ++c)
                tmem_ld32(tmem + lane_base + cDQ + qr0 * 16 + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&v[c * 32]));
            tc_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.dq_free);
#pragma unroll
            for (int q = 0; q < kQuarters; ++q) {      // quarter steps of 16 query rows, two staging buffers in turn
                const int qr = qr0 + q;
                if (lane == 0) bulk_wait_read_1(); __syncwarp();
                {   // this thread's channel, 16 rows: four 16-byte stores (see BwdParams::dQacc for the block's layout)
                    uint8_t* line = reinterpret_cast<uint8_t*>(&S.dq_stage[dw][q & 1][0][0]) + lane * 64;
#pragma unroll
                    for (int qq = 0; qq < 4; ++qq)
                        *reinterpret_cast<uint4*>(line + ((qq ^ ((lane >> 1) & 3)) << 4)) =
                            make_uint4(v[q * 16 + 4 * qq], v[q * 16 + 4 * qq + 1], v[q * 16 + 4 * qq + 2], v[q * 16 + 4 * qq + 3]);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0 && i0 + qr * 16 < P.L) {       // (rows beyond L inside the block land in the accumulator's padding)
                    float* blk = P.dQacc + ((((size_t)(b * P.Hq + hk * P.G + g) * P.Lblk + (i0 >> 4) + qr) * (kD / 32) + ch) << 9);
                    bulk_reduce_add_f32(blk, &S.dq_stage[dw][q & 1][0][0], 2048);
                }
                if (lane == 0) bulk_commit();
            }
        }
        if (lane == 0) bulk_wait_all();
    } else {
        if (warp == 12) {
            // ============================ producer ============================
            bool ok = true;
            for (int n = 0; n < n_steps && ok; ++n) {
                const uint32_t e = S.sched[n];
                const int h = hk * P.G + (int)(e >> 11), i0 = (int)((e >> 1) & 0x3FF) * 128 + (int)(e & 1) * 64;
                const int st = n % kStages;
                if (n >= kStages) ok = mbar_wait_warp(&S.qd_empty[st], ((n / kStages) - 1) & 1, abort_flag);
                if (!ok) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&S.qd_full[st], kHalves * kQBytes);
                    for (int hf = 0; hf < kHalves; ++hf) {
                        tma_load_4d(&S.q[st][hf * (kQBytes / 2)], &tmQ, &S.qd_full[st], hf * 64, i0, h, b);
                        tma_load_4d(&S.g[st][hf * (kQBytes / 2)], &tmG, &S.qd_full[st], hf * 64, i0, h, b);
                    }
                }
            }
            for (int n = max(0, n_steps - kStages); n < n_steps && ok; ++n)
                ok = mbar_wait_warp(&S.qd_empty[n % kStages], (n / kStages) & 1, abort_flag);
        } else if (warp == 15) {
            // ============================ stager: ninth k-step B operand (-lse / scale, -D) of each step's query rows, loaded one step ahead ============================
            auto fetch = [&](int n, float (&lv)[2], float (&dv)[2]) {
                const uint32_t e = S.sched[n];
                const int h = hk * P.G + (int)(e >> 11), i0 = (int)((e >> 1) & 0x3FF) * 128 + (int)(e & 1) * 64;
                const size_t rowbase = (size_t)(b * P.Hq + h) * P.L;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int i = i0 + lane + 32 * t;
                    lv[t] = i < P.L ? P.lse[rowbase + i] : 0.0f;
                    dv[t] = i < P.L ? P.Dv[rowbase + i] : 0.0f;
                }
            };
            float lv[2] = {0.f, 0.f}, dv[2] = {0.f, 0.f};
            if (n_steps > 0) fetch(0, lv, dv);
            bool ok = true;
            for (int n = 0; n < n_steps && ok; ++n) {
                const int st = n % kStages;
                float ln[2] = {0.f, 0.f}, dn[2] = {0.f, 0.f};
                if (n + 1 < n_steps) fetch(n + 1, ln, dn);
                if (n >= kStages) ok = mbar_wait_warp(&S.qd_empty[st], ((n / kStages) - 1) & 1, abort_flag);
                if (!ok) break;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int r = lane + 32 * t;
                    uint8_t* row = S.qext[st] + (r >> 3) * 256 + (r & 7) * 16;
                    *reinterpret_cast<uint4*>(row) = split3(-lv[t] * P.inv_scale);        // elements 0-2: -lse_i / scale
                    *reinterpret_cast<uint4*>(row + 128) = split3(-dv[t]);                // elements 8-10: -D_i
                    lv[t] = ln[t];
                    dv[t] = dn[t];
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.qd_full[st]);
            }
        } else if (warp == 13) {
            // ============================ MMA issuer 1: S^T = K Q^T, dP^T = V dO^T ============================
            // (two issuing warps: every hand-over between them and the other groups is an explicit mbarrier, nothing
            //  relies on the order of their MMAs. Each walks the schedule as a whole warp with warp-uniform values, so
            //  that descriptors and counters stay in the uniform datapath; one elected lane issues.)
            constexpr uint32_t id_sdp = idesc_bf16(128, 64, 0, 0);     // K|V (K-major) x Q|dO (K-major)       -> 128 x 64
            const uint64_t dK = smem_desc_sw128(smem_u32(S.k), 16, 1024), dV = smem_desc_sw128(smem_u32(S.v), 16, 1024);
            const uint64_t dQ0 = smem_desc_sw128(smem_u32(S.q[0]), 16, 1024), dG0 = smem_desc_sw128(smem_u32(S.g[0]), 16, 1024);
            // ninth k-step: 8-row groups 128 bytes apart, second K core matrix one 2 KB block further (A) / 128 bytes further (B)
            const uint64_t dOnesLo = smem_desc_plain(smem_u32(S.ones[1]), 2048, 128), dOnesHi = smem_desc_plain(smem_u32(S.ones[0]), 2048, 128);
            const uint64_t dX0 = smem_desc_plain(smem_u32(S.qext[0]), 128, 256);
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
            const int n_steps_u = __shfl_sync(0xffffffffu, n_steps, 0);
            bool ok = mbar_wait_warp(&S.kv_full, 0, abort_flag);
            if constexpr (kCompact) fence_proxy_async();     // the gathered rows were written through the generic proxy
            for (int n = 0; n < n_steps_u && ok; ++n) {
                const int st = n % kStages;
                ok = mbar_wait_warp(&S.qd_full[st], (n / kStages) & 1, abort_flag);
                if (ok && n > 0) ok = mbar_wait_warp(&S.sdp_free, (n - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint64_t dQ = dQ0 + (uint64_t)(st * (kQBytes >> 4)), dG = dG0 + (uint64_t)(st * (kQBytes >> 4));
                const uint64_t dX = dX0 + (uint64_t)(st * (2048 >> 4));
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kD / 16; ++kk)
                        mma_ss(tmem_u + cS, dK + (uint64_t)(((kk >> 2) * (kKVBytes / 2) + (kk & 3) * 32) >> 4),
                               dQ + (uint64_t)(((kk >> 2) * (kQBytes / 2) + (kk & 3) * 32) >> 4), id_sdp, kk > 0);
                    mma_ss(tmem_u + cS, dOnesLo, dX, id_sdp, 1u);          // S^T  += 1 (x) (-lse / scale)
#pragma unroll
                    for (int kk = 0; kk < kD / 16; ++kk)
                        mma_ss(tmem_u + cDP, dV + (uint64_t)(((kk >> 2) * (kKVBytes / 2) + (kk & 3) * 32) >> 4),
                               dG + (uint64_t)(((kk >> 2) * (kQBytes / 2) + (kk & 3) * 32) >> 4), id_sdp, kk > 0);
                    mma_ss(tmem_u + cDP, dOnesHi, dX, id_sdp, 1u);         // dP^T += 1 (x) (-D)
                    tc_commit(&S.sdp_full);
                }
                __syncwarp();
            }
        } else if (warp == 14) {
            // ============================ MMA issuer 2: dV += P^T dO, dK += dS^T Q, dQ^T = K^T dS^T ============================
            constexpr uint32_t id_dkv = idesc_bf16(128, kD, 0, 1);     // P^T|dS^T (TMEM) x dO|Q (MN-major)    -> 128 x d
            constexpr uint32_t id_dq = idesc_bf16(128, 64, 1, 1);      // K^T (MN-major) x dS^T (MN-major)     -> 128 x 64
            const uint64_t dKt = smem_desc_sw128(smem_u32(S.k), kKVBytes / 2, 1024), dDs0 = smem_desc_sw128(smem_u32(S.ds), 16, 1024);
            const uint64_t dDs1 = smem_desc_sw128(smem_u32(S.v + kKVBytes / 2), 16, 1024);      // second dS^T buffer (d = 64)
            const uint64_t dGm0 = smem_desc_sw128(smem_u32(S.g[0]), kQBytes / 2, 1024), dQm0 = smem_desc_sw128(smem_u32(S.q[0]), kQBytes / 2, 1024);
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
            const int n_steps_u = __shfl_sync(0xffffffffu, n_steps, 0);
            bool ok = true;
            for (int n = 0; n < n_steps_u && ok; ++n) {
                const int st = n % kStages;
                const int pb = kDouble ? (n & 1) : 0;
                ok = mbar_wait_warp(&S.pds_ready[pb], (kDouble ? (n >> 1) : n) & 1, abort_flag);
                if (ok && n > 0) ok = mbar_wait_warp(&S.dq_free, (n - 1) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tP = tmem_u + (pb ? cP1 : cP), tDS = tmem_u + (pb ? cDS1 : cDS);
                const uint64_t dDs = pb ? dDs1 : dDs0;
                const uint64_t dGm = dGm0 + (uint64_t)(st * (kQBytes >> 4)), dQm = dQm0 + (uint64_t)(st * (kQBytes >> 4));
                const uint32_t acc0 = n > 0 ? 1u : 0u;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)         // 64 query rows = 4 k-steps of 16
                        mma_ts(tmem_u + cDV, tP + kk * 8, dGm + (uint64_t)((kk * 2048) >> 4), id_dkv, kk > 0 ? 1u : acc0);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_ts(tmem_u + cDK, tDS + kk * 8, dQm + (uint64_t)((kk * 2048) >> 4), id_dkv, kk > 0 ? 1u : acc0);
                    tc_commit(&S.qd_empty[st]);            // the dQ GEMM reads K and dS^T only: Q / dO of this stage are free here
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)         // 128 keys = 8 k-steps of 16
                        mma_ss(tmem_u + cDQ, dKt + (uint64_t)((kk * 2048) >> 4), dDs + (uint64_t)((kk * 2048) >> 4), id_dq, kk > 0);
                    tc_commit(&S.pds_free[pb]);
                    tc_commit(&S.dq_full);
                }
                __syncwarp();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 13) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    if (tid == 0 && S.abort_flag) atomicExch(P.status, (int32_t)DMA_ERR_DEVICE_TIMEOUT);
}

// What the backward needs before its main kernel, in one launch: D_i = dO_i . O_i (Alg. 2; kLanes = d / 8 lanes per (b, h, i),
// 16-byte loads) and zeros in the accumulators that are added to. HBM-bound (at L = 16384 with 32 / 8 heads of 128 channels
// 268 MB read, 405 MB written); the CTAs' parts of the zeros are as large as their parts of the rows, so that loads and
// stores are in flight together, and a short problem has one launch instead of four.
struct PrepareParams {
    const __nv_bfloat16* O;
    const __nv_bfloat16* dO;
    float* Dv;
    int B, L, Hq;
    int64_t os_b, os_l, os_h;
    float* zero[3];             // accumulator of dQ, dM, accumulators of dK and dV: 16-byte aligned
    int64_t zero_n[3];          // floats
    int64_t zero_part[3];       // 16-byte chunks per CTA
    int32_t* status;            // the workspace header
    // token-compacted mode: the first perm_ctas CTAs (one per (batch, query head), 1024 threads) make the head's permutation and work items
    int perm_ctas;
    const int32_t* expiry;
    int* perm;
    int2* items;
    int cap, direct;            // as WalkBlocks
    int Tc, causal, max_items;
    int walk;                   // steps of a walk that one CTA takes at most
    int longest_first;          // order of a head's items: by length, or as the permutation has them
};
constexpr int kPrepareRows = 4;     // rows per lane group
constexpr int kPermThreads = 1024;

// Token-compacted mode: per (batch, query head) a stable counting sort of the keys by the band their expiry falls in (latest expiry
// first; keys that no row keeps go last). Within a band the keys stay in index order, so 128 consecutive entries start at nearby rows
// and expire within one band of each other: on i.i.d. importance at L = 16384, w = 2048 the walk covers 1.4 x the (row, key) pairs
// actually kept, against 4.3 x for tiles of consecutive keys. Bands of L / 8 rows, 128 to 2048, at most 62 (counted offline over windows of
// L / 16 to L / 4: within 3 % of the best width at 4096, 8192 and 16384 keys; 2048-row bands cover 15 % more at 4096). Padded with L up to Tc * 128.
// One CTA of 1024 threads per (batch, head). Per 1024-key chunk every warp ranks its 32 keys within their class
// (match_any), the per-warp class counts are turned into start positions by 64 threads (one per class, a running sum over
// the 32 warps and over the chunks), and every key is written to its place: stable in key order, three barriers per chunk.
// Then the work items: a warp per key tile finds its walk, walks longer than P.walk steps are cut into equal parts (as long as the head has
// blocks left for them, in the permutation's order), and with P.longest_first the items are ranked by length, so that no long one starts late.
struct PermShared {
    int hist[64];
    int offs[64];                 // next free position of each class
    int cnt[32][64];              // per warp and class: keys in this chunk, then their start position
    int bounds[1024];             // walk of each key tile, q0 | q1 << 16 (meaningless where parts = 0)
    int parts[1024], len[1024], first[1024];
};
__device__ __forceinline__ void lifetime_perm(const PrepareParams& P, PermShared& S) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, bh = blockIdx.x, L = P.L, Tc = P.Tc;
    const int32_t* e = P.expiry + (size_t)bh * L;
    int* out = P.perm + (size_t)bh * Tc * 128;
    const int band = max((L + 61) / 62, min(2048, max(128, L / 8)));
    auto cls = [&](int j) { return e[j] > (P.causal ? j : 0) ? 1 + (e[j] - 1) / band : 0; };
    if (tid < 64) S.hist[tid] = 0;
    __syncthreads();
    for (int j = tid; j < L; j += kPermThreads) atomicAdd(&S.hist[cls(j)], 1);
    __syncthreads();
    if (tid == 0) {
        int run = 0;
        for (int c = 63; c >= 0; --c) { S.offs[c] = run; run += S.hist[c]; }
    }
    __syncthreads();
    for (int base = 0; base < L; base += kPermThreads) {
        const int j = base + tid;
        const int c = j < L ? cls(j) : -1;
        const uint32_t same = __match_any_sync(0xffffffffu, c);
        const int leader = __ffs(same) - 1, rank = __popc(same & ((1u << lane) - 1));
        S.cnt[warp][lane] = 0;
        S.cnt[warp][lane + 32] = 0;
        __syncwarp();
        if (lane == leader && c >= 0) S.cnt[warp][c] = __popc(same);
        __syncthreads();
        if (tid < 64) {
            int run = S.offs[tid];
            for (int w = 0; w < 32; ++w) {
                const int n = S.cnt[w][tid];
                S.cnt[w][tid] = run;
                run += n;
            }
            S.offs[tid] = run;
        }
        __syncthreads();
        if (c >= 0) out[S.cnt[warp][c] + rank] = j;
        __syncthreads();
    }
    for (int t = L + tid; t < Tc * 128; t += kPermThreads) out[t] = L;
    __syncthreads();                                        // (the CTA reads its own entries back)
    for (int t = warp; t < Tc; t += 32) {
        int first = 0x7fffffff, last = 0;
        for (int u = 0; u < 4; ++u) {
            const int j = out[t * 128 + lane + 32 * u];
            const int ej = j < L ? e[j] : 0, f = P.causal ? j : 0;
            if (ej > f) { first = min(first, f); last = max(last, ej); }
        }
        first = __reduce_min_sync(0xffffffffu, first);
        last = __reduce_max_sync(0xffffffffu, last);
        if (lane == 0) {
            const int q0 = first >> 7, q1 = (last - 1) >> 7, n = last > 0 ? walk_steps(q0, q1, L) : 0;
            const int parts = min(min(kMostParts, P.max_items / Tc), (n + P.walk - 1) / P.walk);        // (0: no row keeps a key of the tile)
            S.bounds[t] = q0 | (q1 << 16);
            S.parts[t] = parts;
            S.len[t] = parts ? n / parts : 0;
        }
    }
    __syncthreads();
    if (P.max_items > Tc) {                                 // walks are cut
        const int later = tid < Tc ? max(S.parts[tid] - P.direct, 0) : 0;
        int to = later;                                     // blocks up to this tile's, in the permutation's order
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, to, o);
            if (lane >= o) to += t;
        }
        if (lane == 31) S.hist[warp] = to;
        __syncthreads();
        to += __reduce_add_sync(0xffffffffu, lane < warp ? S.hist[lane] : 0);
        const int from = min(to - later, P.cap);
        to = min(to, P.cap);
        if (tid < Tc) {
            S.first[tid] = from;
            if (S.parts[tid] > 0) {
                S.parts[tid] = min(S.parts[tid], P.direct + to - from);
                S.len[tid] = walk_steps(S.bounds[tid] & 0xFFFF, S.bounds[tid] >> 16, L) / S.parts[tid];
            }
        }
        __syncthreads();
    }
    int2* items = P.items + (size_t)bh * P.max_items;
    if (tid < Tc) {
        const int parts = S.parts[tid], len = S.len[tid];
        int at = 0;
        for (int u = 0; u < Tc; ++u) at += (P.longest_first ? S.len[u] > len || (S.len[u] == len && u < tid) : u < tid) ? S.parts[u] : 0;
        for (int q = 0; q < parts; ++q) items[at + q] = make_int2(tid | q << 10 | parts << 13 | (parts > 1 ? S.first[tid] + max(q - P.direct, 0) : 0) << 17, S.bounds[tid]);
    }
    int total = 0;
    for (int u = lane; u < Tc; u += 32) total += S.parts[u];
    total = __reduce_add_sync(0xffffffffu, total);
    for (int t = total + tid; t < P.max_items; t += kPermThreads) items[t] = make_int2(-1, 0);
}

template <int kLanes, bool kPerm>
__global__ void __launch_bounds__(kPerm ? kPermThreads : 256) bwd_prepare_kernel(const PrepareParams P) {
    constexpr int nthr = kPerm ? kPermThreads : 256;
    pdl_enter();
    if (blockIdx.x == 0 && threadIdx.x < kWsHeaderBytes / 4) P.status[threadIdx.x] = 0;
    if constexpr (kPerm) {
        __shared__ PermShared S;
        if ((int)blockIdx.x < P.perm_ctas) {
            lifetime_perm(P, S);
            return;
        }
    }
    const int cta = (int)blockIdx.x - (kPerm ? P.perm_ctas : 0);
    const int sub = threadIdx.x % kLanes, per_cta = nthr / kLanes;
    const uint32_t rows = (uint32_t)P.B * P.Hq * P.L, r0 = cta * per_cta * kPrepareRows + threadIdx.x / kLanes;
    uint4 a[kPrepareRows], g[kPrepareRows];
#pragma unroll
    for (int n = 0; n < kPrepareRows; ++n) {
        const uint32_t row = min(r0 + n * per_cta, rows - 1), bh = row / (uint32_t)P.L;
        const int i = (int)(row - bh * P.L), h = (int)(bh % (uint32_t)P.Hq), b = (int)(bh / (uint32_t)P.Hq);
        const int64_t off = b * P.os_b + (int64_t)i * P.os_l + h * P.os_h + sub * 8;
        a[n] = *reinterpret_cast<const uint4*>(P.O + off);
        g[n] = *reinterpret_cast<const uint4*>(P.dO + off);
    }
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        const int64_t n4 = P.zero_n[z] >> 2, e0 = P.zero_part[z] * cta, e1 = min(n4, e0 + P.zero_part[z]);
        float4* dst = reinterpret_cast<float4*>(P.zero[z]);
        for (int64_t e = e0 + threadIdx.x; e < e1; e += nthr) dst[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (cta == 0 && threadIdx.x < (P.zero_n[z] & 3)) P.zero[z][4 * n4 + threadIdx.x] = 0.0f;
    }
#pragma unroll
    for (int n = 0; n < kPrepareRows; ++n) {
        const uint32_t au[4] = {a[n].x, a[n].y, a[n].z, a[n].w}, gu[4] = {g[n].x, g[n].y, g[n].z, g[n].w};
        float s = 0.0f;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            s = fmaf(__uint_as_float(au[t] << 16), __uint_as_float(gu[t] << 16), s);
            s = fmaf(__uint_as_float(au[t] & 0xffff0000u), __uint_as_float(gu[t] & 0xffff0000u), s);
        }
        for (int m = kLanes / 2; m; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
        const uint32_t row = r0 + n * per_cta;
        if (sub == 0 && row < rows) P.Dv[row] = s;
    }
}

// After the main kernel, in one launch (HBM-bound): the first q_blocks CTAs turn the blocked fp32 dQ accumulator (see
// BwdParams::dQacc) into bf16 dQ in the caller's layout, softmax scale applied; the others the fp32 dK, dV accumulators
// [B, L, Hkv, d] where the main kernel did not write dK, dV itself.
//   dQ: kFinishBlocks 2 KB blocks (16 rows x 32 channels) per warp, read as they lie (512 consecutive bytes per instruction, all of a
//   warp's loads in flight), turned around as bf16 in shared memory and written 256 (d = 64: 128) consecutive bytes per row. Reading
//   a channel pair's rows per thread instead, 16 bytes out of every 128, took 32 passes per load: at L = 16384 with 32 heads of 128 channels
//   121 us (backward 2221 -> 2097), 16 heads of 4096 (backward 163 -> 159).
//   dK, dV: 8 elements per thread. nslots > 1: the accumulator is nslots copies, slot_stride elements apart, added in slot
//   order (a fixed order: the result is then the same bits from run to run). Where walks were cut, the blocks of the group's heads after that.
//   dM: only where walks were cut, a thread per key.
struct FinishParams {
    const float* dQacc;
    const float* acc[2];        // of dK, dV
    __nv_bfloat16* dQ;
    __nv_bfloat16* out[2];
    int q_blocks, kv_blocks;    // CTAs of dQ, of each of dK and dV
    int L, Hq, Hkv, Lblk, nslots;
    int64_t nkv, rows;          // elements of dK, of dM
    uint32_t q_rows16;          // 16-row blocks of dQ in all
    int64_t qs[3], st[2][3];
    float scale;
    WalkBlocks blocks;
    float* dM;
};

constexpr int kFinishBlocks = 1;       // (two: more loads in flight, but 8 heads of 500 keys, backward, 21.3 -> 22.1 us, 32 heads of 16384 2139 -> 2154)

// kBlocks: walks have left blocks
template <int kD, bool kBlocks>
__device__ __forceinline__ void finish(const FinishParams& P) {
    constexpr int kCh = kD / 32, kRowBlocks = 8 / kCh * kFinishBlocks;     // channel blocks of a row, 16-row blocks of a CTA
    constexpr int kPitch = kD / 2 + 4;                                     // 4-byte words per row: 16-byte aligned, rows 4 apart 16 banks apart
    __shared__ __align__(16) uint32_t turn[kRowBlocks * 16 * kPitch];
    pdl_enter();
    if ((int)blockIdx.x < P.q_blocks) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ch = warp % kCh;
        const uint32_t blk0 = blockIdx.x * kRowBlocks;
        float4 x[kFinishBlocks][4];
#pragma unroll
        for (int n = 0; n < kFinishBlocks; ++n) {
            const uint32_t blk = min(blk0 + warp / kCh + n * (8 / kCh), P.q_rows16 - 1);
            const float4* src = reinterpret_cast<const float4*>(P.dQacc + ((size_t)blk * kCh + ch) * 512) + lane;
#pragma unroll
            for (int u = 0; u < 4; ++u) x[n][u] = src[32 * u];
        }
#pragma unroll
        for (int n = 0; n < kFinishBlocks; ++n) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = 8 * u + (lane >> 2), q = (lane & 3) ^ ((c >> 1) & 3);       // channel of the block, quad of rows (BwdParams::dQacc)
                __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(turn + ((warp / kCh + n * (8 / kCh)) * 16 + 4 * q) * kPitch) + ch * 32 + c;
                dst[0] = __float2bfloat16_rn(x[n][u].x * P.scale);
                dst[2 * kPitch] = __float2bfloat16_rn(x[n][u].y * P.scale);
                dst[4 * kPitch] = __float2bfloat16_rn(x[n][u].z * P.scale);
                dst[6 * kPitch] = __float2bfloat16_rn(x[n][u].w * P.scale);
            }
        }
        __syncthreads();
        constexpr int kParts = kD / 8;                                     // 16-byte parts of a row
#pragma unroll
        for (int t = threadIdx.x; t < kRowBlocks * 16 * kParts; t += 256) {
            const int r = t / kParts, part = t % kParts;
            const uint32_t blk = blk0 + r / 16;
            if (blk >= P.q_rows16) continue;
            const int bh = (int)(blk / (uint32_t)P.Lblk), i = (int)(blk - (uint32_t)bh * P.Lblk) * 16 + r % 16, h = bh % P.Hq, b = bh / P.Hq;
            if (i < P.L)
                *reinterpret_cast<uint4*>(P.dQ + b * P.qs[0] + (int64_t)i * P.qs[1] + h * P.qs[2] + part * 8) = *reinterpret_cast<const uint4*>(turn + r * kPitch + part * 4);
        }
        return;
    }
    const int blk = (int)blockIdx.x - P.q_blocks, which = blk / P.kv_blocks;
    if (blk >= 2 * P.kv_blocks) {
        const int64_t row = (int64_t)(blk - 2 * P.kv_blocks) * 256 + threadIdx.x;
        const int at = row < P.rows ? P.blocks.where[row] : 0, n = (at >> 7) & 7;
        if (n == 0) return;
        const float* m = P.blocks.m + ((size_t)(row / P.L) * (P.Lblk / 8) + (at >> 19)) * ((kMostParts - 1) * 256) + (at & 127);
        float sum = P.dM[row];
#pragma unroll 4
        for (int p = 0; p < n; ++p) sum += m[p * 256] + m[p * 256 + 128];
        P.dM[row] = sum;
        return;
    }
    const int64_t e = ((int64_t)(blk % P.kv_blocks) * 256 + threadIdx.x) * 8;
    if (e >= P.nkv) return;
    const float* acc = P.acc[which];
    auto add = [](float4& x, float4& y, const float* p) {
        const float4 x2 = *reinterpret_cast<const float4*>(p), y2 = *reinterpret_cast<const float4*>(p + 4);
        x.x += x2.x; x.y += x2.y; x.z += x2.z; x.w += x2.w; y.x += y2.x; y.y += y2.y; y.z += y2.z; y.w += y2.w;
    };
    const uint32_t row = (uint32_t)(e / kD), bl = row / (uint32_t)P.Hkv;
    const int c = (int)(e % kD), h = (int)(row - bl * P.Hkv), b = (int)(bl / (uint32_t)P.L), i = (int)(bl - (uint32_t)b * P.L);
    int at[2] = {0, 0};                                                    // (blocks: one or two query heads per KV head)
    if constexpr (kBlocks) {
        at[0] = P.blocks.where[(size_t)(b * P.Hq + h * (P.Hq / P.Hkv)) * P.L + i];
        if (P.Hq != P.Hkv) at[1] = P.blocks.where[(size_t)(b * P.Hq + h * 2 + 1) * P.L + i];
    }
    float4 a = *reinterpret_cast<const float4*>(acc + e), bb = *reinterpret_cast<const float4*>(acc + e + 4);
    for (int sl = 1; sl < P.nslots; ++sl) add(a, bb, acc + sl * P.nkv + e);
    if constexpr (kBlocks) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int n = ((at[g] >> 7) & 7) + 1 - P.blocks.direct;
            const float* src = P.blocks.kv + (((size_t)(b * P.Hq + h * (P.Hq / P.Hkv) + g) * P.blocks.cap + ((at[g] >> 10) & 0x1FF)) * 2 + which) * (128 * kD) +
                               (at[g] & 127) * kD + c;
#pragma unroll 2
            for (int p = 0; p < n; ++p) add(a, bb, src + p * (2 * 128 * kD));
        }
    }
    const float scale = which == 0 ? P.scale : 1.0f;
    uint4 o;
    o.x = ptx::pack_bf16(a.x * scale, a.y * scale); o.y = ptx::pack_bf16(a.z * scale, a.w * scale);
    o.z = ptx::pack_bf16(bb.x * scale, bb.y * scale); o.w = ptx::pack_bf16(bb.z * scale, bb.w * scale);
    *reinterpret_cast<uint4*>(P.out[which] + b * P.st[which][0] + (int64_t)i * P.st[which][1] + h * P.st[which][2] + c) = o;
}

template <int kD>
__global__ void __launch_bounds__(256) bwd_finish_kernel(const FinishParams P) { finish<kD, false>(P); }
// (registers for six CTAs per SM instead of four: 8 heads of 8192 keys, backward 189 -> 185 us)
template <int kD>
__global__ void __launch_bounds__(256, 6) bwd_finish_blocks_kernel(const FinishParams P) { finish<kD, true>(P); }

}  // namespace

// workspace layout: header | D [rows] | dQ accumulator [B x Hq x (Tr x 128) x d] | (token-compacted mode) permutation, work items, where each
// key's walk left its later parts' sums | dK, dV accumulators | those sums
static size_t bwd_rows64(const Prob& P) { return ((((size_t)P.B * P.Hq * P.L) + 63) / 64) * 64; }
static size_t bwd_acc_floats(const Prob& P) { return (size_t)P.B * P.Hq * P.Tr * 128 * P.d; }     // rows padded to whole query tiles
// permutation and work items
static size_t bwd_perm_ints(const Prob& P) { return (size_t)P.B * P.Hq * P.Tc * 128; }
static size_t bwd_item_ints(const Prob& P) { return ((size_t)P.B * P.Hq * P.Tc * 2 * kMostParts + 63) / 64 * 64; }
// What cut walks take (WalkBlocks). Walks are never cut with DMA_FLAG_DETERMINISTIC.
static bool bwd_may_cut(const Prob& P) { return (P.flags & DMA_FLAG_COMPACT_KV) && !(P.flags & DMA_FLAG_DETERMINISTIC); }
static int bwd_heads(const Prob& P) { return P.bwd_heads ? P.bwd_heads : P.B * P.Hq; }
static size_t bwd_where_ints(const Prob& P) { return bwd_may_cut(P) ? bwd_rows64(P) : 0; }
static size_t bwd_part_floats(const Prob& P) { return bwd_may_cut(P) ? (size_t)P.B * P.Hq * P.Tc * (kMostParts - 1) * 256 : 0; }
static size_t bwd_blocks(const Prob& P) { return bwd_may_cut(P) && P.G <= 2 ? std::min((size_t)P.B * P.Hq * P.Tc * (kMostParts - 1), (size_t)kWalkBlocks) : 0; }
static int bwd_blocks_per_head(const Prob& P) { return P.G <= 2 ? std::min(P.Tc * (kMostParts - 1), kWalkBlocks / bwd_heads(P)) : 0; }

// Tile mode: a CTA owns a key tile of one KV head and walks all its query heads. Where few CTAs wait for the heaviest one, the
// group's heads are dealt out to several CTAs, whose parts of dK and dV go to slots of their own. The number is the divisor of G
// (every (key, query head) keeps one writer of dM) with the shortest estimate, in 64-row steps: the heaviest CTA's walk of
// 2 G Tr / n and kCtaSteps of fixed cost (prologue, write-out of dK and dV, its slot's pass through memory); with more CTAs than
// SMs also the work per SM and one more fixed cost for the uneven end. Fitted to 62 shapes of 1 to 64 tiles, 16 to 256 CTAs and
// groups of 2 to 16 heads, each timed with every divisor: within 7 % of the best one everywhere. us with one / the rule's / every
// divisor that leaves under 296 CTAs room: 2 x 1000 rows, 16 / 4 heads, d = 64 73 / 39 / 39, 8 x 512 rows, 16 / 4 heads, d = 128
// 73 / 78 / 101, 32 x 128 rows 45 / 45 / 92, 2048 rows, 32 / 8 heads 192 / 131 / 156.
constexpr int kMostSplitCtas = 384;        // (no shape gained from more; the slots' space is bounded by it)
int tc_bwd_splits(const Prob& P) {
    if (P.flags & DMA_FLAG_COMPACT_KV) return 1;
    if (P.bwd_split) return P.bwd_split;
    constexpr double kCtaSteps = 7.0, kSms = 148.0;
    const double ctas = (double)P.B * P.Hkv * P.Tc;
    auto steps = [&](int n) {
        const double heaviest = kCtaSteps + 2.0 * P.Tr * P.G / n;
        return ctas * n <= kSms ? heaviest : std::max(heaviest, ctas * (kCtaSteps * n + (P.Tr + 1.0) * P.G) / kSms + kCtaSteps);
    };
    int best = 1;
    for (int n = 2; n <= P.G && ctas * n <= kMostSplitCtas; ++n)
        if (P.G % n == 0 && steps(n) < steps(best)) best = n;
    return best;
}
// Tile mode without a split: from 256 64-row steps per SM on (about 0.36 ms) the instance that knows of no split and leaves the wait for
// its predecessor to the stream. Both only precede the main loop but cost it 2 %, while an overlapped launch saves 2 us: 16384 rows,
// 32 / 8 heads, backward at full clocks 4.95 -> 4.88 ms, over 20 calls at the power cap 5.56 -> 5.48 (4.85 and 5.43 before either
// existed; the split's constant alone 4.90, 5.51). At 8192 rows of 16 heads (450 steps, 0.74 ms) runs differ by more than that.
bool bwd_long(const Prob& P) {
    return !(P.flags & DMA_FLAG_COMPACT_KV) && tc_bwd_splits(P) == 1 && (int64_t)P.B * P.Hq * P.Tc * (P.Tr + 1) >= 256 * 148;
}
// Token-compacted mode: the longest walk of one CTA, in 64-row steps. A long-lived key's tile is walked over all later rows, 2 L / 128 steps,
// which few heads cannot hide behind other tiles: then walks are cut into parts of about what an SM gets of the whole work (its share of
// the kept pairs, and half as much again that the tiles' walks cover beyond them), which are work items of their own. The later parts' sums
// go through blocks (WalkBlocks); with DMA_FLAG_DETERMINISTIC nothing is cut.
// Backward, us, whole walks / this rule and items by length: one head of 9663 keys (w = 1442) 233 / 60, 2 heads of 4728 (w = 1044) 117 /
// 47, 8 heads of 8192 (w = 1024) 240 / 183, 16 heads of 4096 (w = 1024) 202 / 157 (nothing cut, long walks first), 32 heads of 16384
// 2282 / 2060 (K and V gathered by eight warps). The blocks cost 1 to 3 us of that: with all parts on the accumulators 57, 45, 180. Cutting every
// walk above 0.8 of the share was slower where the longest exceeds it by little (16 heads, w = 2375 of 14353 keys).
static int bwd_walk(const Prob& P) {
    const int longest = 2 * P.Tr;
    if (P.flags & DMA_FLAG_DETERMINISTIC) return longest;
    const double w = P.w, pairs = P.causal ? w * (w + 1) / 2 + (P.L - w) * w : w * P.L;
    const double share = (P.causal ? 1.55 : 1.0) * bwd_heads(P) * pairs / (128.0 * 64.0) / 148.0;
    if (longest <= 1.3 * share) return longest;
    return std::max(std::max(16, (int)(0.8 * share)), (longest + kMostParts - 1) / kMostParts);
}

// copies of the dK, dV accumulators (0: the main kernel writes dK, dV itself)
static size_t bwd_slots(const Prob& P) {
    if (P.flags & DMA_FLAG_COMPACT_KV) return (P.flags & DMA_FLAG_DETERMINISTIC) ? (size_t)P.G : 1;
    return tc_bwd_splits(P) > 1 ? (size_t)tc_bwd_splits(P) : 0;
}

static size_t bwd_base_bytes(const Prob& P) { return kWsHeaderBytes + (bwd_rows64(P) + bwd_acc_floats(P)) * sizeof(float); }
// what the call uses beyond that
static size_t bwd_extra_bytes(const Prob& P) {
    const size_t perm = P.flags & DMA_FLAG_COMPACT_KV ? (bwd_perm_ints(P) + bwd_item_ints(P) + bwd_where_ints(P)) * sizeof(int) : 0;
    return perm + (2 * bwd_slots(P) * (size_t)P.B * P.L * P.Hkv * P.d + bwd_part_floats(P) + bwd_blocks(P) * 2 * 128 * P.d) * sizeof(float);
}

size_t tc_bwd_need(const Prob& P) { return bwd_base_bytes(P) + bwd_extra_bytes(P); }

// The slots of the split go away where a longer sequence or a larger batch has CTAs enough, but a workspace of that size serves
// the shorter ones too: the bound for all of them, n CTAs for each of B Hkv Tc key tiles with n <= G and n B Hkv Tc <=
// kMostSplitCtas.
size_t tc_bwd_ws_bytes(const Prob& P) {
    size_t extra = bwd_extra_bytes(P);
    if (P.G > 1 && (!(P.flags & DMA_FLAG_COMPACT_KV) || P.chose_compact)) {
        const size_t ctas = std::min((size_t)P.B * P.Hq * P.Tc, (size_t)kMostSplitCtas);
        extra = std::max(extra, 2 * ctas * 128 * P.d * sizeof(float));
    }
    return bwd_base_bytes(P) + extra;
}

int launch_tc_bwd(const Prob& P, const void* Q, const void* K, const void* V, const void* O, const void* dO,
                  const float* lse, const float* bias, const int32_t* expiry, const uint32_t* bitmap, void* dQ,
                  void* dK, void* dV, float* dM, void* ws, cudaStream_t st) {
    const bool compact = (P.flags & DMA_FLAG_COMPACT_KV) != 0;
    if (!P.causal && !compact) return DMA_ERR_UNSUPPORTED;
    if ((size_t)P.G * P.Tr * 2 > (size_t)kMaxSteps || P.G > 16 || P.Tr > 1024) return DMA_ERR_UNSUPPORTED;
    const size_t rows = (size_t)P.B * P.Hq * P.L, nkv = (size_t)P.B * P.L * P.Hkv * P.d;
    float* Dv = reinterpret_cast<float*>((char*)ws + kWsHeaderBytes);
    float* acc = Dv + bwd_rows64(P);
    int* perm = reinterpret_cast<int*>(acc + bwd_acc_floats(P));
    const size_t slots = bwd_slots(P);
    const int nsplit = tc_bwd_splits(P);
    int2* items = reinterpret_cast<int2*>(perm + bwd_perm_ints(P));
    const size_t where_ints = compact ? bwd_where_ints(P) : 0;
    int* where = reinterpret_cast<int*>(items) + bwd_item_ints(P);
    float* accK = reinterpret_cast<float*>(compact ? where + where_ints : perm);
    float* accV = accK + slots * nkv;
    WalkBlocks blocks;
    blocks.cap = bwd_blocks_per_head(P);
    blocks.direct = P.G > 2 ? kMostParts : 3 - P.G;
    blocks.m = accV + slots * nkv;
    blocks.kv = blocks.m + bwd_part_floats(P);
    CUtensorMap tmQ, tmK, tmV, tmG;
    int rc;
    if ((rc = make_tmap_bf16(&tmQ, Q, P.B, P.L, P.Hq, P.d, P.qs, 64))) return rc;
    if ((rc = make_tmap_bf16(&tmG, dO, P.B, P.L, P.Hq, P.d, P.os, 64))) return rc;
    if ((rc = make_tmap_bf16(&tmK, K, P.B, P.L, P.Hkv, P.d, P.ks, 128))) return rc;
    if ((rc = make_tmap_bf16(&tmV, V, P.B, P.L, P.Hkv, P.d, P.vs, 128))) return rc;
    PrepareParams pp;
    pp.O = (const __nv_bfloat16*)O; pp.dO = (const __nv_bfloat16*)dO; pp.Dv = Dv; pp.B = P.B; pp.L = P.L; pp.Hq = P.Hq;
    pp.os_b = P.os[0]; pp.os_l = P.os[1]; pp.os_h = P.os[2];
    pp.status = (int32_t*)ws;
    pp.zero[0] = acc; pp.zero_n[0] = (int64_t)bwd_acc_floats(P);
    pp.zero[1] = dM; pp.zero_n[1] = (int64_t)rows;                                       // two sums, over the halves of the query columns, are added per key
    pp.zero[2] = accK; pp.zero_n[2] = compact ? (int64_t)(2 * slots * nkv) : 0;
    const int walk = compact ? bwd_walk(P) : 1, max_items = compact ? P.Tc * ((2 * P.Tr + walk - 1) / walk) : P.Tc;
    blocks.where = compact && max_items > P.Tc ? where : nullptr;
    if (blocks.where) { pp.zero[2] = reinterpret_cast<float*>(where); pp.zero_n[2] += (int64_t)where_ints; }   // (the accumulators are behind it)
    const int threads = compact ? kPermThreads : 256, per_cta = threads / (P.d / 8) * kPrepareRows;
    const unsigned prep_ctas = (unsigned)((rows + per_cta - 1) / per_cta);
    for (int z = 0; z < 3; ++z) pp.zero_part[z] = ((pp.zero_n[z] >> 2) + prep_ctas - 1) / prep_ctas;
    pp.perm_ctas = compact ? P.B * P.Hq : 0;
    pp.cap = blocks.cap; pp.direct = blocks.direct;
    pp.expiry = expiry; pp.perm = perm; pp.items = items; pp.Tc = P.Tc; pp.causal = P.causal; pp.max_items = max_items; pp.walk = walk;
    // (of more rows than one scheduling group, below, the order of the permutation keeps the rows in use in L2)
    pp.longest_first = (double)P.B * P.Hq * P.L * P.d * 8 <= 160.0 * 1024 * 1024 ? 1 : 0;
    auto prepare = compact ? (P.d == 128 ? bwd_prepare_kernel<16, true> : bwd_prepare_kernel<8, true>)
                           : (P.d == 128 ? bwd_prepare_kernel<16, false> : bwd_prepare_kernel<8, false>);
    if ((rc = launch_overlapped(prepare, dim3(pp.perm_ctas + prep_ctas), dim3(threads), 0, st, 1, pp))) return rc;
    BwdParams bp;
    bp.lse = lse; bp.Dv = Dv; bp.bias = bias; bp.expiry = expiry; bp.bitmap = bitmap; bp.dQacc = acc; bp.Lblk = P.Tr * 8;
    bp.dK = (__nv_bfloat16*)dK; bp.dV = (__nv_bfloat16*)dV; bp.dM = dM; bp.status = (int32_t*)ws;
    bp.B = P.B; bp.Hq = P.Hq; bp.Hkv = P.Hkv; bp.G = P.G; bp.L = P.L; bp.Tr = P.Tr; bp.Tc = P.Tc; bp.Wd = P.Wd;
    bp.ignore_bitmap = (P.flags & DMA_FLAG_IGNORE_BITMAP) ? 1 : 0;
    {
        // CTA start order: all key tiles of a few (batch, KV head) entries before the next few, so that the
        // rows those CTAs stream (Q, dO) and add to (the fp32 dQ accumulator: 8 bytes per element and query head in all)
        // stay in L2 while they are in use. About 160 MB of such rows per group was the best of the orders measured at
        // L = 16384 with 32 / 8 heads (two KV heads per group: 1.3 % faster in a long run than all eight at once; one
        // KV head per group starts the heaviest CTAs of the last group too late).
        const int gx = compact ? P.B * P.Hq : P.B * P.Hkv * nsplit;
        int sg = gx;
        {
            const double per_entry = (double)(compact ? 1 : P.G / nsplit) * P.L * P.d * 8;     // token-compacted mode: an entry is one query head
            // (token-compacted mode, eight heads at L = 16384: 1.69 ms against 1.74 with four and 1.82 with sixteen, once the
            //  CTAs walk backwards; with the forward walk four at a time was the best, 1.77 against 1.88)
            int want = (int)(160.0 * 1024 * 1024 / per_entry);
            want = want < 1 ? 1 : want;
            for (sg = want < gx ? want : gx; gx % sg; --sg) {}
        }
        bp.sched_group = sg;
    }
    bp.scale = P.scale; bp.scale_log2 = P.scale * 1.4426950408889634f; bp.inv_scale = 1.0f / P.scale;
    bp.ks_b = P.ks[0]; bp.ks_l = P.ks[1]; bp.ks_h = P.ks[2]; bp.vs_b = P.vs[0]; bp.vs_l = P.vs[1]; bp.vs_h = P.vs[2];
    bp.perm = perm; bp.items = items; bp.blocks = blocks; bp.causal = P.causal; bp.Kg = (const __nv_bfloat16*)K; bp.Vg = (const __nv_bfloat16*)V;
    bp.dKacc = accK; bp.dVacc = accV; bp.acc_slot = slots > 1 ? (int64_t)nkv : 0; bp.nsplit = nsplit;
    const size_t smem = sizeof(SharedStorage) + 1024;
    const bool lng = bwd_long(P);
    auto kern = compact ? (P.d == 128 ? bwd_kernel<true, 128> : bwd_kernel<true, 64>)
                : lng   ? (P.d == 128 ? bwd_kernel<false, 128, true> : bwd_kernel<false, 64, true>)
                        : (P.d == 128 ? bwd_kernel<false, 128> : bwd_kernel<false, 64>);
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return DMA_ERR_CUDA;
    timing_mark(1, false, st);
    const dim3 grid(compact ? P.B * P.Hq : P.B * P.Hkv * nsplit, max_items);
    rc = lng ? launch_plain(kern, grid, dim3(kThreads), smem, st, tmQ, tmK, tmV, tmG, bp)
             : launch_overlapped(kern, grid, dim3(kThreads), smem, st, 1, tmQ, tmK, tmV, tmG, bp);
    timing_mark(1, true, st);
    if (rc) return rc;
    FinishParams f;
    f.dQacc = acc; f.acc[0] = accK; f.acc[1] = accV; f.dQ = (__nv_bfloat16*)dQ; f.out[0] = (__nv_bfloat16*)dK; f.out[1] = (__nv_bfloat16*)dV;
    f.L = P.L; f.Hq = P.Hq; f.Hkv = P.Hkv; f.Lblk = P.Tr * 8; f.nslots = (int)slots; f.nkv = (int64_t)nkv;
    f.q_rows16 = (uint32_t)((size_t)P.B * P.Hq * P.Tr * 8);
    const int per = 8 / (P.d / 32) * kFinishBlocks;                        // 16-row blocks per CTA
    f.q_blocks = (int)((f.q_rows16 + per - 1) / per);
    f.kv_blocks = (int)((nkv / 8 + 255) / 256);
    for (int t = 0; t < 3; ++t) { f.qs[t] = P.qs[t]; f.st[0][t] = P.ks[t]; f.st[1][t] = P.vs[t]; }
    f.scale = P.scale;
    f.blocks = blocks; f.dM = dM; f.rows = (int64_t)rows;
    const int m_blocks = blocks.where ? (int)((rows + 255) / 256) : 0;
    auto finish = blocks.where && P.G <= 2 ? (P.d == 128 ? bwd_finish_blocks_kernel<128> : bwd_finish_blocks_kernel<64>)
                                           : (P.d == 128 ? bwd_finish_kernel<128> : bwd_finish_kernel<64>);
    return launch_overlapped(finish, dim3(f.q_blocks + (slots ? 2 * f.kv_blocks : 0) + m_blocks), dim3(256), 0, st,
                             1, f);
}

}  // namespace dma
