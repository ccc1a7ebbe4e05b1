// Mask generation (Sec. 4.1): value projection + gating (Eq. delta_calc), exact per-row top-w selection in
// compact "expiry" form (Eq. mask_combine read per query row over the causally visible keys), and the
// (query tile, key tile) activity bitmap (the Judge test of Alg. 1 / Alg. 2).
//
// Kernels
//   delta_kernel        V read once (HBM-bound); z, softplus, exp in a fixed fp32 operation order
//   tree_block_kernel, expiry_search_kernel (longer heads: tree_merge_kernel, expiry_tree_kernel)
//                       selection as a rank tree: the passes of a merge sort of (delta bits, ~index) keys leave one bit per key and
//                       level, and a key's expiry (the w-th smallest index among the keys that beat it) is a walk of log2(L) steps.
//                       Heads of up to 1024 keys, and of up to 4096 where there are many: sort, walk and bitmap in the one block kernel
//                       (launch_mask_build has the rules)
//   bitmap_square_kernel, bitmap_kernel   per key tile: union of the query-tile intervals its keys are kept in
#include <algorithm>
#include <cmath>
#include <mutex>
#include <utility>
#include <type_traits>

#include "common.cuh"

namespace dma {
namespace {

constexpr int kChunk = 256;   // the sort pads a head to a multiple of this many keys

// ---- fixed-order fp32 routines: every step is one correctly rounded IEEE operation -----------------------

__device__ __forceinline__ float exp_fixed(float x) {
    x = fminf(fmaxf(x, -87.0f), 88.0f);
    const float magic = 12582912.0f;
    float t = __fmul_rn(x, 0x1.715476p+0f);
    float n = __fadd_rn(__fadd_rn(t, magic), -magic);
    float r = __fmaf_rn(n, -0x1.62e4p-1f, x);
    r = __fmaf_rn(n, -0x1.7f7d1cp-20f, r);
    float q = 0x1.a01a02p-13f;
    q = __fmaf_rn(q, r, 0x1.6c16c2p-10f);
    q = __fmaf_rn(q, r, 0x1.111112p-7f);
    q = __fmaf_rn(q, r, 0x1.555556p-5f);
    q = __fmaf_rn(q, r, 0x1.555556p-3f);
    q = __fmaf_rn(q, r, 0.5f);
    q = __fmaf_rn(q, r, 1.0f);
    q = __fmaf_rn(q, r, 1.0f);
    return __fmul_rn(q, __int_as_float(((int)n + 127) << 23));
}

__device__ __forceinline__ float log1p_fixed(float t) {
    float s = __fdiv_rn(t, __fadd_rn(2.0f, t));
    float u = __fmul_rn(s, s);
    float q = 0x1.111112p-4f;
    q = __fmaf_rn(q, u, 0x1.3b13b2p-4f);
    q = __fmaf_rn(q, u, 0x1.745d18p-4f);
    q = __fmaf_rn(q, u, 0x1.c71c72p-4f);
    q = __fmaf_rn(q, u, 0x1.24924ap-3f);
    q = __fmaf_rn(q, u, 0x1.99999ap-3f);
    q = __fmaf_rn(q, u, 0x1.555556p-2f);
    q = __fmaf_rn(q, u, 1.0f);
    return __fmul_rn(__fmul_rn(2.0f, s), q);
}

__device__ __forceinline__ float delta_fixed(float z, float a) {
    float sp = __fadd_rn(fmaxf(z, 0.0f), log1p_fixed(exp_fixed(-fabsf(z))));
    return exp_fixed(__fmul_rn(a, sp));
}

// eight consecutive channels of one value row as fp32
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
    float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) {
    uint4 a = *reinterpret_cast<const uint4*>(p);
    uint32_t u[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}

// eight consecutive channels of one value row, as loaded (converted to fp32 only when the chain runs)
struct Raw8f { float4 a, b; };
__device__ __forceinline__ Raw8f load_raw8(const float* p) { return {*reinterpret_cast<const float4*>(p), *reinterpret_cast<const float4*>(p + 4)}; }
__device__ __forceinline__ uint4 load_raw8(const __nv_bfloat16* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ void widen8(const Raw8f& r, float (&v)[8]) {
    v[0] = r.a.x; v[1] = r.a.y; v[2] = r.a.z; v[3] = r.a.w; v[4] = r.b.x; v[5] = r.b.y; v[6] = r.b.z; v[7] = r.b.w;
}
__device__ __forceinline__ void widen8(const uint4& a, float (&v)[8]) {
    const uint32_t u[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}
template <typename T> struct RawOf { using type = uint4; };
template <> struct RawOf<float> { using type = Raw8f; };

// Sum over the LPR lanes of a row group of NB per-lane partials (one per head of a block of NB heads), in the order of the
// xor butterfly (adjacent lanes first: a balanced pairwise tree over the row's 8-channel chunks). The first log2(NB) levels
// are "transposing": a lane keeps half of its values and hands the other half to its partner, so the block costs
// log2(NB) + ... shuffles in all instead of NB log2(LPR) (the additions are the same, and IEEE addition commutes, so the
// bits are those of the plain butterfly). On return p[0] of lane `sub` is the complete sum of head bitrev(sub mod NB) of
// the block (the same value in every lane of the group with those low bits).
template <int NB, int LPR>
__device__ __forceinline__ void block_reduce(float (&p)[NB], int sub) {
    int keep = NB >> 1;
#pragma unroll
    for (int m = 1; m < LPR; m <<= 1) {
        if (keep >= 1) {
            const bool up = (sub & m) != 0;
#pragma unroll
            for (int q = 0; q < NB / 2; ++q) {
                if (q < keep) {
                    const float stay = up ? p[q + keep] : p[q];
                    const float give = up ? p[q] : p[q + keep];
                    p[q] = __fadd_rn(stay, __shfl_xor_sync(0xffffffffu, give, m));
                }
            }
            keep >>= 1;
        } else {
            p[0] = __fadd_rn(p[0], __shfl_xor_sync(0xffffffffu, p[0], m));
        }
    }
}

// One CTA: tiles of kRows consecutive keys of one (batch, KV head), taken in turn with the other CTAs of that pair (grid-
// stride); writes delta for the G query heads of the group. A group of D/8 lanes owns a row: each lane forms the fma chain
// over its 8 channels, an xor butterfly adds adjacent partials pairwise (IEEE addition commutes, so every lane of the group
// holds the same sum). The kernel streams V once and is bound by that stream, so it is built around memory-level
// parallelism: a warp requests ALL value rows of its NEXT tile (kPass 16-byte loads per lane) before it runs the chains of
// the current one, W is staged once per CTA, and softplus / exp of tile t (one (row, head) pair per thread, from the z
// values in shared memory) overlap the chains of tile t + 1 (two z buffers, one barrier per tile).
// Three shapes (keys per tile, CTAs per SM): launch_delta.
template <typename T, int D, int kRows, int kCtas>
__global__ void __launch_bounds__(256, sizeof(T) == 2 ? kCtas : 1) delta_kernel(const T* __restrict__ V, const float* __restrict__ W,
                                                    const float* __restrict__ A, float* __restrict__ delta,
                                                    int L, int Hq, int G, int64_t vs_b, int64_t vs_l, int64_t vs_h,
                                                    int j_off, int64_t ld) {
    constexpr int LPR = D / 8;            // lanes per row
    constexpr int RPW = 32 / LPR;         // rows per warp and pass
    constexpr int kPass = kRows / (8 * RPW);
    using Raw = typename RawOf<T>::type;
    extern __shared__ float smem[];
    float* sW = smem;                     // [G][D]
    float* sOut = smem + G * D;           // [2][G][kRows]
    const int hk = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = lane % LPR, grp = lane / LPR;
    pdl_enter_restrict(V, W, A, delta);
    const int ntiles = (L - j_off + kRows - 1) / kRows;        // keys [j_off, L) of a row of ld entries
    const T* Vb = V + b * vs_b + hk * vs_h + sub * 8;
    auto request = [&](int tile, Raw (&raw)[kPass]) {
        const int j0 = j_off + tile * kRows;
#pragma unroll
        for (int t = 0; t < kPass; ++t) {
            const int j = j0 + warp * RPW + grp + t * 8 * RPW;
            if (tile < ntiles && j < L) raw[t] = load_raw8(Vb + (int64_t)j * vs_l);
            else raw[t] = Raw{};
        }
    };
    Raw cur[kPass], nxt[kPass];
    request(blockIdx.x, cur);
    // (a lane's eight weights in two halves, each next to the other lanes' same half: a group's 16-byte reads meet every bank once)
    for (int i = tid; i < G * D; i += 256) sW[i / D * D + (i >> 2 & 1) * (D / 2) + i % D / 8 * 4 + (i & 3)] = W[(size_t)hk * G * D + i];
    __syncthreads();
    int buf = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, buf ^= 1) {
        request(tile + gridDim.x, nxt);
        const int j0 = j_off + tile * kRows, rows = min(kRows, L - j0);
        float* z = sOut + buf * G * kRows;
        // heads in blocks of 4 (then 2, then 1): the chains of a block, then one transposing reduction per pass
        auto block = [&](int g0, auto nb_tag) {
            constexpr int NB = decltype(nb_tag)::value;
            float w[NB][8];
#pragma unroll
            for (int q = 0; q < NB; ++q) {
                const float4 wa = *reinterpret_cast<const float4*>(sW + (g0 + q) * D + sub * 4), wb = *reinterpret_cast<const float4*>(sW + (g0 + q) * D + D / 2 + sub * 4);
                w[q][0] = wa.x; w[q][1] = wa.y; w[q][2] = wa.z; w[q][3] = wa.w; w[q][4] = wb.x; w[q][5] = wb.y; w[q][6] = wb.z; w[q][7] = wb.w;
            }
            int mine = 0;                 // head of the block this lane ends up with: the low bits of sub, reversed
#pragma unroll
            for (int m = 1, t = NB >> 1; m < NB; m <<= 1, t >>= 1) mine |= (sub & m) ? t : 0;
#pragma unroll
            for (int t = 0; t < kPass; ++t) {
                if (warp * RPW + t * 8 * RPW >= rows) continue;      // (warp-uniform) a short range, e.g. the one appended key of a decoding step
                float v[8], p[NB];
                widen8(cur[t], v);
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    float a = 0.0f;
#pragma unroll
                    for (int c = 0; c < 8; ++c) a = __fmaf_rn(v[c], w[q][c], a);
                    p[q] = a;
                }
                block_reduce<NB, LPR>(p, sub);
                const int r = warp * RPW + grp + t * 8 * RPW;
                if (sub < NB && r < rows) z[(g0 + mine) * kRows + r] = p[0];
            }
        };
        int g0 = 0;
        for (; g0 + 4 <= G; g0 += 4) block(g0, std::integral_constant<int, 4>{});
        if (g0 + 2 <= G) { block(g0, std::integral_constant<int, 2>{}); g0 += 2; }
        if (g0 < G) block(g0, std::integral_constant<int, 1>{});
        __syncthreads();                  // z of this tile is complete (and the other buffer's readers of two tiles ago are long done)
        for (int i = tid; i < G * kRows; i += 256) {
            const int g = i / kRows, r = i % kRows;
            if (r < rows) delta[((size_t)b * Hq + hk * G + g) * ld + j0 + r] = delta_fixed(z[i], A[hk * G + g]);
        }
#pragma unroll
        for (int t = 0; t < kPass; ++t) cur[t] = nxt[t];
    }
}

// A few keys (the one that a decoding step appends): a group of D / 8 lanes per (key, head), every load of a step at once and no barrier, so that the kernel is one
// round trip to memory and the chain of its arithmetic. The chains and the butterfly add in the order of delta_kernel: the same bits. One key of 32 heads, a token of
// a captured loop of 16384 keys 11.7 -> 10.1 us.
constexpr int kFewKeys = 8;
template <typename T, int D>
__global__ void __launch_bounds__(128) delta_few_kernel(const T* __restrict__ V, const float* __restrict__ W, const float* __restrict__ A, float* __restrict__ delta,
                                                        int Hq, int G, int64_t vs_b, int64_t vs_l, int64_t vs_h, int j_off, int64_t ld) {
    constexpr int LPR = D / 8;
    const int h = (blockIdx.x * 128 + threadIdx.x) / LPR, sub = threadIdx.x % LPR, j = j_off + blockIdx.y, b = blockIdx.z;
    pdl_enter_restrict(V, W, A, delta);
    const int hc = min(h, Hq - 1);                                    // (idle groups repeat the last head: the shuffles take whole warps)
    float v[8], w[8];
    load8(V + b * vs_b + (int64_t)j * vs_l + hc / G * vs_h + sub * 8, v);
    load8(W + (size_t)hc * D + sub * 8, w);
    const float gate = A[hc];
    float p = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c) p = __fmaf_rn(v[c], w[c], p);
#pragma unroll
    for (int m = 1; m < LPR; m <<= 1) p = __fadd_rn(p, __shfl_xor_sync(0xffffffffu, p, m));
    if (sub == 0 && h < Hq) delta[((size_t)b * Hq + h) * ld + j] = delta_fixed(p, gate);
}

// Full sampling weights (Eq. delta_calc as stated: all Hkv*D channels of the value row feed every head's score, the
// linear layer of the App. A listing): z[h] = sum over KV heads hk of (v_hk . W[h, hk*D : (hk+1)*D]), the per-head dot
// products formed as in delta_kernel (8-channel fma chains, pairwise tree over adjacent chunks) and added over hk
// from left to right. One CTA owns kFullRows keys of one batch and all heads. A group of D/8 lanes owns two rows; it forms the
// chains of D/8 heads at a time and adds them with a transposing butterfly (at each step a lane keeps half of its
// values and hands the other half to its partner: the same additions as the plain butterfly, a quarter of the
// shuffles), after which lane `sub` holds the dot product of head bitrev(sub) and carries that head's running sum.
// kFullRows keys per CTA: 64, or 32 where 64 would leave SMs without a CTA (4096 keys, 16 heads, 512 channels: 15.5 -> 14.2 us when it was measured, with the weights' reads in conflict).
constexpr size_t kFullSmem = 200 * 1024;     // the most dynamic shared memory of a CTA

template <typename T, int D, int kFullRows>
__global__ void __launch_bounds__(256) delta_full_kernel(const T* __restrict__ V, const float* __restrict__ W,
                                                         const float* __restrict__ A, float* __restrict__ delta,
                                                         int L, int Hq, int Hkv, int64_t vs_b, int64_t vs_l,
                                                         int64_t vs_h, int j_off, int64_t ld) {
    constexpr int LPR = D / 8;            // lanes per row = heads per batch
    constexpr int RPW = 32 / LPR;         // row groups per warp
    constexpr int kPass = 16 * RPW;       // rows per pass of the CTA (two per lane group)
    static_assert(kFullRows % kPass == 0, "a pass stays inside the CTA's rows");
    extern __shared__ float smem[];
    const int C = Hkv * D, HqP = (Hq + LPR - 1) / LPR * LPR;
    float* sW = smem;                     // [HqP][C], rows beyond Hq zero
    float* sZ = smem + (size_t)HqP * C;   // [HqP][kFullRows]
    const int b = blockIdx.y, j0 = j_off + blockIdx.x * kFullRows;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = lane % LPR, grp = lane / LPR;
    int mine = 0;                         // the head (within a batch) this lane ends up with: sub, bit-reversed
#pragma unroll
    for (int m = 1, t = LPR >> 1; m < LPR; m <<= 1, t >>= 1) mine |= (sub & m) ? t : 0;
    pdl_enter_restrict(V, W, A, delta);
    // (a lane's eight weights in two halves, each next to the other lanes' same half: a group's 16-byte reads meet every bank once
    // instead of half of them twice. us: 4096 keys, 16 heads, 512 channels 9.3 -> 7.4, 16384 keys 27.2 -> 19.4, 16384 keys, 8 heads of 1024 channels 51.1 -> 35.4)
#pragma unroll 4
    for (int i = tid; i < HqP * C / 4; i += 256)
        reinterpret_cast<float4*>(sW)[i / (D / 4) * (D / 4) + (i & 1) * LPR + i % (D / 4) / 2] =
            i < Hq * C / 4 ? __ldg(reinterpret_cast<const float4*>(W) + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    __syncthreads();
    for (int r0 = 0; r0 < kFullRows; r0 += kPass) {
        int r[2];
        r[0] = r0 + warp * 2 * RPW + grp;
        r[1] = r[0] + RPW;
        for (int hk = 0; hk < Hkv; ++hk) {
            float v[2][8];
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                if (j0 + r[n] < L) {
                    load8(V + b * vs_b + (int64_t)(j0 + r[n]) * vs_l + hk * vs_h + sub * 8, v[n]);
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c) v[n][c] = 0.0f;
                }
            }
            for (int hb = 0; hb < HqP; hb += LPR) {
                float p[2][LPR];
#pragma unroll
                for (int q = 0; q < LPR; ++q) {
                    const float* wp = sW + (size_t)(hb + q) * C + hk * D + sub * 4;
                    const float4 wa = *reinterpret_cast<const float4*>(wp), wb = *reinterpret_cast<const float4*>(wp + D / 2);
                    const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
                    for (int n = 0; n < 2; ++n) {
                        float a = 0.0f;
#pragma unroll
                        for (int c = 0; c < 8; ++c) a = __fmaf_rn(v[n][c], w[c], a);
                        p[n][q] = a;
                    }
                }
#pragma unroll
                for (int m = 1, keep = LPR >> 1; m < LPR; m <<= 1, keep >>= 1) {
                    const bool up = (sub & m) != 0;
#pragma unroll
                    for (int n = 0; n < 2; ++n)
#pragma unroll
                        for (int q = 0; q < keep; ++q) {
                            const float stay = up ? p[n][q + keep] : p[n][q];
                            const float give = up ? p[n][q] : p[n][q + keep];
                            p[n][q] = __fadd_rn(stay, __shfl_xor_sync(0xffffffffu, give, m));
                        }
                }
                const int h = hb + mine;
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    float* z = sZ + h * kFullRows + r[n];
                    *z = hk == 0 ? p[n][0] : __fadd_rn(*z, p[n][0]);
                }
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < Hq * kFullRows; i += 256) {
        const int h = i / kFullRows, r = i % kFullRows;
        if (j0 + r < L) delta[((size_t)b * Hq + h) * ld + j0 + r] = delta_fixed(sZ[i], A[h]);
    }
}

// ---- selection --------------------------------------------------------------------------------------------
// Order: key a beats key b iff (delta_a, -a) > (delta_b, -b). delta > 0, so its bit pattern orders like the
// value and one unsigned 64-bit compare decides.
__device__ __forceinline__ unsigned long long sort_key(float dl, int j) {
    return ((unsigned long long)__float_as_uint(dl) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)j);
}

// this CTA's share of zeros (a later kernel of the stage ORs bits into the bitmap)
__device__ __forceinline__ void zero_share(uint32_t* p, int64_t n) {
    const int64_t cta = (int64_t)blockIdx.y * gridDim.x + blockIdx.x, ctas = (int64_t)gridDim.x * gridDim.y;
    for (int64_t i = n * cta / ctas + threadIdx.x; i < n * (cta + 1) / ctas; i += blockDim.x) p[i] = 0u;
}

// ---- selection as a rank tree -------------------------------------------------------------------------------
// expiry[j] is the w-th smallest INDEX among the keys that beat j, i.e. among the first r entries of the head's keys in
// descending order, r = rank of j. That is a quantile query on a prefix, answered by a tree over key indices: the node of an
// aligned block of 2^k indices stores, for the block's keys in descending order, one bit per key (lower / upper half of
// the block) with running counts. A query walks from the root to a leaf: with c = how many of the first r keys lie in the
// node and z of them in its lower half, the k-th smallest index is in the lower half iff k <= z. log2(L) steps of one
// 8-byte load each, for every key in parallel, whatever w.
// The tree is what a bottom-up merge sort leaves behind: merging the sorted lower and upper half of a block yields the
// block's sorted sequence, and "this output came from the upper half" is the node's bit. tree_block_kernel builds the
// levels up to 1024 or 4096 keys; one tree_merge_kernel launch per level does the rest (runs of R keys -> runs of 2R).
// Level l (0 = root) of head bh lives at lev[(bh * m + l) * W + position / 32]: x = ones of the node before this word,
// y = the bits. A trailing run shorter than R (L is not a power of two) merges with what exists; the nodes stay
// left-aligned, which is all a query needs (it never looks past the real keys).
constexpr int kMergeThreads = 256;
constexpr int kMergeOut = 1024;       // outputs per CTA of tree_merge_kernel (four per thread)
constexpr int kBlockKeys = 4096, kSmallBlock = 1024;      // keys one CTA of tree_block_kernel sorts in shared memory
constexpr int kBlockThreads = 512;

// Comparator of two keys: the larger one to x.
__device__ __forceinline__ void order_desc(unsigned long long& x, unsigned long long& y) {
    const bool swap = y > x;
    const unsigned long long t = swap ? y : x;
    y = swap ? x : y;
    x = t;
}

// kN consecutive outputs of the merge of two descending runs A (na keys) and B (nb keys), starting at output x.
// i = how many of the first x outputs come from A: the first i for which "A[i] goes before the last B taken" fails, found by quartering the
// range `steps` times (at least (log2 of the shorter run's length + 1) / 2, rounded up) without a branch. Then the kN largest of A[i ..]
// and B[x - i ..] are the pairwise larger ones of one list and the other reversed, and a bitonic network orders them: all loads are in
// flight together, where kN steps of a merge would wait for one another. Keys are distinct and non-zero; 0 stands for "run exhausted".
// Returns i. at(p): the key at position p of the array that holds both, A from pa on and B from pb on.
template <int kN, typename At>
__device__ __forceinline__ int merge_outputs(At&& at, int pa, int na, int pb, int nb, int x, int steps, unsigned long long (&out)[kN]) {
    int lo = max(0, x - nb), hi = min(x, na);
    for (int t = 0; t < steps; ++t) {
        const int len = hi - lo, m2 = lo + (len >> 1), m1 = lo + (len >> 2), m3 = m2 + ((hi - m2) >> 1);
        auto before = [&](int mid) {                                 // (an empty range probes A[0] against itself: false)
            const bool in = mid < hi;
            return at(in ? pa + mid : pa) > at(in ? pb + x - mid - 1 : pa);
        };
        const bool p1 = before(m1), p2 = before(m2), p3 = before(m3);
        lo = p3 ? m3 + 1 : p2 ? m2 + 1 : p1 ? m1 + 1 : lo;
        hi = !p1 ? min(m1, hi) : !p2 ? m2 : !p3 ? min(m3, hi) : hi;
    }
    unsigned long long b[kN];
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        out[u] = lo + u < na ? at(pa + lo + u) : 0ull;
        b[u] = x - lo + u < nb ? at(pb + x - lo + u) : 0ull;
    }
#pragma unroll
    for (int u = 0; u < kN; ++u) out[u] = out[u] > b[kN - 1 - u] ? out[u] : b[kN - 1 - u];
#pragma unroll
    for (int h = kN / 2; h; h >>= 1)
#pragma unroll
        for (int u = 0; u < kN; ++u)
            if (!(u & h)) order_desc(out[u], out[u + h]);
    return lo;
}
// Which of the keys lie in the upper half of their block of 2 R = 2 << bit keys (a key's low word is ~index; R a power of two, blocks aligned)
template <int kN>
__device__ __forceinline__ uint32_t upper_half(const unsigned long long (&key)[kN], int bit) {
    uint32_t prov = 0u;
#pragma unroll
    for (int u = 0; u < kN; ++u) prov |= ((~(uint32_t)key[u] >> bit) & 1u) << u;
    return prov;
}

// the 32-bit word of 32 / kN neighbouring threads' kN provenance bits each (valid in the lanes with lane % (32 / kN) == 0)
template <int kN>
__device__ __forceinline__ uint32_t gather_bits(uint32_t prov, int lane) {
    uint32_t wv = prov << (kN * (lane & (32 / kN - 1)));
#pragma unroll
    for (int m = 1; m < 32 / kN; m <<= 1) wv |= __shfl_xor_sync(0xffffffffu, wv, m);
    return wv;
}

// Place of key p in the block kernel's buffers: one 8-byte word is skipped after every 16, so that neighbouring threads, whose searches and
// outputs lie 4 or 8 keys apart, use different banks (16 heads of 4096 keys in blocks of 4096, all levels merged in shared memory: mask build 34 -> 30 us).
__host__ __device__ constexpr int padded(int p) { return p + (p >> 4); }

// ones among the first c entries (c >= 1) of the node that starts at position s of a level; word(q) is the level's word of position q
template <typename Word>
__device__ __forceinline__ int ones_of(Word&& word, int s, int c) {
    const int q = s + c - 1;                                     // last entry of the prefix
    const uint2 wd = word(q);
    const uint32_t upto = (2u << (q & 31)) - 1u, from = ~((1u << (s & 31)) - 1u);             // a node smaller than a word starts inside it
    return (int)wd.x + __popc(wd.y & upto & from);
}

// Expiry of the key j at rank r of its head; word(l, q) is the word of position q in level l (0: the root).
// kMode 2 (non-causal): every row sees every key, so the key is kept by all rows iff fewer than w keys beat it.
// kMode 1: sequences packed along the key axis (sequence s owns the keys cu[s] <= j < cu[s+1]). A key competes only with
// the keys of its own sequence [s0, s1): of the first r keys of the head, n0 have an index below s0 (a first walk, along
// the path of s0, adds up the lower halves it leaves to its left), so the w-th beater inside the sequence is the
// (n0 + w)-th smallest index overall, if that exists and lies below s1; otherwise the key lives to the end of its sequence.
template <int kMode, typename Word>
__device__ __forceinline__ int expiry_of(Word&& word, int r, int j, int L, int w, int m, const int32_t* cu, int nseq) {
    int s0 = 0, s1 = L, k = w;
    if (kMode == 1) {
        int lo = 0, hi = nseq;                                   // largest s with cu[s] <= j
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (cu[mid] <= j) lo = mid; else hi = mid;
        }
        s0 = max(cu[lo], 0);
        s1 = min(cu[lo + 1], L);
        if (r >= w && s0 > 0) {
            int c = r, s = 0, n0 = 0;
            for (int l = 0; l < m && c > 0; ++l) {
                const int half = 1 << (m - 1 - l);
                const int ones = ones_of([&](int q) { return word(l, q); }, s, c);
                if (s0 & half) { n0 += c - ones; c = ones; s += half; } else { c -= ones; }
            }
            k = w + n0;
        }
    }
    if (r < k) return s1;                                        // fewer than w keys beat it (inside its sequence): never dropped
    if (kMode == 2) return 0;
    int c = r, s = 0;                                            // k-th smallest among the first c entries of the node starting at s
    for (int l = 0; l < m; ++l) {
        const int half = 1 << (m - 1 - l);
        const int ones = ones_of([&](int q) { return word(l, q); }, s, c), zeros = c - ones;
        if (k <= zeros) c = zeros; else { k -= zeros; c = ones; s += half; }
    }
    return (kMode == 1 && s >= s1) ? s1 : max(j, s);
}

// Bitmap words of square tiles (bm = bn): all keys of key tile kt that any row keeps enter in query tile kt (non-causal: 0), so the union of
// their intervals ends with the latest expiry of the tile, `last` (0: no key kept).
__device__ __forceinline__ uint32_t bitmap_word(const int* last, int kt0, int n, int qt, int bm, int causal) {
    uint32_t word = 0u;
    for (int k = 0; k < n; ++k) word |= (qt >= (causal ? kt0 + k : 0) && qt * bm < last[k]) ? 1u << k : 0u;
    return word;
}

// All levels with nodes of up to kBlock keys in one launch, a CTA per block of kBlock keys. A thread takes kPer consecutive keys; the
// levels inside a thread and inside a warp (up to 32 kPer keys) are bitonic merges in registers and by shuffles, the wider runs are merged
// in shared memory, kPer consecutive outputs per thread. A node's bit is a bit of the key's index, and the count of ones before a word is,
// in shared memory, the word's position minus the A keys taken so far. Padding keys (beyond L) sort below every real key (delta > 0)
// and keep their index in the low word.
// kMode >= 0: the head is one block (Lc = its padded length <= kBlock) and the CTA goes on from the tree in shared memory: expiry (the modes of
// expiry_of) and, with Tr > 0 (square tiles, at most 32), the bitmap. Otherwise sorted keys and levels go to global memory.
// 1024 keys are bound by latency, each level a chain of probes or shuffles (7.7 us); 4096 on one SM by its integer pipe (issue slots 57 %
// busy, 20 us), which is why few heads take blocks of 1024 (launch_mask_build).
template <int kBlock, int kMode>
__global__ void __launch_bounds__(kBlockThreads) tree_block_kernel(const float* __restrict__ delta, unsigned long long* __restrict__ sorted,
                                                                   uint2* __restrict__ lev, int L, int Lc, int m, int32_t* __restrict__ expiry,
                                                                   uint32_t* __restrict__ bitmap, int w, const int32_t* __restrict__ cu, int nseq,
                                                                   int bm, int Tr, int causal, int64_t zero_words, int* __restrict__ idx) {
    constexpr int kPer = kBlock > 2048 ? 8 : 4, kWarpKeys = 32 * kPer, kWarpBit = kPer == 8 ? 8 : 7;
    static_assert(kWarpKeys == 1 << kWarpBit && kPer * kBlockThreads >= kBlock, "a thread's keys, a warp's keys");
    constexpr int kWords = kBlock / 32;
    extern __shared__ __align__(16) unsigned long long sk[];         // two buffers of keys; kMode >= 0: the levels
    __shared__ int last[32];
    const int bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = blockIdx.x * kBlock, nreal = min(kBlock, Lc - base);
    const size_t Wl = (size_t)Lc / 32;
    unsigned long long* cur = sk;
    unsigned long long* nxt = sk + padded(kBlock);
    uint2* slev = reinterpret_cast<uint2*>(sk + 2 * padded(kBlock)); // [level][kWords]
    pdl_enter_restrict(delta, sorted, lev, expiry, bitmap, cu, idx);
    if (zero_words) zero_share(bitmap, zero_words);
    // the word of position p of the block in the level of nodes of 2 << bit keys
    auto put_word = [&](int bit, int p, uint32_t before, uint32_t bits) {
        if (kMode >= 0) slev[(m - 1 - bit) * kWords + (p >> 5)] = make_uint2(before, bits);
        else lev[((size_t)bh * m + (m - 1 - bit)) * Wl + ((base + p) >> 5)] = make_uint2(before, bits);
    };
    constexpr int kPerWord = 32 / kPer;                              // threads per word of a level
    const int o = kPer * tid;                                        // this thread's keys, and its outputs of every level: o .. o + kPer - 1 of the block
    const bool exists = o < nreal;                                   // (all of a warp's or none: nreal is a multiple of 256)
    unsigned long long key[kPer];
    if (exists) {
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int j = base + o + u;
            key[u] = j < L ? sort_key(delta[(size_t)bh * L + j], j) : (unsigned long long)(0xFFFFFFFFu - (unsigned)j);
        }
        // a level in order in the warp's registers: the bits, and per word the ones of its node before it
        auto emit = [&](int bit) {
            const uint32_t wv = gather_bits<kPer>(upper_half(key, bit), lane);
            const int words = max(1, (2 << bit) / 32), word = (lane / kPerWord) & (words - 1), ones = __popc(wv);
            int upto = ones;
            for (int d = 1; d < words; d <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, upto, d * kPerWord);
                if (word >= d) upto += y;
            }
            if (lane % kPerWord == 0) put_word(bit, o, (uint32_t)(upto - ones), wv);
        };
#pragma unroll
        for (int h = 1; h < kPer; h *= 2) {                          // in the thread: runs of h keys, the second one reversed against the first
#pragma unroll
            for (int g = 0; g < kPer; g += 2 * h) {
#pragma unroll
                for (int u = 0; u < h; ++u) order_desc(key[g + u], key[g + 2 * h - 1 - u]);
#pragma unroll
                for (int d = h / 2; d; d >>= 1)
#pragma unroll
                    for (int u = 0; u < 2 * h; ++u)
                        if (!(u & d)) order_desc(key[g + u], key[g + u + d]);
            }
            emit(h == 1 ? 0 : h == 2 ? 1 : 2);
        }
#pragma unroll
        for (int t = 0; t < 5; ++t) {                                // in the warp: runs of kPer << t keys
#pragma unroll
            for (int d = t; d >= 0; --d) {
                // first the second run reversed against the first, then the distances of 2^(t-1) .. 1 threads
                const int mask = d == t ? (2 << t) - 1 : 1 << d;
                const bool upper = (lane >> d) & 1;
                unsigned long long y[kPer];
#pragma unroll
                for (int u = 0; u < kPer; ++u) y[u] = __shfl_xor_sync(0xffffffffu, key[d == t ? kPer - 1 - u : u], mask);
#pragma unroll
                for (int u = 0; u < kPer; ++u) key[u] = (key[u] > y[u]) != upper ? key[u] : y[u];
            }
#pragma unroll
            for (int d = kPer / 2; d; d >>= 1)
#pragma unroll
                for (int u = 0; u < kPer; ++u)
                    if (!(u & d)) order_desc(key[u], key[u + d]);
            emit(kWarpBit - 5 + t);
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) cur[padded(o) + u] = key[u];
    }
    __syncthreads();
    for (int bit = kWarpBit; (1 << bit) < kBlock && (1 << bit) < Lc; ++bit) {        // wider runs, of R = 1 << bit keys
        const int R = 1 << bit, pair = o & ~(2 * R - 1), x = o - pair;
        const int na = max(0, min(R, nreal - pair)), nb = max(0, min(R, nreal - pair - R));
        int i0 = 0;
        if (exists) {
            i0 = merge_outputs<kPer>([&](int p) { return cur[padded(p)]; }, pair, na, pair + R, nb, x, bit / 2 + 1, key);
#pragma unroll
            for (int u = 0; u < kPer; ++u) nxt[padded(o) + u] = key[u];
        }
        const uint32_t wv = gather_bits<kPer>(exists ? upper_half(key, bit) : 0u, lane);
        if (lane % kPerWord == 0 && exists) put_word(bit, o, (uint32_t)(x - i0), wv);
        unsigned long long* tmp = cur; cur = nxt; nxt = tmp;
        __syncthreads();
    }
    if constexpr (kMode < 0) {
        for (int i = tid; i < nreal; i += kBlockThreads) {
            const unsigned long long k = cur[padded(i)];
            if (idx) {                                               // for expiry_search_kernel: delta bits and key numbers apart
                reinterpret_cast<uint32_t*>(sorted)[(size_t)bh * Lc + base + i] = (uint32_t)(k >> 32);
                idx[(size_t)bh * Lc + base + i] = (int)(0xFFFFFFFFu - (uint32_t)k);
            } else {
                sorted[(size_t)bh * Lc + base + i] = k;
            }
        }
    } else {
        int* sexp = reinterpret_cast<int*>(nxt);
        for (int r = tid; r < L; r += kBlockThreads) {
            const int j = (int)(0xFFFFFFFFu - (uint32_t)cur[padded(r)]);
            sexp[j] = expiry_of<kMode>([&](int l, int q) { return slev[l * kWords + (q >> 5)]; }, r, j, L, w, m, cu, nseq);
        }
        __syncthreads();
        if (Tr > 0) {                                                // a warp per key tile
            for (int kt = warp; kt < Tr; kt += kBlockThreads / 32) {
                int top = 0;
                for (int j = kt * bm + lane; j < min(L, kt * bm + bm); j += 32) {
                    const int e = sexp[j];
                    expiry[(size_t)bh * L + j] = e;
                    top = max(top, e > (causal ? j : 0) ? e : 0);
                }
                top = __reduce_max_sync(0xffffffffu, top);
                if (lane == 0) last[kt] = top;
            }
            __syncthreads();
            if (tid < Tr) bitmap[(size_t)bh * Tr + tid] = bitmap_word(last, 0, Tr, tid, bm, causal);
        } else {
            for (int j = tid; j < L; j += kBlockThreads) expiry[(size_t)bh * L + j] = sexp[j];
        }
    }
}

// Shared memory of tree_block_kernel
constexpr size_t block_smem(int keys, bool whole) { return 2 * (size_t)padded(keys) * sizeof(unsigned long long) + (whole ? 12 * (keys / 32) * sizeof(uint2) : 0); }

// One level per launch for runs of R >= 1024 keys: a CTA produces 1024 consecutive outputs of one pair of runs. Warp 0
// finds where they start in the two runs (32 probes per round), the CTA stages up to 1024 keys of each run in shared
// memory, and every thread merges four outputs from there.
__global__ void __launch_bounds__(kMergeThreads) tree_merge_kernel(const unsigned long long* __restrict__ src,
                                                                   unsigned long long* __restrict__ dst,
                                                                   uint2* __restrict__ lev_l, int Lc, int R, int m) {
    __shared__ __align__(16) unsigned long long sAB[2 * kMergeOut];       // A | B
    __shared__ int s_a0;
    pdl_enter_restrict(src, dst, lev_l);
    const int bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int o0 = blockIdx.x * kMergeOut;                       // first output position of this CTA within the head
    const int base = o0 & ~(2 * R - 1), t0 = o0 - base;
    const int na = min(R, Lc - base), nb = max(0, min(R, Lc - base - R));
    const unsigned long long* A = src + (size_t)bh * Lc + base;
    const unsigned long long* Bv = A + R;
    if (warp == 0) {
        int lo = max(0, t0 - nb), hi = min(t0, na);
        while (lo < hi) {
            const int len = hi - lo, stride = (len + 31) / 32;
            const int i = lo + lane * stride;
            const bool pr = i < hi && A[i] > Bv[t0 - i - 1];      // (i < hi implies i < na and t0 - i > 0)
            const int cnt = __popc(__ballot_sync(0xffffffffu, pr));
            if (cnt == 0) { hi = lo; break; }
            const int last_true = lo + (cnt - 1) * stride;
            lo = last_true + 1;
            hi = min(hi, last_true + stride);
        }
        if (lane == 0) s_a0 = lo;
    }
    __syncthreads();
    const int a0 = s_a0, b0 = t0 - a0;
    const int la = min(kMergeOut, na - a0), lb = min(kMergeOut, nb - b0);
#pragma unroll
    for (int k = 0; k < kMergeOut / kMergeThreads; ++k) {
        const int i = tid + k * kMergeThreads;
        sAB[i] = i < la ? A[a0 + i] : 0ull;
        sAB[kMergeOut + i] = i < lb ? Bv[b0 + i] : 0ull;
    }
    __syncthreads();
    const int x = 4 * tid;
    const bool exists = t0 + x < na + nb;
    unsigned long long out[4];
    const int i0 = merge_outputs<4>([&](int p) { return sAB[p]; }, 0, la, kMergeOut, lb, x, 6, out);      // (staged runs of up to 1024 keys)
    const uint32_t prov = upper_half(out, 31 - __clz(R));
    if (exists) {
        unsigned long long* d = dst + (size_t)bh * Lc + o0 + x;
        *reinterpret_cast<ulonglong2*>(d) = make_ulonglong2(out[0], out[1]);
        *reinterpret_cast<ulonglong2*>(d + 2) = make_ulonglong2(out[2], out[3]);
    }
    const uint32_t wv = gather_bits<4>(exists ? prov : 0u, lane);
    if ((lane & 7) == 0 && exists) lev_l[(size_t)bh * m * (Lc / 32) + ((o0 + x) >> 5)] = make_uint2((uint32_t)(b0 + x - i0), wv);
}

// One thread per rank r of a head: the key at rank r, the walk down the tree, expiry[j] = max(j, index found).
template <int kMode>
__global__ void __launch_bounds__(256) expiry_tree_kernel(const unsigned long long* __restrict__ sorted, const uint2* __restrict__ lev,
                                                          int32_t* __restrict__ expiry, int L, int Lc, int w, int m,
                                                          const int32_t* __restrict__ cu, int nseq) {
    const int r = blockIdx.x * 256 + threadIdx.x, bh = blockIdx.y;
    pdl_enter_restrict(sorted, lev, expiry, cu);
    if (r >= L) return;                                          // ranks from L on are padding
    const int j = (int)(0xFFFFFFFFu - (uint32_t)sorted[(size_t)bh * Lc + r]);
    const size_t W = (size_t)Lc / 32;
    const uint2* lv = lev + (size_t)bh * m * W;
    expiry[(size_t)bh * L + j] = expiry_of<kMode>([&](int l, int q) { return lv[l * W + (q >> 5)]; }, r, j, L, w, m, cu, nseq);
}

// Heads of up to kSearchKeys keys: no levels above the blocks. A key's beaters are counted block by block: in its own block they are the entries before it, in any other
// a binary search over the block's sorted delta bits, which the CTA holds in shared memory with the whole head's. (Equal bits beat it in blocks of lower
// indices.) The block in which the running count reaches w holds the key's expiry, found by the walk down that block's own tree. A CTA takes the keys of one block, in
// descending order, so that a warp's 32 searches read the same few words, and since a block's keys are whole key tiles, it writes their bits of the bitmap, too.
// This replaces a merge launch per level, the walk from the root and the bitmap kernel, each a chain of dependent loads after a launch. Bound by the latency
// of its own chain and, from 16 blocks on, by the searches ((blocks - 1) log2(block) reads per key). Mask build, us, merged / searched (G = 4, 64 channels): 16 heads of 4096 keys 23.9 / 15.8,
// 16 of 8192 28.7 / 18.8, 32 of 16384 55 / 43, of 32768 101 / 94, 128 of 16384 184 / 163, 8 of 6000 28.1 / 16.8; packed documents 28.3 / 19.3, 32.8 / 22.5, 65.5 / 56, 121 / 122 (launch_mask_build).
// (With the walk in global memory, a key after the other, 17.9, 27.0, 52.3, 114, 213.)
constexpr int kSearchKeys = 32768;
constexpr int kSearchThreads = 1024;
// c[u]: how many entries of the sorted (descending) block of kBlock entries at A[u] lie above than[u]
template <int kBlock, int kPer>
__device__ __forceinline__ void count_above(const uint32_t* (&A)[kPer], const uint32_t (&than)[kPer], int (&c)[kPer]) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) c[u] = 0;
#pragma unroll
    for (int s = kBlock / 2; s; s >>= 1)
#pragma unroll
        for (int u = 0; u < kPer; ++u) c[u] += A[u][c[u] + s - 1] > than[u] ? s : 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) c[u] += A[u][c[u]] > than[u] ? 1 : 0;
}

template <int kBlock, int kMode>
__global__ void __launch_bounds__(kSearchThreads) expiry_search_kernel(const uint32_t* __restrict__ vals, const int* __restrict__ idx, const uint2* __restrict__ lev,
                                                                       int32_t* __restrict__ expiry, uint32_t* __restrict__ bitmap, int L, int Lc, int w, int m,
                                                                       const int32_t* __restrict__ cu, int nseq, int bm, int T, int Wd, int causal) {
    constexpr int kPer = kBlock / kSearchThreads, kBits = kBlock == 4096 ? 12 : 10;
    static_assert(kBlock == 1 << kBits && kPer >= 1, "block sizes of the sort");
    extern __shared__ __align__(16) uint32_t sv[];                   // the head's sorted blocks, [nb][kBlock], zeros beyond its keys; expiry of the CTA's block; `last`
    const int nb = gridDim.x, a = blockIdx.x, bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, base = a * kBlock;
    int* sexp = reinterpret_cast<int*>(sv + nb * kBlock);
    int* last = sexp + kBlock;                                       // [kBlock / 32]
    pdl_enter_restrict(vals, idx, lev, expiry, bitmap, cu);
    int key[kPer];                                                   // the keys of ranks tid, tid + 1024, ... of the block
#pragma unroll
    for (int u = 0; u < kPer; ++u) key[u] = base + u * kSearchThreads + tid < Lc ? idx[(size_t)bh * Lc + base + u * kSearchThreads + tid] : L;
    for (int i = 4 * tid; i < nb * kBlock; i += 4 * kSearchThreads)
        *reinterpret_cast<uint4*>(sv + i) = i < Lc ? *reinterpret_cast<const uint4*>(vals + (size_t)bh * Lc + i) : make_uint4(0u, 0u, 0u, 0u);
    const int Wl = Lc / 32, Wt = nb * kBlock / 32;
    uint2* tree = reinterpret_cast<uint2*>(sv);                      // [kBits][Wt], once the searches are over
    // ones of the first c entries of the node that starts at s, l levels below its block
    auto ones_at = [&](const uint2* level, int s, int c) { return ones_of([&](int q) { return level[q >> 5]; }, s, c); };
    int s0[kPer], s1[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        s0[u] = 0;
        s1[u] = L;
        if (kMode == 1 && key[u] < L) {
            int lo = 0, hi = nseq;                                   // largest s with cu[s] <= j
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (cu[mid] <= key[u]) lo = mid; else hi = mid;
            }
            s0[u] = min(max(cu[lo], 0), L - 1);
            s1[u] = min(cu[lo + 1], L);
        }
    }
    __syncthreads();
    uint32_t v[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) v[u] = sv[base + u * kSearchThreads + tid];
    // Packed sequences: of the beaters in the block in which the key's sequence starts, those of earlier sequences, the ones along the path of s0
    int before[kPer];
    if constexpr (kMode == 1) {
        int c[kPer];
        const uint32_t* A[kPer];
        uint32_t than[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            A[u] = sv + s0[u] / kBlock * kBlock;
            than[u] = v[u] - (s0[u] / kBlock < a ? 1u : 0u);
        }
        count_above<kBlock, kPer>(A, than, c);
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            before[u] = 0;
            if (s0[u] / kBlock == a) c[u] = u * kSearchThreads + tid;
            if (s0[u] % kBlock == 0) c[u] = 0;
        }
        const uint2* level = lev + ((size_t)bh * m + (m - kBits)) * Wl;
        for (int l = 0; l < kBits; ++l, level += Wl) {
            const int half = kBlock >> (l + 1);
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                if (c[u] == 0) continue;
                const int ones = ones_at(level, s0[u] & ~(2 * half - 1), c[u]);
                if (s0[u] & half) { before[u] += c[u] - ones; c[u] = ones; } else { c[u] -= ones; }
            }
        }
    }
    int seen[kPer], s[kPer], c[kPer], k[kPer];                       // beaters in the blocks so far (of the key's sequence); the block of the w-th, its beaters there, which of them
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        seen[u] = c[u] = k[u] = 0;
        s[u] = -1;
    }
    for (int b = 0; b < nb; ++b) {
        int cb[kPer];
        if (b == a) {
#pragma unroll
            for (int u = 0; u < kPer; ++u) cb[u] = u * kSearchThreads + tid;
        } else {
            const uint32_t less = b < a ? 1u : 0u;                   // equal bits of a lower index count: those above v - 1
            const uint32_t* A[kPer];
            uint32_t than[kPer];
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                A[u] = sv + b * kBlock;
                than[u] = v[u] - less;
            }
            count_above<kBlock, kPer>(A, than, cb);
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            int early = 0;
            if (kMode == 1) early = (b + 1) * kBlock <= s0[u] ? cb[u] : b * kBlock <= s0[u] ? before[u] : 0;
            if (key[u] < L && s[u] < 0 && seen[u] + cb[u] - early >= w) {       // (padding takes no walk: its rank may lie beyond the block's entries)
                s[u] = b * kBlock;
                c[u] = cb[u];
                k[u] = w - seen[u] + early;
            }
            seen[u] += cb[u] - early;
        }
    }
    if constexpr (kMode != 2) {
        // the blocks' trees take the place of their keys
        __syncthreads();
        const uint2* lv = lev + ((size_t)bh * m + (m - kBits)) * Wl;
        for (int i = 2 * tid; i < kBits * Wl; i += 2 * kSearchThreads) {
            const int l = i / Wl, q = i % Wl;
            *reinterpret_cast<uint4*>(tree + l * Wt + q) = *reinterpret_cast<const uint4*>(lv + i);
        }
        __syncthreads();
        const uint2* level = tree;
        for (int l = 0; l < kBits; ++l, level += Wt) {               // k-th smallest among the first c entries of the node starting at s
#pragma unroll
            for (int u = 0; u < kPer; ++u) {
                if (s[u] < 0) continue;
                const int ones = ones_at(level, s[u], c[u]), zeros = c[u] - ones;
                if (k[u] <= zeros) c[u] = zeros; else { k[u] -= zeros; c[u] = ones; s[u] += kBlock >> (l + 1); }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int j = key[u];
        if (j >= L) continue;
        // (s < 0: fewer than w keys beat it inside its sequence: never dropped)
        const int e = s[u] < 0 ? s1[u] : kMode == 2 ? 0 : (kMode == 1 && s[u] >= s1[u]) ? s1[u] : max(j, s[u]);
        sexp[j - base] = e;
    }
    __syncthreads();
    for (int j = base + tid; j < min(L, base + kBlock); j += kSearchThreads) expiry[(size_t)bh * L + j] = sexp[j - base];
    if (bm > 0) {                                                    // square tiles, a multiple of eight of them per block
        const int n = kBlock / bm, kt0 = base / bm;
        for (int kt = warp; kt < n; kt += kSearchThreads / 32) {
            int top = 0;
            for (int j = kt * bm + lane; j < min(L - base, kt * bm + bm); j += 32) top = max(top, sexp[j] > (causal ? base + j : 0) ? sexp[j] : 0);
            top = __reduce_max_sync(0xffffffffu, top);
            if (lane == 0) last[kt] = top;
        }
        __syncthreads();
        // (the last block's CTA writes the rest of the row's words, too)
        const int bytes = n / 8, all = a == nb - 1 ? Wd * 4 - kt0 / 8 : min(bytes, Wd * 4 - kt0 / 8);
        uint8_t* out = reinterpret_cast<uint8_t*>(bitmap) + (size_t)bh * T * Wd * 4 + kt0 / 8;
        for (int i = tid; i < T * all; i += kSearchThreads) {
            const int qt = i / all, g = i % all;
            out[(size_t)qt * Wd * 4 + g] = g < bytes ? (uint8_t)bitmap_word(last + 8 * g, kt0 + 8 * g, 8, qt, bm, causal) : (uint8_t)0;
        }
    }
}
constexpr size_t search_smem(int nb, int block) { return ((size_t)nb * block + block + block / 32) * 4; }

__global__ void fill_i32_kernel(int32_t* p, size_t n, int32_t v, uint32_t* bitmap, int64_t bitmap_words) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_enter_restrict(p, bitmap);
    if (bitmap_words) zero_share(bitmap, bitmap_words);
    if (i < n) p[i] = v;
}

// Square tiles of a multiple of 32 rows: one CTA per (word of 32 key tiles, head), a warp per key tile finds the latest expiry, then a thread per
// query tile forms its word: no atomics, and the bitmap needs no zeros. A difference array per key tile and
// atomics into the bitmap took 7.8 us for 32 heads of 16384 keys.
__global__ void __launch_bounds__(1024) bitmap_square_kernel(const int32_t* __restrict__ expiry, uint32_t* __restrict__ bitmap,
                                                             int L, int bm, int T, int Wd, int causal) {
    __shared__ int last[32];
    const int kt0 = blockIdx.x * 32, bh = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_enter_restrict(expiry, bitmap);
    int top = 0;
    // (a tile side may be anything: neither a tile beyond the last nor the end of one is formed, they need not fit 32 bits)
    const int j0 = kt0 + warp < T ? (kt0 + warp) * bm : L, jend = bm < L - j0 ? j0 + bm : L;
    for (int j = j0 + lane; j < jend; j += 32) {
        const int e = expiry[(size_t)bh * L + j];
        top = max(top, e > (causal ? j : 0) ? e : 0);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) last[warp] = top;
    __syncthreads();
    for (int qt = threadIdx.x; qt < T; qt += 1024)
        bitmap[((size_t)bh * T + qt) * Wd + blockIdx.x] = bitmap_word(last, kt0, min(32, T - kt0), qt, bm, causal);
}

// Any other tiles. One CTA per (key tile, head): key j is kept by rows [j, expiry[j]), i.e. by query tiles j/bm .. (expiry[j]-1)/bm.
// A difference array over query tiles forms the union; bits are OR-ed into the (pre-zeroed) bitmap.
// (non-causal mode: key j is kept by rows [0, expiry[j]), so its interval of query tiles starts at tile 0)
__global__ void __launch_bounds__(128) bitmap_kernel(const int32_t* __restrict__ expiry, uint32_t* __restrict__ bitmap,
                                                     int L, int bm, int bn, int Tr, int Wd, int causal) {
    extern __shared__ int diff[];                 // [Tr + 1]
    const int kt = blockIdx.x, bh = blockIdx.y, t = threadIdx.x;
    pdl_enter_restrict(expiry, bitmap);
    for (int i = t; i <= Tr; i += blockDim.x) diff[i] = 0;
    __syncthreads();
    const int jend = min(L, (kt + 1) * bn);
    for (int j = kt * bn + t; j < jend; j += blockDim.x) {
        const int e = expiry[(size_t)bh * L + j];
        if (e > (causal ? j : 0)) {
            atomicAdd(&diff[causal ? j / bm : 0], 1);
            atomicAdd(&diff[(e - 1) / bm + 1], -1);
        }
    }
    __syncthreads();
    {   // running sum over the query tiles: each thread owns a contiguous segment, the segment totals are scanned by warp shuffles
        __shared__ int wtot[4];
        const int seg = (Tr + 127) / 128, q0 = t * seg, q1 = min(Tr, q0 + seg);
        int tot = 0;
        for (int q = q0; q < q1; ++q) tot += diff[q];
        int incl = tot;
        const int lane = t & 31, warp = t >> 5;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        int run = incl - tot;
        for (int k = 0; k < warp; ++k) run += wtot[k];
        for (int q = q0; q < q1; ++q) { run += diff[q]; diff[q] = run > 0; }
    }
    __syncthreads();
    for (int q = t; q < Tr; q += blockDim.x)
        if (diff[q]) atomicOr(&bitmap[((size_t)bh * Tr + q) * Wd + (kt >> 5)], 1u << (kt & 31));
}

}  // namespace

constexpr int kStaticChunk = kChunk;

// levels of the rank tree over a head of Lc (a multiple of 256) keys: the smallest m with 2^m >= Lc
static int tree_levels(int Lc) {
    int m = 8;
    while ((1ll << m) < Lc) ++m;
    return m;
}

// workspace: header | two buffers of sort keys (8 bytes per padded key each: the merge passes alternate between them) |
// the rank tree (m levels of 8 bytes per 32 padded keys)
size_t mask_ws_bytes(const Prob& P) {
    const size_t nchunk = (P.L + kChunk - 1) / kChunk, keys = (size_t)P.B * P.Hq * nchunk * kChunk;
    return kWsHeaderBytes + keys * 2 * sizeof(unsigned long long) + keys / 32 * tree_levels((int)(nchunk * kChunk)) * sizeof(uint2);
}

template <typename T, int D>
static int launch_delta(const Prob& P, const void* V, const float* W, const float* A, float* bias, cudaStream_t st,
                        int j_begin = 0, int j_end = -1, int64_t ld = -1) {
    if (j_end < 0) j_end = P.L;
    if (ld < 0) ld = P.L;
    if (j_end <= j_begin) return DMA_OK;
    if (P.flags & DMA_FLAG_FULL_DELTA) {
        const size_t HqP = (size_t)(P.Hq + D / 8 - 1) / (D / 8) * (D / 8);
        if ((HqP * P.Hkv * D + HqP * 64) * sizeof(float) > kFullSmem) return DMA_ERR_UNSUPPORTED;
        constexpr int kFewRows = D == 128 ? 32 : 64;          // (one pass of the CTA covers 32 rows at d = 128, 64 at d = 64)
        const int rows = (int64_t)P.B * ((j_end - j_begin + 63) / 64) < 148 ? kFewRows : 64;
        const size_t bytes = (HqP * P.Hkv * D + HqP * rows) * sizeof(float);
        auto kern = rows == 64 ? delta_full_kernel<T, D, 64> : delta_full_kernel<T, D, kFewRows>;
        // (state of the function, which other threads' calls share: always the limit)
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFullSmem) != cudaSuccess) return DMA_ERR_CUDA;
        return launch_overlapped(kern, dim3((j_end - j_begin + rows - 1) / rows, P.B), dim3(256), bytes, st, 1, (const T*)V, W, A, bias, j_end, P.Hq, P.Hkv,
                                 P.vs[0], P.vs[1], P.vs[2], j_begin, ld);
    }
    const size_t smem = (size_t)P.G * (D + 2 * 128) * sizeof(float);
    if (smem > 48 * 1024) return DMA_ERR_UNSUPPORTED;
    if (j_end - j_begin <= kFewKeys)
        return launch_overlapped(delta_few_kernel<T, D>, dim3((P.Hq * (D / 8) + 127) / 128, j_end - j_begin, P.B), dim3(128), 0, st, 1, (const T*)V, W, A, bias, P.Hq, P.G,
                                 P.vs[0], P.vs[1], P.vs[2], j_begin, ld);
    // Two CTAs per SM in all (what the register file holds at once), each walking its (batch, KV head) pair's tiles of 128 keys grid-stride. us, tiles of 128 / the other shape:
    // Tiles of 64 keys where a CTA then walks at most three quarters of the keys and all CTAs run at once: 8 heads of 500 keys 3.3 / 2.6, 4 of 12000 6.2 / 5.2, 32 / 8 heads of 6000 8.7 / 7.2, but 16 heads of
    // 1500 (192 CTAs either way) 3.9 / 4.1, 32 / 8 heads of 8192 8.8 / 9.0, 8 of 16384 with 64 channels (448 keys against 512) 6.1 / 6.7.
    // Tiles of 32 and four CTAs per SM, where a KV head has one query head, whose tiles are short work, and tiles of 128 take more than one wave of CTAs: 16 heads of 8192 keys 12.8 / 9.5, of 65536 91 / 60,
    // 32 of 6000 18.0 / 17.3, 64 of 16384 87.9 / 85.1, but 8 heads (one wave) of 65536 30.2 / 32.3, 128 of 8192 75 / 85. With 64 channels only where they are one wave: 16 heads of 4096 keys 5.1 / 4.7, but 32
    // of 16384 24.5 / 30.4, 128 85 / 147.
    const int64_t pairs = (int64_t)P.Hkv * P.B;
    const int keys = j_end - j_begin;
    auto grid = [&](int rows, int ctas) { return (int)std::min<int64_t>((ctas * 148 + pairs - 1) / pairs, (keys + rows - 1) / rows); };      // CTAs per pair
    auto walk = [&](int rows) { return ((keys + rows - 1) / rows + grid(rows, 2) - 1) / grid(rows, 2) * rows; };                             // keys of a CTA
    auto launch = [&](auto kern, int rows, int ctas) {
        const size_t bytes = (size_t)P.G * (D + 2 * rows) * sizeof(float);
        return launch_overlapped(kern, dim3(grid(rows, ctas), P.Hkv, P.B), dim3(256), bytes, st, 1, (const T*)V, W, A, bias, j_end, P.Hq, P.G, P.vs[0], P.vs[1], P.vs[2], j_begin, ld);
    };
    if (pairs * grid(64, 2) <= 2 * 148 && 4 * walk(64) <= 3 * walk(128)) return launch(delta_kernel<T, D, 64, 2>, 64, 2);
    if (sizeof(T) == 2 && P.G == 1 && pairs * grid(128, 2) > 2 * 148 && (D == 128 ? pairs <= 64 : pairs * grid(32, 4) <= 4 * 148))
        return launch(delta_kernel<T, D, 32, 4>, 32, 4);
    return launch(delta_kernel<T, D, 128, 2>, 128, 2);
}

// delta for the keys [j_begin, j_end) only, into rows of ld entries (a decoding cache that grows)
int launch_delta_range(const Prob& P, const void* V, const float* W, const float* A, float* delta, int64_t ld, int j_begin,
                       int j_end, cudaStream_t st) {
    if (P.dtype == DMA_BF16)
        return P.d == 128 ? launch_delta<__nv_bfloat16, 128>(P, V, W, A, delta, st, j_begin, j_end, ld)
                          : launch_delta<__nv_bfloat16, 64>(P, V, W, A, delta, st, j_begin, j_end, ld);
    return P.d == 128 ? launch_delta<float, 128>(P, V, W, A, delta, st, j_begin, j_end, ld)
                      : launch_delta<float, 64>(P, V, W, A, delta, st, j_begin, j_end, ld);
}

// size limits of the stage's kernels (shared-memory footprints), checked before anything is enqueued
static int mask_build_limits(const Prob& P) {
    if (P.flags & DMA_FLAG_FULL_DELTA) {
        const size_t lanes = (size_t)P.d / 8, HqP = (P.Hq + lanes - 1) / lanes * lanes;
        if ((HqP * P.Hkv * P.d + HqP * 64) * sizeof(float) > kFullSmem) return DMA_ERR_UNSUPPORTED;
    } else if ((size_t)P.G * (P.d + 2 * 128) * sizeof(float) > 48 * 1024) {
        return DMA_ERR_UNSUPPORTED;
    }
    if ((size_t)(P.Tr + 1) * sizeof(int) > 48 * 1024) return DMA_ERR_UNSUPPORTED;
    return DMA_OK;
}

int launch_mask_build(const Prob& P, const void* V, const float* W, const float* A, float* bias, int32_t* expiry,
                      uint32_t* bitmap, void* ws, cudaStream_t st, const int32_t* cu, int nseq) {
    int rc;
    if ((rc = mask_build_limits(P))) return rc;          // an error return means that no kernel has been launched
    if (P.dtype == DMA_BF16)
        rc = P.d == 128 ? launch_delta<__nv_bfloat16, 128>(P, V, W, A, bias, st)
                        : launch_delta<__nv_bfloat16, 64>(P, V, W, A, bias, st);
    else
        rc = P.d == 128 ? launch_delta<float, 128>(P, V, W, A, bias, st) : launch_delta<float, 64>(P, V, W, A, bias, st);
    if (rc) return rc;

    const int BH = P.B * P.Hq;
    const int nchunk = (P.L + kChunk - 1) / kChunk;
    // (the general bitmap kernel ORs bits into zeros that an earlier kernel of the stage leaves)
    const bool square = P.bm == P.bn && P.bm % 32 == 0;
    const int64_t zero_words = square ? 0 : (int64_t)BH * P.Tr * P.Wd;
    if (P.w >= P.L && !cu) {   // every visible key is kept
        size_t n = (size_t)BH * P.L;
        rc = launch_overlapped(fill_i32_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st, 1, expiry, n, P.L, bitmap, zero_words);
        if (rc) return rc;
    } else {
        // rank tree: sorted blocks, then a search over the blocks and a walk in one of them per key (heads beyond kSearchKeys: one merge pass per further level and a
        // walk from the root); or everything in the block kernel. Blocks of 4096 keys keep few SMs busy for long where there are few, and blocks of 1024 take more
        // searches: blocks of 1024 / a head whole in one CTA, mask build, us: 8 heads of 2000 keys 14.3 / 16.9, 16 of 3000 16.0 / 23.5, 64 of 3000 25.3 / 27.7,
        // but 128 of 2000 24.2 / 21.3, 128 of 3000 36.8 / 32.6
        const int Lc = nchunk * kChunk, m = tree_levels(Lc);
        const int64_t small_blocks = (int64_t)BH * ((Lc + kSmallBlock - 1) / kSmallBlock);
        const bool few = small_blocks <= 2 * 148, whole = Lc <= (!few ? kBlockKeys : small_blocks > 200 ? 2 * kSmallBlock : kSmallBlock);
        bool small = few, search = !whole && Lc <= kSearchKeys;
        if (search && Lc > kBlockKeys) {
            // Estimates, us: with blocks of 1024 the SMs' share of the blocks by the searches of each; with 4096, whose trees leave an SM one CTA, waves of CTAs; packed sequences, which walk twice, also
            // against blocks of 4096 and merge launches. Fitted to 1 to 256 heads of 4097 to 32768 keys, 73 shapes, where they choose the best within 0.2 % in the mean. Mask build, us, 1024 /
            // 4096: 16 heads of 8192 keys 19 / 34, 32 of 9000 31 / 39, 64 of 4097 35 / 38, 64 of 9000 56 / 70, 128 of 4097 54 / 68, but 8 of 32768 54 / 48, 48 of 8192 40 / 38, 32 of 16384 63 / 43, 128 of 16384
            // 216 / 163; packed, 1024 / 4096 / merged: 64 of 9000 67 / 91 / 86, 128 of 4097 66 / 95 / 78, 32 of 16384 75 / 57 / 65, 64 of 32768 417 / 251 / 239, 8 of 32768 64 / 62 / 54.
            const double blocks = (Lc + kSmallBlock - 1) / kSmallBlock, large = (Lc + kBlockKeys - 1) / kBlockKeys, share = BH * blocks / 148.0;
            const double ctas = BH * large / 148.0, waves = ctas > 3.0 ? ctas : std::ceil(ctas);       // (behind three waves their ends have drifted apart)
            const double by_small = cu ? 12.0 + share * (9.2 + 0.6 * blocks) : P.causal ? 10.0 + share * (7.4 + 0.52 * blocks) : 9.0 + share * (6.8 + 0.45 * blocks);
            const double by_large = waves * (cu ? 45.0 + 2.6 * large : P.causal ? 29.4 + 2.33 * large : 24.3 + 2.16 * large);
            const double merged = 2.0 + 28.0 * std::ceil(BH * large / 296.0) + 3.4 * (m - 12) + share * (7.7 + 1.2 * (m - 12));
            small = by_small < by_large;
            if (cu && merged < std::min(by_small, by_large)) small = search = false;
        }
        const int per_block = whole ? (Lc <= kSmallBlock ? kSmallBlock : kBlockKeys) : small ? kSmallBlock : kBlockKeys;
        const bool fused_bitmap = whole && square && P.Tr <= 32;
        const size_t keys = (size_t)BH * Lc, Wl = (size_t)Lc / 32;
        auto* buf0 = reinterpret_cast<unsigned long long*>((char*)ws + kWsHeaderBytes);
        auto* buf1 = buf0 + keys;
        uint2* lev = reinterpret_cast<uint2*>(buf1 + keys);
        int* idx = search ? reinterpret_cast<int*>(buf1) : nullptr;
        const int mode = !whole ? -1 : cu ? 1 : P.causal ? 0 : 2;
        auto pick = [&](auto n) {
            constexpr int kN = decltype(n)::value;
            return mode < 0 ? tree_block_kernel<kN, -1> : mode == 0 ? tree_block_kernel<kN, 0> : mode == 1 ? tree_block_kernel<kN, 1> : tree_block_kernel<kN, 2>;
        };
        auto block = per_block == kSmallBlock ? pick(std::integral_constant<int, kSmallBlock>{}) : pick(std::integral_constant<int, kBlockKeys>{});
        // (state of the function, which other threads' calls share: always the limit)
        if (cudaFuncSetAttribute(block, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)block_smem(kBlockKeys, true)) != cudaSuccess) return DMA_ERR_CUDA;
        rc = launch_overlapped(block, dim3((Lc + per_block - 1) / per_block, BH), dim3(kBlockThreads), block_smem(per_block, whole), st, 1, bias, buf0, lev, P.L, Lc, m,
                               expiry, fused_bitmap || zero_words ? bitmap : nullptr, P.w, cu, nseq, P.bm, fused_bitmap ? P.Tr : 0, P.causal, zero_words, idx);
        if (rc) return rc;
        if (fused_bitmap) return DMA_OK;
        if (search) {
            const int nb = (Lc + per_block - 1) / per_block;
            const bool bits = square && P.bm <= per_block / 8 && per_block % (8 * P.bm) == 0;
            auto pick_search = [&](auto n) {
                constexpr int kN = decltype(n)::value;
                return cu ? expiry_search_kernel<kN, 1> : P.causal ? expiry_search_kernel<kN, 0> : expiry_search_kernel<kN, 2>;
            };
            auto kern = per_block == kSmallBlock ? pick_search(std::integral_constant<int, kSmallBlock>{}) : pick_search(std::integral_constant<int, kBlockKeys>{});
            // (state of the function, which other threads' calls share: always the limit)
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)search_smem(kSearchKeys / kBlockKeys, kBlockKeys)) != cudaSuccess) return DMA_ERR_CUDA;
            rc = launch_overlapped(kern, dim3(nb, BH), dim3(kSearchThreads), search_smem(nb, per_block), st, 1, reinterpret_cast<const uint32_t*>(buf0), (const int*)idx, lev,
                                   expiry, bitmap, P.L, Lc, P.w, m, cu, nseq, bits ? P.bm : 0, P.Tr, P.Wd, P.causal);
            if (rc || bits) return rc;
        }
        int l = m - (per_block == kSmallBlock ? 11 : 13);         // level of the nodes of two blocks
        for (int R = per_block; !whole && !search && R < Lc; R *= 2, --l) {
            rc = launch_overlapped(tree_merge_kernel, dim3((Lc + kMergeOut - 1) / kMergeOut, BH), dim3(kMergeThreads), 0, st, 1, buf0, buf1, lev + (size_t)l * Wl, Lc, R, m);
            if (rc) return rc;
            std::swap(buf0, buf1);
        }
        if (!whole && !search) {
            const dim3 grid((P.L + 255) / 256, BH);
            rc = launch_overlapped(cu ? expiry_tree_kernel<1> : P.causal ? expiry_tree_kernel<0> : expiry_tree_kernel<2>, grid, dim3(256), 0, st, 1, buf0, lev,
                                   expiry, P.L, Lc, P.w, m, cu, nseq);
            if (rc) return rc;
        }
    }
    if (square) return launch_overlapped(bitmap_square_kernel, dim3(P.Wd, BH), dim3(1024), 0, st, 1, expiry, bitmap, P.L, P.bm, P.Tr, P.Wd, P.causal);
    return launch_overlapped(bitmap_kernel, dim3(P.Tc, BH), dim3(128), (size_t)(P.Tr + 1) * sizeof(int), st, 1, expiry, bitmap, P.L, P.bm, P.bn, P.Tr, P.Wd, P.causal);
}

}  // namespace dma

// ---------------------------------------------------------------------------------------------------------------
// dma_mask_build_static: mask generation for callers that cannot hand over a workspace.
// The selection's scratch (sort keys and rank tree) lives in this file-scope device array, which every GPU that loads the library keeps
// until the process exits. In host code the array's name is only a stand-in; its device address is looked up
// once per device with cudaGetSymbolAddress and that pointer is what the kernels receive.
// ---------------------------------------------------------------------------------------------------------------
namespace {
// 1 Mi padded keys: two buffers of sort keys (8 MiB each) and a rank tree of at most 20 levels (8 bytes per 32 keys and
// level: 5 MiB). B * Hq * roundup(L, 256) must not exceed this.
constexpr size_t kStaticKeys = 1u << 20;
static __device__ __align__(256) unsigned long long g_static_scratch[dma::kWsHeaderBytes / 8 + 2 * kStaticKeys + kStaticKeys / 32 * 20];
constexpr int kMaxDevices = 64;
void* g_static_ptr[kMaxDevices];            // per-device address of g_static_scratch (0 = not looked up yet)
std::mutex g_static_mutex;
}  // namespace

extern "C" int dma_mask_build_static(const dma_problem_t* p, const void* V, const float* W_delta, const float* A,
                                     float* bias, int32_t* expiry, uint32_t* bitmap, void* cuda_stream) {
    dma::Prob P;
    int rc = dma::resolve(p, &P);
    if (rc) return rc;
    if (!V || !W_delta || !A || !bias || !expiry || !bitmap) return DMA_ERR_NULL;
    const uintptr_t bits = (uintptr_t)V | (uintptr_t)W_delta | (uintptr_t)bias | (uintptr_t)expiry | (uintptr_t)bitmap;
    if (bits & 15) return DMA_ERR_ALIGN;
    const size_t keys = (size_t)P.B * P.Hq * ((P.L + dma::kStaticChunk - 1) / dma::kStaticChunk) * dma::kStaticChunk;
    if (keys > kStaticKeys) return DMA_ERR_WORKSPACE;          // larger problems must use dma_mask_build
    int dev = -1, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DMA_ERR_CUDA;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess || major != 10) return DMA_ERR_CUDA;
    void* scratch;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {       // first call on this device (which is current): resolve the symbol's address
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) return DMA_ERR_CUDA;
            g_static_ptr[dev] = ptr;
        }
        scratch = g_static_ptr[dev];
    }
    return dma::launch_mask_build(P, V, W_delta, A, bias, expiry, bitmap, scratch, (cudaStream_t)cuda_stream);
}
