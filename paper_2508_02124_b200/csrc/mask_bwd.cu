// Mask-generation backward (Sec. 4.3: the bias gradient dM flows on to the sampling weights W_delta and the gate A;
// Eq. delta_calc differentiated, the top-w selection held fixed):
//   z = v . W_h, sp = softplus(z), delta = exp(A_h sp)   (delta is taken from the forward's bias output)
//   g = dM delta;  dA_h = sum g sp;  dz = g A_h sigmoid(z);  dW_h = sum dz v;  dV[j, kv head] += sum_h dz W_h
// HBM-bound: V and dV rows are read once, dV written once. A CTA walks keys of one (batch, KV head) with all G query heads of
// the group; its dW / dA sums go to the workspace and a second kernel adds them in a fixed order (no floating-point atomics:
// the result does not depend on the launch schedule).
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace dma {
namespace {

constexpr int kRows = 8;       // keys per warp and unit
constexpr int kThreads = 256;
constexpr int kMaxGroup = 16;  // query heads per KV head

__device__ __forceinline__ void load8f(const float* p, float (&v)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8f(const __nv_bfloat16* p, float (&v)[8]) {
    const uint4 a = *reinterpret_cast<const uint4*>(p);
    const uint32_t u[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}
__device__ __forceinline__ void store8f(float* p, const float (&v)[8]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8f(__nv_bfloat16* p, const float (&v)[8]) {
    uint4 o;
    o.x = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[0])) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[1])) << 16);
    o.y = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[2])) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[3])) << 16);
    o.z = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[4])) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[5])) << 16);
    o.w = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[6])) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v[7])) << 16);
    *reinterpret_cast<uint4*>(p) = o;
}

// A warp takes units of eight consecutive keys of its (batch, KV head) pair, grid-stride; a group of D/8 lanes owns a row (8
// channels per lane). Nothing is shared between warps until the end, so there is no barrier in the loop: the next unit's value
// rows and dM, delta are requested before the current unit is worked on, z of four heads at a time goes through a transposing
// butterfly, softplus / sigmoid are evaluated once per (row, head) pair by one lane of the row's group, and the sums dW, dA stay
// in registers over all units (kG = G heads; kG = 0, any other G: in the warp's part of shared memory). Two CTAs per SM in all,
// one partial sum per CTA: at L = 16384, 32 / 8 heads, d = 128 (105 MB) 64 -> 28.9 us and the sum of the partials 13.4 -> 4.1
// us, against CTAs of 64 keys that each staged, synchronised and wrote partials.
// partial [CTAs of the pair][G][D + 1]: the sums over the CTA's keys of dz v (D values) and of g sp (1 value).
template <typename T> struct Row8;
template <> struct Row8<__nv_bfloat16> {
    uint4 a;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { a = *reinterpret_cast<const uint4*>(p); }
    __device__ __forceinline__ void clear() { a = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void get(float (&v)[8]) const {
        const uint32_t u[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) { v[2 * i] = __uint_as_float(u[i] << 16); v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u); }
    }
};
template <> struct Row8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float* p) { a = *reinterpret_cast<const float4*>(p); b = *reinterpret_cast<const float4*>(p + 4); }
    __device__ __forceinline__ void clear() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void get(float (&v)[8]) const { v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w; }
};

template <typename T, int D, int kG>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 2 ? 2 : 1) mask_bwd_kernel(const T* __restrict__ V, const float* __restrict__ W,
                                                            const float* __restrict__ A, const float* __restrict__ delta,
                                                            const float* __restrict__ dM, T* __restrict__ dV,
                                                            float* __restrict__ partial, int L, int Hq, int G_,
                                                            int64_t vs_b, int64_t vs_l, int64_t vs_h) {
    constexpr int LPR = D / 8;                       // lanes per row
    constexpr int RPW = 32 / LPR;                    // rows per warp instruction
    constexpr int NR = kRows / RPW;                  // rows per thread and unit
    const int G = kG ? kG : G_;
    constexpr int kPairs = kG ? (NR * kG + LPR - 1) / LPR : 1;      // (row, head) pairs per lane whose dM, delta are requested ahead
    extern __shared__ float smem[];
    float* sW = smem;                                // [G][D]
    float* sAcc = smem + G * D;                      // [8 warps][G][D + 1]
    const int hk = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = lane % LPR, grp = lane / LPR;
    float* myZ = sAcc + 8 * G * (D + 1) + (warp * RPW + grp) * 2 * NR * G;      // z, then dz, of the group's (row, head) pairs
    float* myGs = myZ + NR * G;                      // dM delta softplus(z)
    float* wAcc = sAcc + (size_t)warp * G * (D + 1);
    pdl_enter(V, W, A, delta, dM, dV, partial);
    // (a lane's eight weights in two halves, each next to the other lanes' same half: a group's 16-byte reads meet every bank once
    // instead of half of them twice: 26.9 -> 25.9 us at 16384 keys, 32 / 8 heads; one head per KV head 20.5 -> 20.7 at 8192 keys, 16 heads)
    for (int i = tid; i < G * D; i += kThreads) sW[i / D * D + (i >> 2 & 1) * (D / 2) + i % D / 8 * 4 + (i & 3)] = W[(size_t)hk * G * D + i];
    if (kG == 0)
        for (int i = lane; i < G * (D + 1); i += 32) wAcc[i] = 0.0f;
    __syncthreads();
    const T* Vb = V + b * vs_b + hk * vs_h + sub * 8;
    T* dVb = dV + b * vs_b + hk * vs_h + sub * 8;
    const size_t head0 = ((size_t)b * Hq + hk * G) * L;
    const int units = (L + kRows - 1) / kRows, stride = gridDim.x * 8;
    auto weights = [&](int g, float (&w)[8]) {
        const float4 lo = *reinterpret_cast<const float4*>(sW + g * D + sub * 4), hi = *reinterpret_cast<const float4*>(sW + g * D + D / 2 + sub * 4);
        w[0] = lo.x; w[1] = lo.y; w[2] = lo.z; w[3] = lo.w; w[4] = hi.x; w[5] = hi.y; w[6] = hi.z; w[7] = hi.w;
    };
    auto request = [&](int u, Row8<T> (&v)[NR], float (&gd)[kPairs]) {
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            const int j = u * kRows + n * RPW + grp;
            if (u < units && j < L) v[n].load(Vb + (int64_t)j * vs_l);
            else v[n].clear();
        }
        if constexpr (kG > 0) {
#pragma unroll
            for (int q = 0; q < kPairs; ++q) {
                const int pr = sub + q * LPR, j = u * kRows + pr / kG * RPW + grp;
                const bool in = pr < NR * kG && u < units && j < L;
                const size_t at = head0 + (size_t)(pr % kG) * L + j;
                gd[q] = in ? dM[at] * delta[at] : 0.0f;
            }
        }
    };
    float pw[kG ? kG : 1][8], ga[kPairs];
#pragma unroll
    for (int g = 0; g < (kG ? kG : 1); ++g)
#pragma unroll
        for (int c = 0; c < 8; ++c) pw[g][c] = 0.0f;
#pragma unroll
    for (int q = 0; q < kPairs; ++q) ga[q] = 0.0f;
    Row8<T> cur[NR], nxt[NR];
    float gd[kPairs], gdn[kPairs];
    int u = blockIdx.x * 8 + warp;
    request(u, cur, gd);
    for (; u < units; u += stride) {
        Row8<T> old[NR];                             // the dV rows to be updated
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            const int j = u * kRows + n * RPW + grp;
            if (j < L) old[n].load(dVb + (int64_t)j * vs_l);
        }
        request(u + stride, nxt, gdn);
        // z of the unit's (row, head) pairs: heads in blocks of 4 (then 2, then 1)
        auto block = [&](int g0, auto nb_tag) {
            constexpr int NB = decltype(nb_tag)::value;
            float w[NB][8];
#pragma unroll
            for (int q = 0; q < NB; ++q) weights(g0 + q, w[q]);
#pragma unroll
            for (int n = 0; n < NR; ++n) {
                float v[8], p[NB];
                cur[n].get(v);
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    p[q] = 0.0f;
#pragma unroll
                    for (int c = 0; c < 8; ++c) p[q] = fmaf(v[c], w[q][c], p[q]);
                }
#pragma unroll
                for (int m = 1, keep = NB >> 1; m < LPR; m <<= 1, keep >>= 1) {      // a lane keeps half of its heads per level, then plain sums
                    if (keep >= 1) {
                        const bool up = (sub & m) != 0;
#pragma unroll
                        for (int q = 0; q < NB / 2; ++q) {
                            if (q < keep) {
                                const float stay = up ? p[q + keep] : p[q], give = up ? p[q] : p[q + keep];
                                p[q] = stay + __shfl_xor_sync(0xffffffffu, give, m);
                            }
                        }
                    } else {
                        p[0] += __shfl_xor_sync(0xffffffffu, p[0], m);
                    }
                }
                int mine = 0;                        // the head of the block this lane ends up with
#pragma unroll
                for (int m = 1, t = NB >> 1; m < NB; m <<= 1, t >>= 1) mine |= (sub & m) ? t : 0;
                if (sub < NB) myZ[n * G + g0 + mine] = p[0];
            }
        };
        int g0 = 0;
        for (; g0 + 4 <= G; g0 += 4) block(g0, std::integral_constant<int, 4>{});
        if (g0 + 2 <= G) { block(g0, std::integral_constant<int, 2>{}); g0 += 2; }
        if (g0 < G) block(g0, std::integral_constant<int, 1>{});
        __syncwarp();
        auto pair_of = [&](int pr, float gdv) {      // dz to the row group's scratch; returns g softplus(z)
            const float z = myZ[pr], e = expf(-fabsf(z));            // e in (0, 1]
            myZ[pr] = gdv * A[hk * G + pr % G] * ((z >= 0.0f ? 1.0f : e) / (1.0f + e));
            return gdv * (fmaxf(z, 0.0f) + log1pf(e));
        };
        if constexpr (kG > 0) {
#pragma unroll
            for (int q = 0; q < kPairs; ++q)
                if (sub + q * LPR < NR * kG) ga[q] += pair_of(sub + q * LPR, gd[q]);       // (LPR is a multiple of kG: always head sub % kG)
        } else {
            for (int pr = sub; pr < NR * G; pr += LPR) {
                const int j = u * kRows + pr / G * RPW + grp;
                const size_t at = head0 + (size_t)(pr % G) * L + j;
                myGs[pr] = pair_of(pr, j < L ? dM[at] * delta[at] : 0.0f);
            }
        }
        __syncwarp();
        float upd[NR][8];
#pragma unroll
        for (int n = 0; n < NR; ++n)
#pragma unroll
            for (int c = 0; c < 8; ++c) upd[n][c] = 0.0f;
        auto head = [&](int g, float (&pg)[8]) {
            float w[8];
            weights(g, w);
#pragma unroll
            for (int n = 0; n < NR; ++n) {
                const float dz = myZ[n * G + g];
                float v[8];
                cur[n].get(v);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    pg[c] = fmaf(dz, v[c], pg[c]);
                    upd[n][c] = fmaf(dz, w[c], upd[n][c]);
                }
            }
        };
        if constexpr (kG > 0) {
#pragma unroll
            for (int g = 0; g < kG; ++g) head(g, pw[g]);
        } else {
            for (int g = 0; g < G; ++g) {
                float pg[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, pa = 0.0f;
                head(g, pg);
                if (sub == 0)
                    for (int n = 0; n < NR; ++n) pa += myGs[n * G + g];
#pragma unroll
                for (int m = LPR; m < 32; m <<= 1) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) pg[c] += __shfl_xor_sync(0xffffffffu, pg[c], m);
                    pa += __shfl_xor_sync(0xffffffffu, pa, m);
                }
                if (grp == 0) {
#pragma unroll
                    for (int c = 0; c < 8; ++c) wAcc[g * (D + 1) + sub * 8 + c] += pg[c];
                    if (sub == 0) wAcc[g * (D + 1) + D] += pa;
                }
            }
        }
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            const int j = u * kRows + n * RPW + grp;
            if (j < L) {
                float o[8];
                old[n].get(o);
#pragma unroll
                for (int c = 0; c < 8; ++c) o[c] += upd[n][c];
                store8f(dVb + (int64_t)j * vs_l, o);
            }
        }
        __syncwarp();                                // the scratch may be written again
#pragma unroll
        for (int n = 0; n < NR; ++n) cur[n] = nxt[n];
#pragma unroll
        for (int q = 0; q < kPairs; ++q) gd[q] = gdn[q];
    }
    if constexpr (kG > 0) {
        float pa = 0.0f;
#pragma unroll
        for (int q = 0; q < kPairs; ++q) pa += ga[q];
#pragma unroll
        for (int m = kG; m < 32; m <<= 1) pa += __shfl_xor_sync(0xffffffffu, pa, m);      // lanes of the same head: equal sub % kG
#pragma unroll
        for (int g = 0; g < kG; ++g) {
#pragma unroll
            for (int m = LPR; m < 32; m <<= 1)
#pragma unroll
                for (int c = 0; c < 8; ++c) pw[g][c] += __shfl_xor_sync(0xffffffffu, pw[g][c], m);
            if (grp == 0) {
#pragma unroll
                for (int c = 0; c < 8; ++c) wAcc[g * (D + 1) + sub * 8 + c] = pw[g][c];
            }
        }
        if (lane < kG) wAcc[lane * (D + 1) + D] = pa;
    }
    __syncthreads();
    const size_t blk = ((size_t)b * gridDim.y + hk) * gridDim.x + blockIdx.x;
    for (int i = tid; i < G * (D + 1); i += kThreads) {
        float t = 0.0f;
#pragma unroll
        for (int wq = 0; wq < 8; ++wq) t += sAcc[(size_t)wq * G * (D + 1) + i];
        partial[blk * G * (D + 1) + i] = t;
    }
}

// the sums of 16 groups, pair by pair
__device__ __forceinline__ float add_groups(const float (*part)[32], int lane) {
    float s[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) s[q] = part[q][lane];
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1)
#pragma unroll
        for (int q = 0; q < o; ++q) s[q] += s[q + o];
    return s[0];
}

// dW[h][c] and dA[h]: sum of the per-CTA partials over batches and key blocks. 16 groups of threads each add every 16th partial in index
// order, four requested at once, then the group sums are added: a fixed order, whatever the schedule. (A CTA of four or eight groups per head waited
// for one load after another: both kernels 11.2 -> 8.9 us at 4096 keys, 16 heads, 29.8 -> 28.6 at 16384, 32 heads.)
template <int D>
__global__ void __launch_bounds__(512) mask_bwd_reduce_kernel(const float* __restrict__ partial, float* __restrict__ dW, float* __restrict__ dA, int B,
                                                              int Hkv, int G, int nblk) {
    __shared__ float part[16][32];
    pdl_enter(partial, dW, dA);
    const int h = blockIdx.x, hk = h / G, g = h % G, lane = threadIdx.x & 31, c = blockIdx.y * 32 + lane, grp = threadIdx.x >> 5;
    const int total = B * nblk;
    float s = 0.0f;
    if (c <= D)
#pragma unroll 4
        for (int t = grp; t < total; t += 16) {
            const int b = t / nblk;
            s += partial[(((size_t)t + (size_t)(b * (Hkv - 1) + hk) * nblk) * G + g) * (D + 1) + c];
        }
    part[grp][lane] = s;
    __syncthreads();
    if (grp == 0 && c <= D) {
        const float tot = add_groups(part, lane);
        if (c < D) dW[(size_t)h * D + c] = tot; else dA[h] = tot;
    }
}

// ---- full sampling weights: W [Hq, C], C = Hkv * D channels of the value row feed every head ----------------
// One CTA owns R consecutive keys of one batch with their whole value rows in shared memory (fp32):
//   1  z, dz = dM delta A sigmoid(z) and gs = dM delta softplus(z) of a (head, row) per lane
//   2  dW partial [h][col] = sum_rows dz v: a thread owns columns and walks the rows (no cross-thread sums)
//   3  dV += sum_h dz W[h][col]: a thread owns columns of 16 rows
// partial [B * blocks][Hq][C + 1]; mask_bwd_full_reduce_kernel adds them in a fixed order.
// Bound by the loads from shared memory and by latency, not by HBM (8 MB and 0.2 G fmas for 4096 keys, 16 heads of 512 channels), so each step takes
// as many heads by rows (columns) per load as registers hold, all warps have a task, and dM, delta and dV are requested before the sums they meet. Both
// kernels, us, against two heads of all rows per warp, one column per thread and dV summed up in the value tile: 4096 keys, 16 heads, 512 channels 27.3 -> 17.0,
// 8192 38.6 -> 28.6, 4096 keys, 32 heads, 1024 channels 63.6 -> 49.0, 16384 278 -> 209. Half the threads, half the rows and two CTAs per SM: 18.9, 36.5, 58.7, 265.
constexpr size_t kFullSmem = 200 * 1024;    // the most dynamic shared memory of a CTA
constexpr int kFullThreads = 512;

template <typename T, int RW>
__global__ void __launch_bounds__(kFullThreads) mask_bwd_full_kernel(const T* __restrict__ V, const float* __restrict__ W,
                                                                 const float* __restrict__ A, const float* __restrict__ delta,
                                                                 const float* __restrict__ dM, T* __restrict__ dV,
                                                                 float* __restrict__ partial, int L, int Hq, int Hkv, int D,
                                                                 int64_t vs_b, int64_t vs_l, int64_t vs_h) {
    constexpr int R = RW * 8;
    extern __shared__ float smem[];
    const int C = Hkv * D, HqP = (Hq + 7) & ~7;
    float* sV = smem;                              // [R][C]
    float* sDz = sV + (size_t)R * C;               // [R][HqP], heads beyond Hq hold 0
    float* sZ = sDz + (size_t)R * HqP;             // [Hq][R]: dM delta softplus(z)
    const int b = blockIdx.y, j0 = blockIdx.x * R;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int C8 = C / 8, D8 = D / 8;
    pdl_enter(V, W, A, delta, dM, dV, partial);

    for (int i = tid; i < R * C8; i += kFullThreads) {
        const int row = i / C8, ch = i % C8, j = j0 + row;
        float v[8];
        if (j < L) {
            load8f(V + b * vs_b + (int64_t)j * vs_l + (ch / D8) * vs_h + (ch % D8) * 8, v);
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = 0.0f;
        }
        store8f(sV + (size_t)row * C + ch * 8, v);
    }
    for (int i = tid; i < R * HqP; i += kFullThreads) sDz[i] = 0.0f;
    __syncthreads();

    // z: a warp takes four heads and eight rows, lanes stride the channels: 12 loads feed 32 fmas, and the butterfly that adds the lanes'
    // sums (a lane keeps half of its accumulators at each step) leaves one (head, row) in each lane
    constexpr int RB = R / 8;
    for (int task = warp; task < (Hq + 3) / 4 * RB; task += kFullThreads / 32) {
        const int h0 = task / RB * 4, r0 = task % RB * 8;
        const int h = h0 + (lane >> 3), row = r0 + (lane & 7), j = j0 + row;
        const size_t at = ((size_t)b * Hq + h) * L + j;
        const bool in = h < Hq && j < L;
        const float gd = in ? dM[at] * delta[at] : 0.0f, ah = in ? A[h] : 0.0f;
        float acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
        const float* wr[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) wr[q] = W + (size_t)min(h0 + q, Hq - 1) * C;
#pragma unroll 4
        for (int col = lane; col < C; col += 32) {
            float w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = __ldg(wr[q] + col);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float v = sV[(size_t)(r0 + r) * C + col];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q * 8 + r] = fmaf(v, w[q], acc[q * 8 + r]);
            }
        }
#pragma unroll
        for (int keep = 16; keep >= 1; keep >>= 1) {
            const bool up = (lane & keep) != 0;
#pragma unroll
            for (int i = 0; i < keep; ++i) {
                const float stay = up ? acc[i + keep] : acc[i], give = up ? acc[i] : acc[i + keep];
                acc[i] = stay + __shfl_xor_sync(0xffffffffu, give, keep);
            }
        }
        if (h < Hq) {
            const float z = acc[0], e = expf(-fabsf(z));
            sZ[h * R + row] = in ? gd * (fmaxf(z, 0.0f) + log1pf(e)) : 0.0f;
            sDz[row * HqP + h] = in ? gd * ah * ((z >= 0.0f ? 1.0f : e) / (1.0f + e)) : 0.0f;
        }
    }
    __syncthreads();

    // dW: a thread owns two columns of eight heads (half a row apart, so that loads and stores are whole lines)
    float* out = partial + ((size_t)b * gridDim.x + blockIdx.x) * Hq * (C + 1);
    const int half = C / 2;
    for (int i = tid; i < half * (HqP / 8); i += kFullThreads) {
        const int hc = i / half * 8, col = i % half;
        float acc[8][2];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q][0] = acc[q][1] = 0.0f;
#pragma unroll 8
        for (int row = 0; row < R; ++row) {
            const float v0 = sV[(size_t)row * C + col], v1 = sV[(size_t)row * C + half + col];
            float a[8];
            *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(sDz + row * HqP + hc);
            *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(sDz + row * HqP + hc + 4);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                acc[q][0] = fmaf(a[q], v0, acc[q][0]);
                acc[q][1] = fmaf(a[q], v1, acc[q][1]);
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (hc + q < Hq) {
                out[(size_t)(hc + q) * (C + 1) + col] = acc[q][0];
                out[(size_t)(hc + q) * (C + 1) + half + col] = acc[q][1];
            }
    }
    for (int h = warp; h < Hq; h += kFullThreads / 32) {
        float s = 0.0f;
        for (int row = lane; row < R; row += 32) s += sZ[h * R + row];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[(size_t)h * (C + 1) + C] = s;
    }

    // dV: a thread owns two neighbouring columns of RT rows, whose values it requests before it adds up the heads
    constexpr int RT = R < 16 ? R : 16;
    using T2 = typename std::conditional<std::is_same<T, float>::value, float2, __nv_bfloat162>::type;
    for (int i = tid; i < half * (R / RT); i += kFullThreads) {
        const int r0 = i / half * RT, col = i % half * 2;
        T* p = dV + b * vs_b + (int64_t)(j0 + r0) * vs_l + (col / D) * vs_h + col % D;
        T2 cur[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r)
            if (j0 + r0 + r < L) cur[r] = *reinterpret_cast<const T2*>(p + r * vs_l);
        float u[RT][2];
#pragma unroll
        for (int r = 0; r < RT; ++r) u[r][0] = u[r][1] = 0.0f;
#pragma unroll 1
        for (int hc = 0; hc < HqP; hc += 4) {             // (unrolled it spills: 4096 keys 17.0 -> 18.1 us)
            float w[4][2];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float* wp = W + (size_t)min(hc + q, Hq - 1) * C + col;
                w[q][0] = __ldg(wp);
                w[q][1] = __ldg(wp + 1);
            }
            if (hc + 4 > Hq) {             // (heads beyond Hq have dz = 0, but the last head's weights may be infinite)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (hc + q >= Hq) w[q][0] = w[q][1] = 0.0f;
            }
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const float4 a = *reinterpret_cast<const float4*>(sDz + (r0 + r) * HqP + hc);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float s = a.x * w[0][c];
                    s = fmaf(a.y, w[1][c], s);
                    s = fmaf(a.z, w[2][c], s);
                    u[r][c] += fmaf(a.w, w[3][c], s);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            if (j0 + r0 + r >= L) break;
            if constexpr (std::is_same<T, float>::value) {
                *reinterpret_cast<float2*>(p + r * vs_l) = make_float2(cur[r].x + u[r][0], cur[r].y + u[r][1]);
            } else {
                const float2 f = __bfloat1622float2(cur[r]);
                *reinterpret_cast<__nv_bfloat162*>(p + r * vs_l) = __floats2bfloat162_rn(f.x + u[r][0], f.y + u[r][1]);
            }
        }
    }
}

// dW [Hq][C] and dA [Hq] from partial [n][Hq][C + 1]: 16 groups of threads each add every 16th partial in index order, eight requested
// at once, then the group sums are added.
__global__ void __launch_bounds__(512) mask_bwd_full_reduce_kernel(const float* __restrict__ partial, float* __restrict__ dW,
                                                                   float* __restrict__ dA, int n, int Hq, int C) {
    __shared__ float part[16][32];
    pdl_enter(partial, dW, dA);
    const int h = blockIdx.y, lane = threadIdx.x & 31, c = blockIdx.x * 32 + lane, grp = threadIdx.x >> 5;
    float s = 0.0f;
    if (c <= C)
#pragma unroll 8
        for (int t = grp; t < n; t += 16) s += partial[((size_t)t * Hq + h) * (C + 1) + c];
    part[grp][lane] = s;
    __syncthreads();
    if (grp == 0 && c <= C) {
        const float tot = add_groups(part, lane);
        if (c < C) dW[(size_t)h * C + c] = tot; else dA[h] = tot;
    }
}

static bool full_fits(const Prob& P, int R) {
    const size_t C = (size_t)P.Hkv * P.d, HqP = (P.Hq + 7) & ~7;
    return (R * C + R * HqP + (size_t)P.Hq * R) * sizeof(float) <= kFullSmem;
}
// rows per CTA: the largest of 64, 32, 16, 8 whose tile fits 200 KiB of shared memory (0: none does); 32 instead of 64 where
// twice the CTAs still run at once, one per SM (both kernels, us, 64 / 32 rows, 16 heads, 512 channels: 4096 keys 27.8 / 16.9, but
// 4800 keys, 75 CTAs, 28.2 / 30.0 and 8192 keys 28.1 / 31.1: two waves of half the length cost more than one).
static int full_rows(const Prob& P) {
    int R = 64;
    while (R >= 8 && !full_fits(P, R)) R >>= 1;
    if (R < 8) return 0;
    if (R == 64 && 2 * (int64_t)P.B * ((P.L + R - 1) / R) <= 148) R = 32;
    return R;
}

// CTAs of a (batch, KV head) pair: two per SM in all, eight units of eight keys per CTA and turn
int ctas_per_pair(const Prob& P) {
    const int pairs = P.B * P.Hkv, want = (2 * 148 + pairs - 1) / pairs, most = (P.L + 8 * kRows - 1) / (8 * kRows);
    return want < most ? want : most;
}

}  // namespace

static size_t full_partial_bytes(const Prob& P, size_t ctas) { return ctas * P.Hq * ((size_t)P.Hkv * P.d + 1) * sizeof(float); }
static size_t partial_bytes(const Prob& P, size_t ctas) { return ctas * P.G * (P.d + 1) * sizeof(float); }

size_t mask_bwd_need(const Prob& P) {
    if (P.flags & DMA_FLAG_FULL_DELTA) {
        const int R = full_rows(P);
        return R == 0 ? 0 : full_partial_bytes(P, (size_t)P.B * ((P.L + R - 1) / R));
    }
    return partial_bytes(P, (size_t)P.B * P.Hkv * ctas_per_pair(P));
}

// CTAs go down where a longer sequence takes 64 rows per CTA instead of 32, or where more pairs leave no room for a second CTA per
// pair, but a workspace of that size serves the smaller problems too: the bound for all of them.
size_t mask_bwd_ws_bytes(const Prob& P) {
    if (P.flags & DMA_FLAG_FULL_DELTA) {
        const size_t half = std::min((size_t)P.B * ((P.L + 31) / 32), (size_t)148);        // (of 32 rows, while they run at once)
        return full_fits(P, 64) ? std::max(mask_bwd_need(P), full_partial_bytes(P, half)) : mask_bwd_need(P);
    }
    const size_t pairs = (size_t)P.B * P.Hkv;                              // (pairs * ceil(296 / pairs) < pairs + 296)
    return partial_bytes(P, std::min(pairs * ((P.L + 8 * kRows - 1) / (8 * kRows)), pairs + 2 * 148 - 1));
}

template <typename T, int D>
static int launch_typed(const Prob& P, const void* V, const float* W, const float* A, const float* delta, const float* dM,
                        void* dV, float* dW, float* dA, void* ws, cudaStream_t st) {
    const int nblk = ctas_per_pair(P);
    constexpr size_t smem_head = (D + 8 * (D + 1) + 8 * 2 * kRows) * sizeof(float);
    const size_t smem = P.G * smem_head;
    auto kern = P.G == 1 ? mask_bwd_kernel<T, D, 1> : P.G == 2 ? mask_bwd_kernel<T, D, 2> : P.G == 4 ? mask_bwd_kernel<T, D, 4> : mask_bwd_kernel<T, D, 0>;
    // (state of the function, which other threads' calls share: always the limit)
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxGroup * smem_head)) != cudaSuccess) return DMA_ERR_CUDA;
    const int rc = launch_overlapped(kern, dim3(nblk, P.Hkv, P.B), dim3(kThreads), smem, st, 1, (const T*)V, W, A, delta, dM, (T*)dV, (float*)ws, P.L, P.Hq,
                                     P.G, P.vs[0], P.vs[1], P.vs[2]);
    if (rc) return rc;
    return launch_overlapped(mask_bwd_reduce_kernel<D>, dim3(P.Hq, D / 32 + 1), dim3(512), 0, st, 1, (const float*)ws, dW, dA, P.B, P.Hkv, P.G,
                             nblk);
}

template <typename T, int RW>
static int launch_full(const Prob& P, const void* V, const float* W, const float* A, const float* delta, const float* dM,
                       void* dV, float* dW, float* dA, void* ws, cudaStream_t st) {
    constexpr int R = RW * 8;
    const int nblk = (P.L + R - 1) / R, C = P.Hkv * P.d, HqP = (P.Hq + 7) & ~7;
    const size_t smem = ((size_t)R * C + (size_t)R * HqP + (size_t)P.Hq * R) * sizeof(float);
    if (cudaFuncSetAttribute(mask_bwd_full_kernel<T, RW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFullSmem) != cudaSuccess)
        return DMA_ERR_CUDA;
    const int rc = launch_overlapped(mask_bwd_full_kernel<T, RW>, dim3(nblk, P.B), dim3(kFullThreads), smem, st, 1, (const T*)V, W, A, delta, dM, (T*)dV,
                                     (float*)ws, P.L, P.Hq, P.Hkv, P.d, P.vs[0], P.vs[1], P.vs[2]);
    if (rc) return rc;
    return launch_overlapped(mask_bwd_full_reduce_kernel, dim3(C / 32 + 1, P.Hq), dim3(512), 0, st, 1, (const float*)ws, dW, dA, P.B * nblk, P.Hq, C);
}

template <typename T>
static int launch_full_rows(const Prob& P, const void* V, const float* W, const float* A, const float* delta, const float* dM,
                            void* dV, float* dW, float* dA, void* ws, cudaStream_t st) {
    switch (full_rows(P)) {
        case 64: return launch_full<T, 8>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
        case 32: return launch_full<T, 4>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
        case 16: return launch_full<T, 2>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
        case 8: return launch_full<T, 1>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
    }
    return DMA_ERR_UNSUPPORTED;
}

int launch_mask_bwd(const Prob& P, const void* V, const float* W, const float* A, const float* delta, const float* dM,
                    void* dV, float* dW, float* dA, void* ws, cudaStream_t st) {
    if (P.flags & DMA_FLAG_FULL_DELTA)
        return P.dtype == DMA_BF16 ? launch_full_rows<__nv_bfloat16>(P, V, W, A, delta, dM, dV, dW, dA, ws, st)
                                   : launch_full_rows<float>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
    if (P.G > kMaxGroup) return DMA_ERR_UNSUPPORTED;
    if (P.dtype == DMA_BF16) {
        return P.d == 128 ? launch_typed<__nv_bfloat16, 128>(P, V, W, A, delta, dM, dV, dW, dA, ws, st)
                          : launch_typed<__nv_bfloat16, 64>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
    }
    return P.d == 128 ? launch_typed<float, 128>(P, V, W, A, delta, dM, dV, dW, dA, ws, st)
                      : launch_typed<float, 64>(P, V, W, A, delta, dM, dV, dW, dA, ws, st);
}

}  // namespace dma
