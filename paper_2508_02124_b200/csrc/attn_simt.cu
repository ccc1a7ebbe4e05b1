// CUDA-core (fp32 FMA) attention kernels: the fp32 element type needs full fp32 products, which the tensor
// cores do not give. Same semantics as the tensor-core path: additive per-key bias, per-element validity
// j <= i < expiry[j], key tiles whose bitmap bit is clear are neither loaded nor computed.
//   forward   Alg. 1 with the loop order swapped (a CTA owns query rows, online softmax across key tiles)
//   backward  one launch, two kinds of CTAs: some own keys of one KV head, walk the query heads of the group and their active
//             64-row tiles and keep dK, dV and dM; the others own query rows, walk the key tiles and keep dQ. The scores are
//             formed twice (seven products instead of Alg. 2's five), but nothing is added through memory: no accumulator to
//             clear, add to with atomics and convert, and every gradient is the same bits from run to run.
// All three loops are the same: a WARP holds two or four stationary rows (of Q, or of K) and walks 64-row tiles that the CTA streams
// through shared memory in two buffers. For the products over channels a lane owns two of the tile's rows (its row's 16-byte
// chunks are conflict-free at a pitch of D + 4 floats, the stationary rows are broadcast); the softmax stays within the warp;
// for the products over the tile's rows a lane owns D / 32 channels and reads the weights, left in shared memory by the warp,
// as broadcasts. The only CTA-wide barriers are those around a tile's arrival, and a CTA can be as small as 8 rows, which is
// what a small problem needs: it is bound by the serial walk over its tiles, on as many CTAs as it has. A large one is bound
// by shared-memory reads (12 clocks of them per 8 clocks of FMAs with four rows per warp).
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace dma {
namespace {

constexpr int kTile = 64;              // rows of a streamed tile

// rows r0 .. r0 + n - 1 of a [*, D] operand (zero beyond `limit` rows) to shared memory at a pitch of LD floats, by all threads
template <typename T, int D, int LD>
__device__ __forceinline__ void stage_rows(float* dst, const T* src, int64_t row_stride, int r0, int n, int limit) {
    for (int idx = threadIdx.x; idx < n * (D / 4); idx += blockDim.x) {
        const int r = idx / (D / 4), c = (idx % (D / 4)) * 4;
        const bool in = r0 + r < limit;
        const T* p = src + (int64_t)(in ? r0 + r : 0) * row_stride + c;
        float* d = dst + r * LD + c;
        if constexpr (sizeof(T) == 4) {
            ptx::cp_async16(d, p, in ? 16 : 0);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) d[u] = in ? to_f32(p[u]) : 0.0f;
        }
    }
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }      // all but the newest group

// s[a][t] = own row a . tile row (lane + 32 t)
template <int D, int kOwn>
__device__ __forceinline__ void dots(const float* own, const float* tile, int lane, float (&s)[kOwn][2]) {
    constexpr int LD = D + 4;
#pragma unroll
    for (int a = 0; a < kOwn; ++a) s[a][0] = s[a][1] = 0.0f;
    const float* y0 = tile + lane * LD;
    const float* y1 = y0 + 32 * LD;
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 32) {       // partial sums of 32 channels: shorter chains lose less
        float p[kOwn][2];
#pragma unroll
        for (int a = 0; a < kOwn; ++a) p[a][0] = p[a][1] = 0.0f;
#pragma unroll
        for (int c = c0; c < c0 + 32; c += 4) {
            const float4 u = *reinterpret_cast<const float4*>(y0 + c), v = *reinterpret_cast<const float4*>(y1 + c);
#pragma unroll
            for (int a = 0; a < kOwn; ++a) {
                const float4 x = *reinterpret_cast<const float4*>(own + a * D + c);
                p[a][0] = fmaf(x.x, u.x, p[a][0]); p[a][1] = fmaf(x.x, v.x, p[a][1]);
                p[a][0] = fmaf(x.y, u.y, p[a][0]); p[a][1] = fmaf(x.y, v.y, p[a][1]);
                p[a][0] = fmaf(x.z, u.z, p[a][0]); p[a][1] = fmaf(x.z, v.z, p[a][1]);
                p[a][0] = fmaf(x.w, u.w, p[a][0]); p[a][1] = fmaf(x.w, v.w, p[a][1]);
            }
        }
#pragma unroll
        for (int a = 0; a < kOwn; ++a) {
            s[a][0] += p[a][0];
            s[a][1] += p[a][1];
        }
    }
}

// acc[a][c] += sum over the tile's rows j of wts[a][j] tile[j][lane's channel c]; wts [kOwn][kTile] in shared memory
template <int D, int kOwn>
__device__ __forceinline__ void accumulate(const float* wts, const float* tile, int lane, float (&acc)[kOwn][D / 32]) {
    constexpr int LD = D + 4, CPL = D / 32;
    float sum[kOwn][CPL];                  // of this tile: sums of sums lose less than one long chain
#pragma unroll
    for (int a = 0; a < kOwn; ++a)
#pragma unroll
        for (int c = 0; c < CPL; ++c) sum[a][c] = 0.0f;
#pragma unroll 4
    for (int j = 0; j < kTile; j += 4) {
        float4 p[kOwn];
#pragma unroll
        for (int a = 0; a < kOwn; ++a) p[a] = *reinterpret_cast<const float4*>(wts + a * kTile + j);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float y[CPL];
            const float* row = tile + (j + u) * LD + lane * CPL;
            if constexpr (CPL == 4) {
                const float4 v = *reinterpret_cast<const float4*>(row);
                y[0] = v.x; y[1] = v.y; y[2] = v.z; y[3] = v.w;
            } else {
                const float2 v = *reinterpret_cast<const float2*>(row);
                y[0] = v.x; y[1] = v.y;
            }
#pragma unroll
            for (int a = 0; a < kOwn; ++a) {
                const float w = u == 0 ? p[a].x : u == 1 ? p[a].y : u == 2 ? p[a].z : p[a].w;
#pragma unroll
                for (int c = 0; c < CPL; ++c) sum[a][c] = fmaf(w, y[c], sum[a][c]);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < kOwn; ++a)
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[a][c] += sum[a][c];
}

template <typename T, int D>
__device__ __forceinline__ void store_row(T* dst, const float (&v)[D / 32], float mul, int lane) {
#pragma unroll
    for (int c = 0; c < D / 32; ++c) store_as(dst + lane * (D / 32) + c, v[c] * mul);
}

// Walks the tiles first, next(first), ... while < end: fetch(tile, buffer) stages one, body(tile, buffer) uses it. The next
// tile's copies are in flight while a tile is used.
template <typename Next, typename Fetch, typename Body>
__device__ __forceinline__ void walk_tiles(int first, int end, Next next, Fetch fetch, Body body) {
    int t = first;
    if (t < end) { fetch(t, 0); stage_commit(); }
    for (int buf = 0; t < end; buf ^= 1) {
        const int tn = next(t);
        if (tn < end) fetch(tn, buf ^ 1);
        stage_commit();
        stage_wait();
        __syncthreads();
        body(t, buf);
        __syncthreads();               // the buffer may be filled again
        t = tn;
    }
}

template <typename T, int D, int kOwn, int NW>
__global__ void __launch_bounds__(32 * NW) simt_fwd_kernel(const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V,
                                                           const float* __restrict__ bias, const int32_t* __restrict__ expiry,
                                                           const uint32_t* __restrict__ bitmap, T* __restrict__ O, float* __restrict__ lse,
                                                           Prob P, int use_bitmap, int32_t* __restrict__ status) {
    constexpr int LD = D + 4, BM = kOwn * NW;
    extern __shared__ __align__(16) float sm[];
    float* sQ = sm;                              // [BM][D]
    float* sY = sQ + BM * D;                     // two buffers of K [kTile][LD], V [kTile][LD]
    float* sP = sY + 4 * kTile * LD;             // [NW][kOwn][kTile]
    const int h = blockIdx.y, b = blockIdx.z, hk = h / P.G, bh = b * P.Hq + h;
    const int i0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * BM, L = P.L;       // first row inside the chunk (longest walks first)
    const int ia0 = P.q_off + i0;                // its position in the sequence
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_enter(Q, K, V, bias, expiry, bitmap, O, lse, status);
    static_assert(32 * NW >= kWsHeaderBytes / 4, "one CTA clears the workspace header");       // (a memset in front of the kernel is 2 us and keeps it from overlapping)
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x < kWsHeaderBytes / 4) status[threadIdx.x] = 0;
    const T* q = Q + b * P.qs[0] + h * P.qs[2];
    const T* k = K + b * P.ks[0] + hk * P.ks[2];
    const T* v = V + b * P.vs[0] + hk * P.vs[2];
    const float* own = sQ + warp * kOwn * D;
    float* wts = sP + warp * kOwn * kTile;
    const int r0 = ia0 + warp * kOwn;            // position of the warp's first row

    stage_rows<T, D, D>(sQ, q, P.qs[1], i0, BM, P.Lq);
    float acc[kOwn][D / 32], m[kOwn], l[kOwn];
#pragma unroll
    for (int a = 0; a < kOwn; ++a) {
        m[a] = -INFINITY;
        l[a] = 0.0f;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) acc[a][c] = 0.0f;
    }
    const int keys = P.causal ? min(ia0 + BM, L) : L;          // keys that some row of the CTA can see
    auto next = [&](int j0) {
        j0 += kTile;
        while (use_bitmap && j0 < keys && !bitmap_test(bitmap, P.Tr, P.Wd, bh, ia0 / P.bm, j0 / P.bn)) j0 += kTile;
        return j0;
    };
    auto fetch = [&](int j0, int buf) {
        stage_rows<T, D, LD>(sY + buf * 2 * kTile * LD, k, P.ks[1], j0, kTile, L);
        stage_rows<T, D, LD>(sY + (buf * 2 + 1) * kTile * LD, v, P.vs[1], j0, kTile, L);
    };
    auto body = [&](int j0, int buf) {
        const float* sK = sY + buf * 2 * kTile * LD;
        float bj[2];
        int ej[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int j = j0 + lane + 32 * t;
            bj[t] = j < L ? bias[(size_t)bh * L + j] : 0.0f;
            ej[t] = j < L ? expiry[(size_t)bh * L + j] : 0;
        }
        float s[kOwn][2];
        dots<D, kOwn>(own, sK, lane, s);
#pragma unroll
        for (int a = 0; a < kOwn; ++a) {
            const int i = r0 + a;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int j = j0 + lane + 32 * t;
                s[a][t] = ((j <= i || !P.causal) && i < ej[t]) ? s[a][t] * P.scale + bj[t] : -INFINITY;
            }
            float mx = fmaxf(s[a][0], s[a][1]);
#pragma unroll
            for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float m_new = fmaxf(m[a], mx), m_use = m_new == -INFINITY ? 0.0f : m_new;
            const float alpha = expf(m[a] - m_use), p0 = expf(s[a][0] - m_use), p1 = expf(s[a][1] - m_use);
            m[a] = m_new;
            l[a] = l[a] * alpha + (p0 + p1);     // this lane's part of the row sum
            wts[a * kTile + lane] = p0;
            wts[a * kTile + lane + 32] = p1;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) acc[a][c] *= alpha;
        }
        __syncwarp();
        accumulate<D, kOwn>(wts, sK + kTile * LD, lane, acc);
    };
    walk_tiles(next(-kTile), keys, next, fetch, body);
#pragma unroll
    for (int a = 0; a < kOwn; ++a) {
        const int il = i0 + warp * kOwn + a;
#pragma unroll
        for (int o = 16; o; o >>= 1) l[a] += __shfl_xor_sync(0xffffffffu, l[a], o);
        if (il >= P.Lq) continue;
        store_row<T, D>(O + b * P.os[0] + (int64_t)il * P.os[1] + h * P.os[2], acc[a], l[a] > 0.0f ? 1.0f / l[a] : 0.0f, lane);
        if (lane == 0) lse[(size_t)bh * P.Lq + il] = l[a] > 0.0f ? m[a] + logf(l[a]) : -INFINITY;
    }
    ptx::cp_async_wait_all();
}

// D_i = dO_i . O_i  (Alg. 2): one warp per (b, h, i)
template <typename T>
__global__ void rowdot_kernel(const T* __restrict__ O, const T* __restrict__ dO, float* __restrict__ Dv, Prob P, int32_t* __restrict__ status) {
    const long row = (long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    pdl_enter(O, dO, Dv, status);
    if (blockIdx.x == 0 && threadIdx.x < kWsHeaderBytes / 4) status[threadIdx.x] = 0;         // (the stage's first kernel clears the workspace header)
    if (row >= (long)P.B * P.Hq * P.L) return;
    const int i = row % P.L, h = (row / P.L) % P.Hq, b = row / ((long)P.L * P.Hq);
    const T* o = O + b * P.os[0] + (int64_t)i * P.os[1] + h * P.os[2];
    const T* g = dO + b * P.os[0] + (int64_t)i * P.os[1] + h * P.os[2];
    float s = 0.0f;
    for (int c = lane; c < P.d; c += 32) s = fmaf(to_f32(o[c]), to_f32(g[c]), s);
    for (int m = 16; m; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    if (lane == 0) Dv[row] = s;
}

// Grid: (Hkv + Hq heads of nblk blocks each, B). Head y < Hkv: dK, dV, dM of BM keys of that KV head; else dQ of BM rows of query
// head y - Hkv. (The heads are not blockIdx.y, which ends at 65535: calls with that many query heads are accepted.)
template <typename T, int D, int kOwn, int NW>
__global__ void __launch_bounds__(32 * NW) simt_bwd_kernel(const T* __restrict__ Q, const T* __restrict__ K, const T* __restrict__ V,
                                                           const T* __restrict__ dO, const float* __restrict__ lse, const float* __restrict__ Dv,
                                                           const float* __restrict__ bias, const int32_t* __restrict__ expiry,
                                                           const uint32_t* __restrict__ bitmap, T* __restrict__ dQ, T* __restrict__ dK,
                                                           T* __restrict__ dV, float* __restrict__ dM, Prob P, int use_bitmap, int nblk) {
    constexpr int LD = D + 4, BM = kOwn * NW;
    extern __shared__ __align__(16) float sm[];
    float* sA = sm;                              // stationary rows: K, V (or Q, dO), [BM][D] each
    float* sY = sA + 2 * BM * D;                 // two buffers of Q, dO (or K, V) tiles, [kTile][LD] each
    float* sP = sY + 4 * kTile * LD;             // [NW][2][kOwn][kTile]
    const int b = blockIdx.y, head = blockIdx.x / nblk, blk = blockIdx.x % nblk;
    const int L = P.L, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_enter(Q, K, V, dO, lse, Dv, bias, expiry, bitmap, dQ, dK, dV, dM);
    float* wts = sP + warp * 2 * kOwn * kTile;
    const float* own1 = sA + warp * kOwn * D;
    const float* own2 = own1 + BM * D;

    if (head < P.Hkv) {
        const int hk = head, j0 = blk * BM;       // (causal: the first keys have the longest walks)
        stage_rows<T, D, D>(sA, K + b * P.ks[0] + hk * P.ks[2], P.ks[1], j0, BM, L);
        stage_rows<T, D, D>(sA + BM * D, V + b * P.vs[0] + hk * P.vs[2], P.vs[1], j0, BM, L);
        float adk[kOwn][D / 32], adv[kOwn][D / 32];
#pragma unroll
        for (int a = 0; a < kOwn; ++a)
#pragma unroll
            for (int c = 0; c < D / 32; ++c) adk[a][c] = adv[a][c] = 0.0f;
        for (int g = 0; g < P.G; ++g) {
            const int h = hk * P.G + g, bh = b * P.Hq + h;
            float bj[kOwn], dm[kOwn];
            int ej[kOwn];
#pragma unroll
            for (int a = 0; a < kOwn; ++a) {
                const int j = j0 + warp * kOwn + a;
                bj[a] = j < L ? bias[(size_t)bh * L + j] : 0.0f;
                ej[a] = j < L ? expiry[(size_t)bh * L + j] : 0;
                dm[a] = 0.0f;
            }
            const T* q = Q + b * P.qs[0] + h * P.qs[2];
            const T* go = dO + b * P.os[0] + h * P.os[2];
            auto next = [&](int i0) {
                i0 += kTile;
                while (use_bitmap && i0 < L && !bitmap_test(bitmap, P.Tr, P.Wd, bh, i0 / P.bm, j0 / P.bn)) i0 += kTile;
                return i0;
            };
            auto fetch = [&](int i0, int buf) {
                stage_rows<T, D, LD>(sY + buf * 2 * kTile * LD, q, P.qs[1], i0, kTile, L);
                stage_rows<T, D, LD>(sY + (buf * 2 + 1) * kTile * LD, go, P.os[1], i0, kTile, L);
            };
            auto body = [&](int i0, int buf) {
                const float* sQ = sY + buf * 2 * kTile * LD;
                const float* sG = sQ + kTile * LD;
                float li[2], di[2];
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int i = i0 + lane + 32 * t;
                    li[t] = i < L ? lse[(size_t)bh * L + i] : 0.0f;
                    di[t] = i < L ? Dv[(size_t)bh * L + i] : 0.0f;
                }
                float s[kOwn][2], dp[kOwn][2];
                dots<D, kOwn>(own1, sQ, lane, s);
                dots<D, kOwn>(own2, sG, lane, dp);
#pragma unroll
                for (int a = 0; a < kOwn; ++a) {
                    const int j = j0 + warp * kOwn + a;
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const int i = i0 + lane + 32 * t;
                        const bool ok = (j <= i || !P.causal) && i < ej[a] && i < L;
                        const float p = ok ? expf(s[a][t] * P.scale + bj[a] - li[t]) : 0.0f;
                        const float ds = p * (dp[a][t] - di[t]);
                        wts[a * kTile + lane + 32 * t] = p;
                        wts[(kOwn + a) * kTile + lane + 32 * t] = ds;
                        dm[a] += ds;
                    }
                }
                __syncwarp();
                accumulate<D, kOwn>(wts, sG, lane, adv);
                accumulate<D, kOwn>(wts + kOwn * kTile, sQ, lane, adk);
            };
            walk_tiles(next((P.causal ? j0 / kTile * kTile : 0) - kTile), L, next, fetch, body);
#pragma unroll
            for (int a = 0; a < kOwn; ++a) {
                const int j = j0 + warp * kOwn + a;
#pragma unroll
                for (int o = 16; o; o >>= 1) dm[a] += __shfl_xor_sync(0xffffffffu, dm[a], o);
                if (lane == 0 && j < L) dM[(size_t)bh * L + j] = dm[a];
            }
        }
#pragma unroll
        for (int a = 0; a < kOwn; ++a) {
            const int j = j0 + warp * kOwn + a;
            if (j >= L) continue;
            store_row<T, D>(dK + b * P.ks[0] + (int64_t)j * P.ks[1] + hk * P.ks[2], adk[a], P.scale, lane);
            store_row<T, D>(dV + b * P.vs[0] + (int64_t)j * P.vs[1] + hk * P.vs[2], adv[a], 1.0f, lane);
        }
    } else {
        const int h = head - P.Hkv, hk = h / P.G, bh = b * P.Hq + h;
        const int i0 = (nblk - 1 - blk) * BM;
        stage_rows<T, D, D>(sA, Q + b * P.qs[0] + h * P.qs[2], P.qs[1], i0, BM, L);
        stage_rows<T, D, D>(sA + BM * D, dO + b * P.os[0] + h * P.os[2], P.os[1], i0, BM, L);
        float adq[kOwn][D / 32], li[kOwn], di[kOwn];
#pragma unroll
        for (int a = 0; a < kOwn; ++a) {
            const int i = i0 + warp * kOwn + a;
            li[a] = i < L ? lse[(size_t)bh * L + i] : 0.0f;
            di[a] = i < L ? Dv[(size_t)bh * L + i] : 0.0f;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) adq[a][c] = 0.0f;
        }
        const T* k = K + b * P.ks[0] + hk * P.ks[2];
        const T* v = V + b * P.vs[0] + hk * P.vs[2];
        const int keys = P.causal ? min(i0 + BM, L) : L;
        auto next = [&](int j0) {
            j0 += kTile;
            while (use_bitmap && j0 < keys && !bitmap_test(bitmap, P.Tr, P.Wd, bh, i0 / P.bm, j0 / P.bn)) j0 += kTile;
            return j0;
        };
        auto fetch = [&](int j0, int buf) {
            stage_rows<T, D, LD>(sY + buf * 2 * kTile * LD, k, P.ks[1], j0, kTile, L);
            stage_rows<T, D, LD>(sY + (buf * 2 + 1) * kTile * LD, v, P.vs[1], j0, kTile, L);
        };
        auto body = [&](int j0, int buf) {
            const float* sK = sY + buf * 2 * kTile * LD;
            float bj[2];
            int ej[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int j = j0 + lane + 32 * t;
                bj[t] = j < L ? bias[(size_t)bh * L + j] : 0.0f;
                ej[t] = j < L ? expiry[(size_t)bh * L + j] : 0;
            }
            float s[kOwn][2], dp[kOwn][2];
            dots<D, kOwn>(own1, sK, lane, s);
            dots<D, kOwn>(own2, sK + kTile * LD, lane, dp);
#pragma unroll
            for (int a = 0; a < kOwn; ++a) {
                const int i = i0 + warp * kOwn + a;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int j = j0 + lane + 32 * t;
                    const bool ok = (j <= i || !P.causal) && i < ej[t] && i < L;
                    const float p = ok ? expf(s[a][t] * P.scale + bj[t] - li[a]) : 0.0f;
                    wts[a * kTile + lane + 32 * t] = p * (dp[a][t] - di[a]);
                }
            }
            __syncwarp();
            accumulate<D, kOwn>(wts, sK, lane, adq);
        };
        walk_tiles(next(-kTile), keys, next, fetch, body);
#pragma unroll
        for (int a = 0; a < kOwn; ++a) {
            const int i = i0 + warp * kOwn + a;
            if (i < L) store_row<T, D>(dQ + b * P.qs[0] + (int64_t)i * P.qs[1] + h * P.qs[2], adq[a], P.scale, lane);
        }
    }
    ptx::cp_async_wait_all();
}

template <typename T, int D, int kOwn, int NW>
int fwd_t(const Prob& P, const void* Q, const void* K, const void* V, const float* bias, const int32_t* expiry,
          const uint32_t* bitmap, void* O, float* lse, void* ws, cudaStream_t st) {
    constexpr size_t smem = (size_t)(kOwn * NW * D + 4 * kTile * (D + 4) + NW * kOwn * kTile) * sizeof(float);
    auto kern = simt_fwd_kernel<T, D, kOwn, NW>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return DMA_ERR_CUDA;
    // a chunk of query rows that does not start on a bitmap row boundary (or comes without a bitmap) visits every key tile
    int use_bitmap = bitmap && !(P.flags & DMA_FLAG_IGNORE_BITMAP) && P.bm % kTile == 0 && P.bn % kTile == 0 && P.q_off % kTile == 0;
    timing_mark(0, false, st);
    const int rc = launch_overlapped(kern, dim3((P.Lq + kOwn * NW - 1) / (kOwn * NW), P.Hq, P.B), dim3(32 * NW), smem, st, 1, (const T*)Q, (const T*)K,
                                     (const T*)V, bias, expiry, bitmap, (T*)O, lse, P, use_bitmap, (int32_t*)ws);
    timing_mark(0, true, st);
    return rc;
}

template <typename T, int D, int kOwn, int NW>
int bwd_t(const Prob& P, const void* Q, const void* K, const void* V, const void* O, const void* dO, const float* lse,
          const float* bias, const int32_t* expiry, const uint32_t* bitmap, void* dQ, void* dK, void* dV, float* dM,
          void* ws, cudaStream_t st) {
    constexpr size_t smem = (size_t)(2 * kOwn * NW * D + 4 * kTile * (D + 4) + NW * 2 * kOwn * kTile) * sizeof(float);
    auto kern = simt_bwd_kernel<T, D, kOwn, NW>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return DMA_ERR_CUDA;
    const size_t rows = (size_t)P.B * P.Hq * P.L;
    float* Dv = reinterpret_cast<float*>((char*)ws + kWsHeaderBytes);
    int rc = launch_overlapped(rowdot_kernel<T>, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, 1, (const T*)O, (const T*)dO, Dv, P, (int32_t*)ws);
    if (rc) return rc;
    int use_bitmap = !(P.flags & DMA_FLAG_IGNORE_BITMAP) && P.bm % kTile == 0 && P.bn % kTile == 0;
    const int nblk = (P.L + kOwn * NW - 1) / (kOwn * NW);
    timing_mark(1, false, st);
    rc = launch_overlapped(kern, dim3((unsigned)nblk * (unsigned)(P.Hkv + P.Hq), P.B), dim3(32 * NW), smem, st, 1, (const T*)Q, (const T*)K,
                           (const T*)V, (const T*)dO, lse, Dv, bias, expiry, bitmap, (T*)dQ, (T*)dK, (T*)dV, dM, P, use_bitmap, nblk);
    timing_mark(1, true, st);
    return rc;
}

// CTA size: 32 rows (four per warp, eight warps) when that gives every SM a CTA; else 8 rows (two per warp, four warps), where a
// warp reads twice as much shared memory per product but the serial walk of a CTA is shorter. Forward / backward, us: two
// heads of 256 rows, D = 64, 12.9 / 20.7 (32-row CTAs 22.7 / 31.0); eight heads of 1024 rows, D = 128, 146 / 344 with 32 rows,
// 195 / 559 with 8 (64-row CTAs and scalar reads before: 253 / 522; 47 / 90 at the small size).
bool small_grid(const Prob& P, int rows, int heads) { return (int64_t)((rows + 31) / 32) * heads * P.B < 148; }

}  // namespace

size_t simt_bwd_ws_bytes(const Prob& P) {
    const size_t rows = (size_t)P.B * P.Hq * P.L;
    return kWsHeaderBytes + ((rows + 63) / 64) * 64 * sizeof(float);
}

int launch_simt_fwd(const Prob& P, const void* Q, const void* K, const void* V, const float* bias,
                    const int32_t* expiry, const uint32_t* bitmap, void* O, float* lse, void* ws, cudaStream_t st) {
    const bool small = small_grid(P, P.Lq, P.Hq);
    auto pick = [&](auto t_tag) {
        using T = decltype(t_tag);
        return P.d == 128 ? (small ? fwd_t<T, 128, 2, 4> : fwd_t<T, 128, 4, 8>) : (small ? fwd_t<T, 64, 2, 4> : fwd_t<T, 64, 4, 8>);
    };
    auto f = P.dtype == DMA_FP32 ? pick(float()) : pick(__nv_bfloat16());
    return f(P, Q, K, V, bias, expiry, bitmap, O, lse, ws, st);
}

int launch_simt_bwd(const Prob& P, const void* Q, const void* K, const void* V, const void* O, const void* dO,
                    const float* lse, const float* bias, const int32_t* expiry, const uint32_t* bitmap, void* dQ,
                    void* dK, void* dV, float* dM, void* ws, cudaStream_t st) {
    const bool small = small_grid(P, P.L, P.Hq + P.Hkv);
    auto pick = [&](auto t_tag) {
        using T = decltype(t_tag);
        return P.d == 128 ? (small ? bwd_t<T, 128, 2, 4> : bwd_t<T, 128, 4, 8>) : (small ? bwd_t<T, 64, 2, 4> : bwd_t<T, 64, 4, 8>);
    };
    auto f = P.dtype == DMA_FP32 ? pick(float()) : pick(__nv_bfloat16());
    return f(P, Q, K, V, O, dO, lse, bias, expiry, bitmap, dQ, dK, dV, dM, ws, st);
}

}  // namespace dma
