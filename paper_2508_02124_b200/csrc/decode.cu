// Decoding step (Sec. 3.2 for a single query at the end of the sequence; Alg. 1 with the per-key mask M in R^N, the
// configuration of the paper's decode benchmark): every (batch, query head) keeps the w cached keys with the largest
// dynamic weight delta (ties to the lower index; all N keys if N <= w) and attends to them with delta as the bias.
// HBM / L2-bound: the delta row is read once to select, then only the selected K and V rows are read.
//
// Kernels
//   decode_select_kernel   one cluster of CTAs per (batch, head) row: exact selection and the kept indices in ascending order
//   decode_select_stream_kernel   the same for many rows and rows of one CTA's registers, a CTA per row that reads it once
//   decode_attn_kernel     per (batch, head, split of the kept list): every warp gathers a batch of K and V rows with all its
//                          loads in flight, softmax per batch, warps combined in shared memory -> partial (m, l, o). The CTA
//                          that finishes a row last (a ticket counter, no waiting) combines the row's partials -> o, lse
//   decode_list_attn_kernel, decode_step_combine_kernel   the same for a kept set that is carried from step to step
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace dma {
namespace {

namespace cg = cooperative_groups;

constexpr int kAttnThreads = 256;
constexpr int kMinSplit = 128, kMaxSplit = 512;     // kept keys per CTA of decode_attn_kernel

__device__ __forceinline__ unsigned long long key_of(float dl, int j) {
    return ((unsigned long long)__float_as_uint(dl) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)j);
}

// Selection of a row's `keep` best keys by the delta bit patterns (delta > 0: the sign bit is clear and the pattern orders
// like the value), then an ordered compaction of the keys above the threshold and of the first (lowest-index) keys at it.
// The first histogram divides the row's own range [min, max] into 2048 bins, so that a bin near the threshold holds a few
// dozen keys: those are gathered and ranked against each other. (Bins of fixed bit fields put a row into a few dozen bins in
// all; a warp's shared-memory adds then collide and three passes over the row are needed.) Only a row with more than
// kCandidates keys in the threshold's bin takes further passes, over the bin's own range.
// What bounds it is a chain of barriers and sweeps, not the row's bytes (read once), so the sweeps run on registers: a thread
// holds kKeys keys, key t of lane i of a warp at 32 t + i of the warp's contiguous part, which is both coalesced and in index
// order for the compaction. Rows of up to kCtaKeys keys take one CTA; longer ones a cluster, whose CTAs read each other's
// histograms (one cluster barrier per pass, a histogram buffer per pass; two bins to a word, and the barrier before the end only
// waited for when the list is written: 8 rows of 65536 keys 12.2 -> 10.9 us, of 131072 16.4 -> 14.2 at w = N / 4); rows beyond eight CTAs' registers are read again in
// every sweep (kKeys = 0), and their first range comes from a sample: a threshold in one of its end bins starts over with the
// true range. Measured, kept list written (before: threshold only, and a scan of the delta row in the attention kernel):
// 32 rows of 16384 keys 8.1 us (7.1), 256 rows of 65536 73 us (83 in four launches), 32 rows of 65536 11.4 us, where a
// cluster of two takes 16.8 and one CTA that reads the row again 52. A cluster is slow to start (1024 keys: 3.8 us on one CTA,
// 7.1 on two, 34 on eight), hence only where the registers demand it.
constexpr int kSelectThreads = 1024, kSelectWarps = kSelectThreads / 32;
constexpr int kSelectMaxCluster = 8;
constexpr int kCandidates = 256;
constexpr int kCtaKeys = 32 * kSelectThreads;
constexpr int kStateHeader = 8;               // int32 words before the kept indices in a row of an incremental state

struct alignas(16) SelectShared {
    int hist[4][2048];                        // this CTA's histogram of each pass
    unsigned long long cand[kCandidates];     // keys of this CTA in the threshold's bin ...
    unsigned long long all[kCandidates];      // ... and of the whole row
    int scan[kSelectWarps];
    uint32_t warp_min[kSelectWarps], warp_max[kSelectWarps];
    int warp_gt[kSelectWarps], warp_eq[kSelectWarps];
    uint32_t umin, umax;                      // of this CTA's slice
    int gt, eq;                               // keys above / at the threshold in this CTA's slice
    int ncand;
    uint32_t prefix;
    int need, count, bin;
};

// The row bh, by the cluster's nrank CTAs, from the zeroed S.hist and S.ncand on; out: its list.
// kState: the list is that of an incremental state; count and weakest kept key go to the header before it.
template <int kKeys, bool kState>
__device__ __forceinline__ void select_row(SelectShared& S, cg::cluster_group& cluster, int nrank, int rank, const float* __restrict__ delta, int64_t ld,
                                           int N, int keep, int slice, int bh, int* __restrict__ out) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = rank * slice, n = max(0, min(slice, N - j0));
    // this warp's part of the slice: [i0, i1), `seg` (a multiple of 32) keys per warp
    const int seg = kKeys ? 32 * kKeys : (slice + kSelectThreads - 1) / kSelectThreads * 32;
    const int i0 = warp * seg, i1 = min(n, i0 + seg), sweeps = seg / 32;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(delta + (size_t)bh * ld) + j0 + i0 + lane;
    // Keys beyond the row read as 0xFFFFFFFF, which no pass counts (the sign bit of the others is masked: delta > 0, and a
    // row that breaks this still yields `keep` distinct indices).
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    auto fetch = [&](int t) { return i0 + 32 * t + lane < i1 ? src[32 * t] & 0x7FFFFFFFu : kNone; };
    uint32_t key[kKeys ? kKeys : 1];
    if constexpr (kKeys > 0) {
#pragma unroll
        for (int t = 0; t < kKeys; ++t) key[t] = fetch(t);
    }
    auto sweep = [&](auto&& f) {               // f(t, key) for the warp's keys, in index order
        if constexpr (kKeys > 0) {
#pragma unroll
            for (int t = 0; t < kKeys; ++t) f(t, key[t]);
        } else {
#pragma unroll 8
            for (int t = 0; t < sweeps; ++t) f(t, fetch(t));
        }
    };
    // the range of the row's keys (`part`: of the first four of every lane only)
    auto range = [&](bool part, uint32_t& umin, uint32_t& umax) {
        umin = 0x7FFFFFFFu;
        umax = 0u;
        auto take = [&](int, uint32_t u) { if (u != kNone) { umin = min(umin, u); umax = max(umax, u); } };
        if (part) {
#pragma unroll
            for (int t = 0; t < 4; ++t) take(t, fetch(t));
        } else {
            sweep(take);
        }
        umin = __reduce_min_sync(0xffffffffu, umin);
        umax = __reduce_max_sync(0xffffffffu, umax);
        if (lane == 0) { S.warp_min[warp] = umin; S.warp_max[warp] = umax; }
        __syncthreads();
        umin = __reduce_min_sync(0xffffffffu, S.warp_min[lane]);
        umax = __reduce_max_sync(0xffffffffu, S.warp_max[lane]);
        if (nrank > 1) {
            if (tid == 0) { S.umin = umin; S.umax = umax; }
            cluster.sync();
            if (warp == 0) {                   // a lane per CTA
                const int q = min(lane, nrank - 1);
                umin = __reduce_min_sync(0xffffffffu, *cluster.map_shared_rank(&S.umin, q));
                umax = __reduce_max_sync(0xffffffffu, *cluster.map_shared_rank(&S.umax, q));
                if (lane == 0) { S.warp_min[0] = umin; S.warp_max[0] = umax; }
            }
            __syncthreads();
            umin = S.warp_min[0];
            umax = S.warp_max[0];
            if (kKeys == 0) cluster.sync();    // (a sample's range may be followed by the true one: the words are written again)
        }
    };
    bool sampled = kKeys == 0 && sweeps > 16;
    uint32_t lo, umax;
    range(sampled, lo, umax);                  // (its barrier: the histograms are zero)
    int shift = max(0, 21 - __clz((int)(umax - lo))), need = keep, cgt = 0, ceq = 0;
    bool counted = false;
    uint32_t nbins = 2048u;
    for (int pass = 0;; ++pass) {
        // the keys in [lo, lo + nbins << shift) into nbins bins; all others, and kNone, have a bin number beyond (shift <= 20),
        // or fall into the end bins after a sample
        int* hist = S.hist[pass];
        if (sampled) {
            sweep([&](int, uint32_t u) { if (u != kNone) atomicAdd(&hist[u < lo ? 0u : min((u - lo) >> shift, 2047u)], 1); });
        } else {
            sweep([&](int, uint32_t u) {
                const uint32_t bin = (u - lo) >> shift;
                if (bin < nbins) atomicAdd(&hist[bin], 1);
            });
        }
        // the bin holding the need-th largest key: two bins per thread in descending order
        int c0 = 0, c1 = 0;
        const int top = 2046 - 2 * tid;
        if (nrank > 1) {
            if constexpr (kKeys > 0) {
                // (a bin holds at most 32768 of the CTA's keys: two bins per word, half of what crosses between the SMs)
                __syncthreads();
                const int2 mine = *reinterpret_cast<const int2*>(hist + top);
                __syncthreads();
                uint32_t* packed = reinterpret_cast<uint32_t*>(hist);
                packed[tid] = (uint32_t)mine.x | (uint32_t)mine.y << 16;
                cluster.sync();
                uint32_t v[kSelectMaxCluster];
#pragma unroll
                for (int q = 0; q < kSelectMaxCluster; ++q) v[q] = q < nrank ? cluster.map_shared_rank(packed, q)[tid] : 0u;
#pragma unroll
                for (int q = 0; q < kSelectMaxCluster; ++q) {
                    c0 += (int)(v[q] >> 16);
                    c1 += (int)(v[q] & 0xFFFFu);
                }
            } else {
                cluster.sync();
                int2 v[kSelectMaxCluster];
#pragma unroll
                for (int q = 0; q < kSelectMaxCluster; ++q)
                    v[q] = q < nrank ? *reinterpret_cast<const int2*>(cluster.map_shared_rank(hist, q) + top) : make_int2(0, 0);
#pragma unroll
                for (int q = 0; q < kSelectMaxCluster; ++q) {
                    c0 += v[q].y;
                    c1 += v[q].x;
                }
            }
        } else {
            __syncthreads();
            const int2 v = *reinterpret_cast<const int2*>(hist + top);
            c0 = v.y;
            c1 = v.x;
        }
        const int sum = c0 + c1;
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) S.scan[warp] = incl;
        __syncthreads();
        const int before = __reduce_add_sync(0xffffffffu, lane < warp ? S.scan[lane] : 0);
        const int excl = before + incl - sum;  // keys in bins above this thread's first bin
        const bool in0 = excl < need && need <= excl + c0, in1 = excl + c0 < need && need <= excl + sum;
        if (in0 || in1) {
            S.bin = in0 ? top + 1 : top;
            S.need = need - excl - (in0 ? 0 : c0);
            S.count = in0 ? c0 : c1;
        }
        __syncthreads();
        const int bin = S.bin, count = S.count;
        if (sampled) {
            sampled = false;
            if (bin == 0 || bin == 2047) {     // beyond the sample's range (its ends included): once more with the true one
                range(false, lo, umax);
                shift = max(0, 21 - __clz((int)(umax - lo)));
                continue;
            }
        }
        lo += (uint32_t)bin << shift;
        need = S.need;
        if (shift == 0) break;                 // one pattern left: `need` keys with exactly this delta are kept
        if (count <= kCandidates) {
            // rank the bin's keys against each other; the keys above the bin are counted in the same sweep
            const uint32_t size = 1u << shift;
            sweep([&](int t, uint32_t u) {
                cgt += u - lo >= size && u > lo && u != kNone;
                if (u - lo < size) S.cand[atomicAdd(&S.ncand, 1)] = key_of(__uint_as_float(u), j0 + i0 + 32 * t + lane);
            });
            cgt = __reduce_add_sync(0xffffffffu, cgt);
            if (lane == 0) { S.warp_gt[warp] = cgt; S.warp_eq[warp] = 0; }
            const unsigned long long* cand = S.cand;
            if (nrank > 1) {
                cluster.sync();
                if (warp < kCandidates / 32) {
                    const int n_here = lane < nrank ? *cluster.map_shared_rank(&S.ncand, lane) : 0;
                    unsigned long long x[kSelectMaxCluster];
                    int nq[kSelectMaxCluster];
#pragma unroll
                    for (int q = 0; q < kSelectMaxCluster; ++q) {
                        nq[q] = __shfl_sync(0xffffffffu, n_here, q);
                        x[q] = tid < nq[q] ? cluster.map_shared_rank(S.cand, q)[tid] : 0ull;
                    }
                    int at = 0;
#pragma unroll
                    for (int q = 0; q < kSelectMaxCluster; ++q) {
                        if (tid < nq[q]) S.all[at + tid] = x[q];
                        at += nq[q];
                    }
                }
                cand = S.all;
            }
            __syncthreads();
            if (tid < count) {
                const unsigned long long k = cand[tid];
                int rank_k = 0, above = 0;
                for (int i = 0; i < count; ++i) {
                    const unsigned long long x = cand[i];
                    rank_k += x > k;
                    above += (uint32_t)(x >> 32) > (uint32_t)(k >> 32);
                }
                if (rank_k == need - 1) { S.prefix = (uint32_t)(k >> 32); S.need = need - above; }
            }
            __syncthreads();
            lo = S.prefix;
            need = S.need;
            if (tid < S.ncand) {               // this CTA's candidates join their warps' counts
                const unsigned long long k = S.cand[tid];
                const uint32_t u = (uint32_t)(k >> 32);
                const int owner = (int)(0xFFFFFFFFu - (uint32_t)k - (uint32_t)j0) / seg;
                if (u > lo) atomicAdd(&S.warp_gt[owner], 1);
                else if (u == lo) atomicAdd(&S.warp_eq[owner], 1);
            }
            counted = true;
            break;
        }
        nbins = 1u << min(11, shift);          // the next pass covers this bin and nothing above it
        shift = max(0, shift - 11);
        __syncthreads();                       // everyone has read the pass's result
    }
    const uint32_t prefix = lo;
    // prefix: delta bits of the threshold; `need` of the keys with exactly that delta are kept, lowest index first. Every
    // warp counts its part and writes from the position its lower-index neighbours leave it.
    if (!counted) {
        sweep([&](int, uint32_t u) { cgt += u > prefix && u != kNone; ceq += u == prefix; });
        cgt = __reduce_add_sync(0xffffffffu, cgt);
        ceq = __reduce_add_sync(0xffffffffu, ceq);
        if (lane == 0) { S.warp_gt[warp] = cgt; S.warp_eq[warp] = ceq; }
    }
    __syncthreads();
    cgt = S.warp_gt[warp];
    ceq = S.warp_eq[warp];
    int gtb = __reduce_add_sync(0xffffffffu, lane < warp ? S.warp_gt[lane] : 0);
    int eqb = __reduce_add_sync(0xffffffffu, lane < warp ? S.warp_eq[lane] : 0);
    if (nrank > 1) {
        if (warp == kSelectWarps - 1 && lane == 0) { S.gt = gtb + cgt; S.eq = eqb + ceq; }
        cluster.sync();
        gtb += __reduce_add_sync(0xffffffffu, lane < rank ? *cluster.map_shared_rank(&S.gt, lane) : 0);
        eqb += __reduce_add_sync(0xffffffffu, lane < rank ? *cluster.map_shared_rank(&S.eq, lane) : 0);
        cluster.barrier_arrive();              // (the last read of another CTA's shared memory: the list is written before the wait at the end)
    }
    const uint32_t below = (1u << lane) - 1u;
    if (ceq == 0) {                            // (all but a few warps)
        gtb += min(need, eqb);
        sweep([&](int t, uint32_t u) {
            const bool g = u > prefix && u != kNone;
            const uint32_t bg = __ballot_sync(0xffffffffu, g);
            if (g) out[gtb + __popc(bg & below)] = j0 + i0 + 32 * t + lane;
            gtb += __popc(bg);
        });
    } else {
        sweep([&](int t, uint32_t u) {
            const bool g = u > prefix && u != kNone, e = u == prefix;
            const uint32_t bg = __ballot_sync(0xffffffffu, g), be = __ballot_sync(0xffffffffu, e);
            const int j = j0 + i0 + 32 * t + lane, erank = eqb + __popc(be & below), pos = gtb + __popc(bg & below) + min(need, erank);
            if (g || (e && erank < need)) out[pos] = j;
            if (kState && e && erank == need - 1) {      // the weakest kept key: lowest delta, highest index
                int* hdr = out - kStateHeader;
                const unsigned long long k = key_of(__uint_as_float(u), j);
                hdr[0] = keep;
                hdr[1] = pos;
                hdr[2] = (int)(uint32_t)k;
                hdr[3] = (int)(uint32_t)(k >> 32);
            }
            gtb += __popc(bg);
            eqb += __popc(be);
        });
    }
    if (nrank > 1) cluster.barrier_wait();     // no CTA leaves while another may still read its shared memory
}

// list: row bh's kept indices go to list + bh * list_stride. tickets (may be NULL): one counter per row, zeroed here.
template <int kKeys, bool kState>
__global__ void __launch_bounds__(kSelectThreads, kKeys == 0 ? 2 : 1) decode_select_kernel(const float* __restrict__ delta, int64_t ld, int N, int keep, int slice,
                                                                       int* __restrict__ list, int64_t list_stride, int* __restrict__ tickets) {
    extern __shared__ __align__(16) uint8_t select_smem[];
    SelectShared& S = *reinterpret_cast<SelectShared*>(select_smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int nrank = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int bh = blockIdx.x / nrank, tid = threadIdx.x;
    for (int t = tid; t < (int)sizeof(S.hist) / 4; t += kSelectThreads) (&S.hist[0][0])[t] = 0;
    if (tid == 0) S.ncand = 0;
    pdl_enter(delta, list, tickets);
    int* out = list + (size_t)bh * list_stride;
    if (tickets && rank == 0 && tid == 0) tickets[bh] = 0;
    if (!kState && keep >= N) {                // every key is kept
        for (int i = rank * slice + tid; i < min(N, (rank + 1) * slice); i += kSelectThreads) out[i] = i;
        return;
    }
    select_row<kKeys, kState>(S, cluster, nrank, rank, delta, ld, N, keep, slice, bh, out);
}

// The same selection, one CTA per row, two on an SM, that reads the row once: a sample brackets the threshold (4.5 standard deviations to either side), the sweep
// leaves two bits per key (above the bracket, in it or above), the keys inside, a few per cent of the row, are gathered, and the last of them that
// is kept is found as above. The bits are then the row's list. A word of 32 keys costs some 30 instructions in all, where the histogram of all keys and
// three sweeps over registers took 880 per 1024 and a shared-memory add per key; both kernels are bound by them.
// Weights that crowd: a bracket end whose bin holds more than kHeavy of the sample is narrowed among that bin's samples; where the bracket is one bit pattern
// (equal weights), its first keys are kept by their bits alone, however many there are; and a bracket that misses, or holds more than kInside keys
// of several patterns, is narrowed by a histogram of the row's keys in it and swept again. A warp sweeps neighbouring words, but units of 32 words go around the warps
// afterwards, so that a bracket or a list that lies in one place of the row is not one warp's work.
// Carried state taken up from rows in the L2, us, kernel above / this one, at w = 64, N / 16, N / 4, N / 2, N - 1: 256 rows of 65536 keys 57 / 25, 65 / 30, 71 / 35, 79 / 39,
// 74 / 44, all weights equal 56 / 22 .. 70 / 41, ten values 67 / 28 .. 102 / 42, weights that rise along the row 57 / 26 .. 76 / 42 (before units, narrowing and the
// bits of equal weights: random 23 .. 160, equal 100 .. 114, ten values 26 .. 143, rising 28 .. 167); 148 rows of 131072 random 70 / 26 .. 88 / 55. From memory, up to N / 2: 256 rows of
// 65536 69 / 34, 79 / 39, 84 / 44, 87 / 48; the list in the order of the keys (its place from a count of the words first) 35, 40.3, 45.7, 49.7, a warp's words 32 apart in the sweep 34.6, 39.5, 45, 48.8.
constexpr int kInside = 8192;                  // most keys gathered from the bracket (expected: 6000 of 131072 at w = N / 4)
constexpr int kHeavy = 128;                    // (of 4096 or 8192 samples, where an ordinary row has ten in its fullest bin)
constexpr int kStreamMinKeys = 4097, kStreamMaxKeys = 1 << 17;        // (more keys than the sample;) two bits per key of a row in shared memory: 32 KB
constexpr int kMaxUnits = kStreamMaxKeys / 1024;
struct alignas(16) StreamShared {
    int hist[2048];
    unsigned long long list[kInside], cand[kCandidates];
    int above[kMaxUnits], inside[kMaxUnits], begin[kMaxUnits];         // per unit: keys above the bracket (later: kept), keys in it, where those begin in the list
    int scan[kSelectWarps];
    uint32_t warp_min[kSelectWarps], warp_max[kSelectWarps];
    int bin[2], in_bin[2], over_bin[2];
    int ncand, listed;
    unsigned long long weakest;
};
static size_t stream_smem(int N) { return sizeof(StreamShared) + (size_t)((N + 1023) / 1024) * 32 * sizeof(uint2); }

template <bool kState, int kSample>
__global__ void __launch_bounds__(kSelectThreads, 2) decode_select_stream_kernel(const float* __restrict__ delta, int64_t ld, int N, int keep,
                                                                              int* __restrict__ list, int64_t list_stride, int* __restrict__ tickets) {
    extern __shared__ __align__(16) uint8_t select_smem[];
    StreamShared& S = *reinterpret_cast<StreamShared*>(select_smem);
    uint2* mask = reinterpret_cast<uint2*>(select_smem + sizeof(StreamShared));    // per 32 keys: above the bracket (later: kept), in it or above
    const int bh = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, units = (N + 1023) / 1024;
    for (int t = tid; t < 2048; t += kSelectThreads) S.hist[t] = 0;
    if (tid < kMaxUnits) S.above[tid] = S.inside[tid] = 0;
    if (tid == 0) { S.ncand = S.listed = 0; S.bin[0] = S.bin[1] = -1; }
    pdl_enter(delta, list, tickets);
    int* out = list + (size_t)bh * list_stride;
    if (tickets && tid == 0) tickets[bh] = 0;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(delta + (size_t)bh * ld);
    auto range = [&](uint32_t& umin, uint32_t& umax) {                   // of the CTA (its barrier)
        umin = __reduce_min_sync(0xffffffffu, umin);
        umax = __reduce_max_sync(0xffffffffu, umax);
        if (lane == 0) { S.warp_min[warp] = umin; S.warp_max[warp] = umax; }
        __syncthreads();
        umin = __reduce_min_sync(0xffffffffu, S.warp_min[lane]);
        umax = __reduce_max_sync(0xffffffffu, S.warp_max[lane]);
    };
    // descending running count of the histogram: this thread's bins are top + 1 and top, `excl` keys lie above them. The bins are zeroed again
    const int top = 2046 - 2 * tid;
    auto scan = [&](int& excl, int2& c) {
        c = *reinterpret_cast<const int2*>(S.hist + top);
        *reinterpret_cast<int2*>(S.hist + top) = make_int2(0, 0);
        int incl = c.x + c.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) S.scan[warp] = incl;
        __syncthreads();
        excl = __reduce_add_sync(0xffffffffu, lane < warp ? S.scan[lane] : 0) + incl - c.x - c.y;
    };
    // the bin that holds rank r (from 1) of what was scanned, how many it holds and how many lie above it
    auto find = [&](int r, int excl, int2 c, int which) {
        if (excl < r && r <= excl + c.x + c.y) {
            const bool first = r <= excl + c.y;
            S.bin[which] = first ? top + 1 : top;
            S.in_bin[which] = first ? c.y : c.x;
            S.over_bin[which] = excl + (first ? 0 : c.y);
        }
    };
    auto shift_of = [](uint32_t width) { return max(0, 21 - __clz((int)width)); };        // 2048 bins over width + 1 patterns
    // the sample: one key of every N / kSample, at a scattered place
    uint32_t lo = 0u, hi = 0x7FFFFFFFu;                                   // keys above hi are kept, keys below lo are not
    {
        uint32_t u[kSample / kSelectThreads], umin = 0x7FFFFFFFu, umax = 0u;
#pragma unroll
        for (int t = 0; t < kSample / kSelectThreads; ++t) {
            const uint32_t i = t * kSelectThreads + tid;
            const uint32_t j = (uint32_t)((uint64_t)i * N / kSample) + (((i * 2654435761u) >> 16) * (uint32_t)(N / kSample) >> 16);
            u[t] = src[j] & 0x7FFFFFFFu;
            umin = min(umin, u[t]);
            umax = max(umax, u[t]);
        }
        range(umin, umax);
        const int shift = shift_of(umax - umin);
#pragma unroll
        for (int t = 0; t < kSample / kSelectThreads; ++t) atomicAdd(&S.hist[(u[t] - umin) >> shift], 1);
        __syncthreads();
        int excl;
        int2 c;
        scan(excl, c);
        const float q = (float)keep / (float)N, mid = q * kSample, dev = 4.5f * sqrtf(mid * (1.0f - q)) + 4.0f;
        const int r0 = (int)(mid - dev), r1 = (int)(mid + dev) + 1;       // ranks (from 1) of the bracket's ends
        find(r0, excl, c, 0);
        find(r1, excl, c, 1);
        __syncthreads();
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
            if (S.bin[e] < 0) continue;                                   // (beyond the sample)
            int sh = shift;
            uint32_t a = umin + ((uint32_t)S.bin[e] << sh), b = a + ((1u << sh) - 1u);
            while (S.in_bin[e] > kHeavy && sh > 0) {
                const int r = (e ? r1 : r0) - S.over_bin[e];
                uint32_t m = 0x7FFFFFFFu, M = 0u;
#pragma unroll
                for (int t = 0; t < kSample / kSelectThreads; ++t)
                    if (u[t] - a <= b - a) { m = min(m, u[t]); M = max(M, u[t]); }
                __syncthreads();                                          // (the last range and bin have been read)
                range(m, M);
                a = m;
                b = M;
                if (m == M) break;
                sh = shift_of(M - m);
#pragma unroll
                for (int t = 0; t < kSample / kSelectThreads; ++t)
                    if (u[t] - m <= M - m) atomicAdd(&S.hist[(u[t] - m) >> sh], 1);
                __syncthreads();
                scan(excl, c);
                const int over = S.over_bin[e];
                __syncthreads();
                find(r, excl, c, e);
                if (excl < r && r <= excl + c.x + c.y) S.over_bin[e] += over;
                __syncthreads();
                a = m + ((uint32_t)S.bin[e] << sh);
                b = min(M, a + ((1u << sh) - 1u));
            }
            if (e) lo = a; else hi = min(b, 0x7FFFFFFFu);
        }
        if (r0 < 1 && lo == umax) hi = lo;                                // (equal weights at an end of the row)
        if (r1 > kSample && hi == umin) lo = hi;
    }
    // f(word, its keys) for the CTA's words of 32 consecutive keys, eight words of a warp requested at once
    auto sweep = [&](auto&& f) {
        const int per = (32 * units + 8 * kSelectWarps - 1) / (8 * kSelectWarps) * 8, w1 = min(32 * units, (warp + 1) * per);
        for (int wb = warp * per; wb < w1; wb += 8) {
            uint32_t u[8];
            const uint32_t* at = src + wb * 32 + lane;
            if (wb * 32 + 256 <= N) {
#pragma unroll
                for (int k = 0; k < 8; ++k) u[k] = at[32 * k] & 0x7FFFFFFFu;
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) u[k] = (wb + k) * 32 + lane < N ? at[32 * k] & 0x7FFFFFFFu : 0xFFFFFFFFu;      // (as an int below every key)
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) f(wb + k, u[k]);
        }
    };
    auto before_lane = [&](int n) {                                       // sum of the lower lanes' n
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        return incl - n;
    };
    int* gathered = reinterpret_cast<int*>(S.list);                       // (the low words: first the key's number, then its order key)
    uint32_t bmin = lo, bmax = hi;                                        // of the keys inside, or wider
    int need, inside;
    for (int turn = 0;; ++turn) {
        const bool again = turn > 0;
        if (turn == 8) return;                                            // (three narrow any bracket to one pattern: weights that change under the call)
        if (again) { bmin = 0x7FFFFFFFu; bmax = 0u; }
        auto bits = [&](int word, uint32_t u) {
            const uint32_t ba = __ballot_sync(0xffffffffu, (int)u > (int)hi), bi = __ballot_sync(0xffffffffu, (int)u >= (int)lo);
            if (lane == 0) mask[word] = make_uint2(ba, bi);
        };
        if (!again) {
            sweep(bits);
        } else {
            sweep([&](int word, uint32_t u) {
                bits(word, u);
                if ((int)u >= (int)lo && u <= hi) { bmin = min(bmin, u); bmax = max(bmax, u); }
            });
        }
        __syncthreads();
        for (int unit = warp; unit < units; unit += kSelectWarps) {
            const uint2 m = mask[32 * unit + lane];
            uint32_t in = m.y & ~m.x;
            const int a = __reduce_add_sync(0xffffffffu, __popc(m.x)), n = __popc(in), before = before_lane(n);
            int at = 0;
            if (lane == 31) {
                S.above[unit] = a;
                S.inside[unit] = before + n;
                S.begin[unit] = at = atomicAdd(&S.listed, before + n);
            }
            at = __shfl_sync(0xffffffffu, at, 31) + before;
            if (lo != hi)
                for (; in && at < kInside; in &= in - 1u) gathered[2 * at++] = (32 * unit + lane) * 32 + __ffs(in) - 1;
        }
        if (again) range(bmin, bmax); else __syncthreads();
        int a = 0, i = 0;
#pragma unroll
        for (int k = 0; k < kMaxUnits; k += 32) { a += S.above[k + lane]; i += S.inside[k + lane]; }
        need = keep - __reduce_add_sync(0xffffffffu, a);
        inside = __reduce_add_sync(0xffffffffu, i);
        if (need >= 1 && need <= inside && (inside <= kInside || bmin == bmax)) break;
        // the bracket is narrowed, or the part of the row beside it that holds the threshold
        if (tid == 0) S.listed = 0;
        int r = need, excl;
        int2 c;
        if (need < 1) { lo = hi + 1u; hi = 0x7FFFFFFFu; r = keep; }
        else if (need > inside) { hi = lo - 1u; lo = 0u; r = need - inside; }
        else if (again) { lo = bmin; hi = bmax; }
        const int shift = shift_of(hi - lo);
        sweep([&](int, uint32_t u) { if (u - lo <= hi - lo) atomicAdd(&S.hist[(u - lo) >> shift], 1); });
        __syncthreads();
        scan(excl, c);
        find(r, excl, c, 0);
        __syncthreads();
        lo += (uint32_t)S.bin[0] << shift;
        hi = min(hi, lo + ((1u << shift) - 1u));
    }
    const bool equal = bmin == bmax;                                      // one bit pattern: the first `need` keys inside are kept
    // f(unit, place of its first key among all that `count` counts) for this warp's units
    auto each_unit = [&](const int* count, auto&& f) {
        int run = 0;
        for (int k = 0; k < units; k += 32) {
            const int v = count[k + lane], before = __reduce_add_sync(0xffffffffu, lane < warp ? v : 0);
            if (k + warp < units) f(k + warp, run + before);
            run += __reduce_add_sync(0xffffffffu, v);
        }
    };
    uint32_t* kept_of = reinterpret_cast<uint32_t*>(S.hist);              // one bit per gathered key: kept
    if (!equal) {
        bmin = 0x7FFFFFFFu;
        bmax = 0u;
        for (int e0 = tid; e0 < inside; e0 += 4 * kSelectThreads) {       // four keys of a thread requested at once
            int j[4];
            uint32_t u[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int e = e0 + t * kSelectThreads;
                j[t] = e < inside ? gathered[2 * e] : 0;
                u[t] = src[j[t]] & 0x7FFFFFFFu;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int e = e0 + t * kSelectThreads;
                if (e < inside) {
                    bmin = min(bmin, u[t]);
                    bmax = max(bmax, u[t]);
                    S.list[e] = key_of(__uint_as_float(u[t]), j[t]);
                }
            }
        }
        range(bmin, bmax);
        auto each = [&](auto&& f) {                                       // the bracket's keys
            for (int e = tid; e < inside; e += kSelectThreads) f(S.list[e]);
        };
        // the bin of the need-th, by weight, among equal weights by index
        unsigned long long base = (unsigned long long)bmin << 32;
        int s = 32 + shift_of(bmax - bmin), nbins = 2048, count;
        for (;;) {
            each([&](unsigned long long x) {
                const unsigned long long bin = (x - base) >> s;
                if (bin < (unsigned long long)nbins) atomicAdd(&S.hist[bin], 1);
            });
            __syncthreads();
            int excl;
            int2 c;
            scan(excl, c);
            find(need, excl, c, 0);
            __syncthreads();
            base += (unsigned long long)(uint32_t)S.bin[0] << s;
            need -= S.over_bin[0];
            count = S.in_bin[0];
            if (count <= kCandidates) break;
            if (s > 32) {                                                 // the next bins cover this one and nothing above it
                nbins = 1 << min(11, s - 32);
                s = max(32, s - 11);
            } else {                                                      // one weight: the low words of N <= 2^17 keys, 64 to a bin
                base += 0xFFFFFFFFu - (uint32_t)(N - 1);
                nbins = 2048;
                s = 6;
            }
        }
        each([&](unsigned long long x) { if ((x - base) >> s == 0ull) S.cand[atomicAdd(&S.ncand, 1)] = x; });
        __syncthreads();
        if (tid < count) {
            const unsigned long long k = S.cand[tid];
            int above = 0;
            for (int i = 0; i < count; ++i) above += S.cand[i] > k;
            if (above == need - 1) S.weakest = k;
        }
        __syncthreads();
        const unsigned long long weakest = S.weakest;
        for (int e = tid; e - lane < inside; e += kSelectThreads) {
            const uint32_t k = __ballot_sync(0xffffffffu, e < inside && S.list[e] >= weakest);
            if (lane == 0) kept_of[e >> 5] = k;
        }
    }
    __syncthreads();
    // the kept keys' bits
    if (equal) each_unit(S.inside, [&](int unit, int at) { S.begin[unit] = at; });         // (by index)
    __syncwarp();
    for (int unit = warp; unit < units; unit += kSelectWarps) {
        const uint2 m = mask[32 * unit + lane];
        uint32_t in = m.y & ~m.x, word = m.x;
        const int n = __popc(in), at = S.begin[unit] + before_lane(n);
        uint32_t keep_bits;                                               // of the word's n keys inside
        if (equal) {
            const int k = min(max(need - at, 0), n);
            keep_bits = k == 32 ? 0xFFFFFFFFu : (1u << k) - 1u;
            if (kState && at < need && need <= at + n) {                  // the weakest kept key
                uint32_t rest = in;
                for (int t = need - at; t > 1; --t) rest &= rest - 1u;
                S.weakest = key_of(__uint_as_float(bmin), (32 * unit + lane) * 32 + __ffs(rest) - 1);
            }
        } else {
            keep_bits = __funnelshift_r(kept_of[at >> 5], kept_of[(at >> 5) + 1], at & 31);
            if (n < 32) keep_bits &= (1u << n) - 1u;
        }
        if (keep_bits == (n == 32 ? 0xFFFFFFFFu : (1u << n) - 1u)) {
            word |= in;
        } else {
            for (; keep_bits; keep_bits >>= 1, in &= in - 1u)
                if (keep_bits & 1u) word |= in & -in;
        }
        mask[32 * unit + lane].x = word;
        const int kept = __reduce_add_sync(0xffffffffu, __popc(word));
        if (lane == 0) S.above[unit] = kept;
    }
    __syncthreads();
    // the bits -> indices
    constexpr int kTurn = 2 * kInside / kSelectWarps;
    int* buf = reinterpret_cast<int*>(S.list) + warp * kTurn;             // (its keys have been read)
    const uint32_t below = (1u << lane) - 1u;
    const unsigned long long weakest = kState ? S.weakest : 0ull;
    const int last = (int)(0xFFFFFFFFu - (uint32_t)weakest);
    each_unit(S.above, [&](int unit, int at) {
        uint32_t word = mask[32 * unit + lane].x;
        int pos = before_lane(__popc(word));
        const int all = __shfl_sync(0xffffffffu, pos + __popc(word), 31), j0 = (32 * unit + lane) * 32;
        if (kState && last >> 5 == 32 * unit + lane) {
            int* hdr = out - kStateHeader;
            hdr[0] = keep;
            hdr[1] = at + pos + __popc(word & ((1u << (last & 31)) - 1u));
            hdr[2] = (int)(uint32_t)weakest;
            hdr[3] = (int)(uint32_t)(weakest >> 32);
        }
        if (all > kTurn) {                                                // a lane per key: whole lines as they are
            for (int w = 0; w < 32; ++w) {
                const uint32_t b = __shfl_sync(0xffffffffu, word, w);
                const int p = at + __shfl_sync(0xffffffffu, pos, w);
                if ((b >> lane) & 1u) out[p + __popc(b & below)] = (32 * unit + w) * 32 + lane;
            }
        } else {                                                          // a lane per word: the short runs meet in shared memory and leave as whole lines
            for (; word; word &= word - 1u) buf[pos++] = j0 + __ffs(word) - 1;
            __syncwarp();
            for (int i = lane; i < all; i += 32) out[at + i] = buf[i];
            __syncwarp();
        }
    });
}

// 16 bytes of a K, V or q row, widened to fp32
template <typename T> struct Wide;
template <> struct Wide<float> {
    static constexpr int kN = 4;
    static __device__ __forceinline__ void get(const uint4& a, float (&v)[4]) {
        v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y); v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
    }
};
template <> struct Wide<__nv_bfloat16> {
    static constexpr int kN = 8;
    static __device__ __forceinline__ void get(const uint4& a, float (&v)[8]) {
        const uint32_t u[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(u[i] << 16);
            v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
        }
    }
};

// Sum over the LPR lanes of a row group of eight per-lane partials: after three levels in which a lane keeps half of its
// values and hands the other half to its partner, lane `sub` holds the sum of value bitrev(sub & 7). 7 + log2(LPR / 8)
// shuffles for eight rows.
template <int LPR>
__device__ __forceinline__ float reduce8(float (&p)[8], int sub) {
#pragma unroll
    for (int m = 1, keep = 4; m < 8; m <<= 1, keep >>= 1) {
        const bool up = (sub & m) != 0;
#pragma unroll
        for (int q = 0; q < keep; ++q) {
            const float stay = up ? p[q + keep] : p[q], give = up ? p[q] : p[q + keep];
            p[q] = stay + __shfl_xor_sync(0xffffffffu, give, m);
        }
    }
#pragma unroll
    for (int m = 8; m < LPR; m <<= 1) p[0] += __shfl_xor_sync(0xffffffffu, p[0], m);
    return p[0];
}
__device__ __forceinline__ int bitrev3(int x) { return ((x & 1) << 2) | (x & 2) | ((x >> 2) & 1); }

// The attention part shared by the two decoding kernels: `list` (shared memory) holds `count` key indices of this CTA;
// partial [D + 2]: o (unnormalised, relative to m), m (log2 domain), l.
// A step's attention is a gather of 2 * D * sizeof(T) bytes per kept key, bound by how many of those bytes are in flight, so
// a warp takes batches of eight 16-byte K loads AND eight V loads per lane (bf16, D = 128: 16 keys, 8 KB per warp) issued
// back to back, and spends few instructions per key: one transposing reduction and one exponential per lane for the whole
// batch. Measured against the form before (8 bytes per lane, four keys in flight, five shuffles and two exponentials in every
// lane per key): 256 rows of 4096 kept keys in 65536 (537 MB of rows) 254 -> 99 us, 5.4 TB/s; 32 rows of 2048 in 16384,
// 21 -> 8 us; a step with a carried state 12.2 -> 7 us.
template <typename T, int D>
__device__ __forceinline__ void decode_attend(const int* list, int count, const T* __restrict__ q, const T* __restrict__ K,
                                              const T* __restrict__ V, const float* __restrict__ dl, float* __restrict__ out,
                                              int bh, int b, int hk, float scale_log2, int64_t ks_b, int64_t ks_l, int64_t ks_h,
                                              int64_t vs_b, int64_t vs_l, int64_t vs_h) {
    constexpr int CPL = Wide<T>::kN;           // channels per lane
    constexpr int LPR = D / CPL;               // lanes per key row
    constexpr int RPI = 32 / LPR;              // key rows per warp instruction
    constexpr int kBatch = 8 * RPI;            // keys a warp takes at a time
    __shared__ __align__(16) float s_part[8][D + 4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sub = lane % LPR, grp = lane / LPR;
    float qv[CPL];
    Wide<T>::get(*reinterpret_cast<const uint4*>(q + (size_t)bh * D + sub * CPL), qv);
    float m = -INFINITY, l = 0.0f, o[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) o[c] = 0.0f;
    const T* Kb = K + b * ks_b + hk * ks_h + sub * CPL;
    const T* Vb = V + b * vs_b + hk * vs_h + sub * CPL;
    const int mine = bitrev3(sub & 7) * RPI + grp;                 // the key of the batch whose score ends up in this lane
    for (int base = warp * kBatch; base < count; base += 8 * kBatch) {
        uint4 kr[8], vr[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {                              // (entries beyond the list repeat its last key)
            const int64_t j = list[min(base + u * RPI + grp, count - 1)];
            kr[u] = __ldg(reinterpret_cast<const uint4*>(Kb + j * ks_l));
            vr[u] = __ldg(reinterpret_cast<const uint4*>(Vb + j * vs_l));
        }
        const bool real = base + mine < count;
        const float bias = dl[list[min(base + mine, count - 1)]];
        float p[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            float kv[CPL], a = 0.0f;
            Wide<T>::get(kr[u], kv);
#pragma unroll
            for (int c = 0; c < CPL; ++c) a = fmaf(qv[c], kv[c], a);
            p[u] = a;
        }
        const float s = reduce8<LPR>(p, sub);
        const float x = real ? fmaf(s, scale_log2, bias * 1.4426950408889634f) : -INFINITY;
        float mx = x;
#pragma unroll
        for (int mm = 1; mm < 32; mm <<= 1)
            if (mm < 8 || mm >= LPR) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, mm));
        const float m_new = fmaxf(m, mx), m_use = m_new == -INFINITY ? 0.0f : m_new;
        const float f = exp2f(m - m_use), w = exp2f(x - m_use);
        m = m_new;
        l = l * f + (sub < 8 ? w : 0.0f);                          // (lanes 8 and up of a row group repeat the first eight)
#pragma unroll
        for (int c = 0; c < CPL; ++c) o[c] *= f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float wu = __shfl_sync(0xffffffffu, w, grp * LPR + bitrev3(u));
            float vv[CPL];
            Wide<T>::get(vr[u], vv);
#pragma unroll
            for (int c = 0; c < CPL; ++c) o[c] = fmaf(wu, vv[c], o[c]);
        }
    }
    // the row groups of a warp share m: plain sums; then the warps are combined in shared memory
#pragma unroll
    for (int mm = LPR; mm < 32; mm <<= 1)
#pragma unroll
        for (int c = 0; c < CPL; ++c) o[c] += __shfl_xor_sync(0xffffffffu, o[c], mm);
#pragma unroll
    for (int mm = 1; mm < 32; mm <<= 1) l += __shfl_xor_sync(0xffffffffu, l, mm);
    if (grp == 0) {
#pragma unroll
        for (int c = 0; c < CPL; c += 4) *reinterpret_cast<float4*>(&s_part[warp][sub * CPL + c]) = make_float4(o[c], o[c + 1], o[c + 2], o[c + 3]);
        if (sub == 0) { s_part[warp][D] = m; s_part[warp][D + 1] = l; }
    }
    __syncthreads();
    float mx = -INFINITY;
#pragma unroll
    for (int wq = 0; wq < 8; ++wq) mx = fmaxf(mx, s_part[wq][D]);
    for (int c = tid; c < D + 2; c += kAttnThreads) {
        if (c == D) { out[c] = mx; continue; }
        float acc = 0.0f;
#pragma unroll
        for (int wq = 0; wq < 8; ++wq) {
            const float mw = s_part[wq][D];
            const float f = mw == -INFINITY ? 0.0f : exp2f(mw - mx);
            acc += s_part[wq][c] * f;                 // c == D + 1 is l
        }
        out[c] = acc;
    }
}

// The row's partials -> o, log-sum-exp; every thread of a 256-thread CTA takes part: warp g takes the splits s = g, g + 8, ...
// with D / 32 channels per lane, then the eight warps are merged in shared memory. The partials come from other CTAs: read at L2.
template <typename T, int D>
__device__ __forceinline__ void combine_row(const float* __restrict__ partial, T* __restrict__ o, float* __restrict__ lse, int nsplit, int bh) {
    constexpr int CPL = D / 32;                // channels per lane
    __shared__ float s_m[8], s_l[8], s_o[8][D];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const float* p = partial + (size_t)bh * nsplit * (D + 2);
    float mx = -INFINITY, l = 0.0f, acc[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) acc[c] = 0.0f;
    constexpr int kBatch = 4;                  // splits of a warp whose loads are in flight together (the maxima first, then the sums: one more round trip to L2)
    for (int s0 = g; s0 < nsplit; s0 += 8 * kBatch) {
        float ms[kBatch], ls[kBatch], as[kBatch][CPL], m = mx;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float* ps = p + (size_t)(s0 + 8 * u) * (D + 2);
            const bool in = s0 + 8 * u < nsplit;
            ms[u] = in ? __ldcg(&ps[D]) : -INFINITY;
            ls[u] = in ? __ldcg(&ps[D + 1]) : 0.0f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) as[u][c] = in ? __ldcg(&ps[lane * CPL + c]) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) m = fmaxf(m, ms[u]);
        if (mx != -INFINITY) {
            const float f = exp2f(mx - m);
            l *= f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) acc[c] *= f;
        }
        mx = m;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float f = ms[u] == -INFINITY ? 0.0f : exp2f(ms[u] - mx);
            l += ls[u] * f;
#pragma unroll
            for (int c = 0; c < CPL; ++c) acc[c] += as[u][c] * f;
        }
    }
#pragma unroll
    for (int c = 0; c < CPL; ++c) s_o[g][lane * CPL + c] = acc[c];
    if (lane == 0) { s_m[g] = mx; s_l[g] = l; }
    __syncthreads();
    if (threadIdx.x < D) {
        const int c = threadIdx.x;
        float m_all = -INFINITY;
#pragma unroll
        for (int q = 0; q < 8; ++q) m_all = fmaxf(m_all, s_m[q]);
        float lt = 0.0f, at = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float f = s_m[q] == -INFINITY ? 0.0f : exp2f(s_m[q] - m_all);
            lt += s_l[q] * f;
            at += s_o[q][c] * f;
        }
        const float v = lt > 0.0f ? at / lt : 0.0f;
        if constexpr (sizeof(T) == 2) o[(size_t)bh * D + c] = __float2bfloat16_rn(v); else o[(size_t)bh * D + c] = v;
        if (c == 0) lse[bh] = lt > 0.0f ? 0.6931471805599453f * (m_all + log2f(lt)) : -INFINITY;
    }
}

// Called by every thread of an attention CTA after its partial is written: the CTA that finishes its row last (a ticket
// counter, which it resets for the next call; nobody waits) combines the row. Returns true in that CTA.
__device__ __forceinline__ bool last_of_row(int* ticket, int nsplit) {
    __shared__ int s_last;
    __syncthreads();                                   // every thread's part of the partial is written ...
    if (threadIdx.x == 0) {
        __threadfence();                               // ... and visible device-wide before the ticket is taken (the fence is cumulative)
        const int t = atomicAdd(ticket, 1);
        s_last = t == nsplit - 1;
        if (s_last) {
            *ticket = 0;
            __threadfence();                           // the other CTAs' partials, published before their tickets, are visible from here on
        }
    }
    __syncthreads();
    return s_last != 0;
}

// One CTA per (row, split of `per_split` entries of the row's kept list).
template <typename T, int D>
__global__ void __launch_bounds__(kAttnThreads, 2) decode_attn_kernel(const T* __restrict__ q, const T* __restrict__ K, const T* __restrict__ V,
                                                                      const float* __restrict__ delta, int64_t ld,
                                                                      const int* __restrict__ kept, int64_t kept_stride, float* __restrict__ partial,
                                                                      int keep, int per_split, int Hq, int G, float scale_log2, int nsplit,
                                                                      int64_t ks_b, int64_t ks_l, int64_t ks_h, int64_t vs_b, int64_t vs_l,
                                                                      int64_t vs_h, int* __restrict__ tickets, T* __restrict__ o,
                                                                      float* __restrict__ lse) {
    __shared__ int list[kMaxSplit];
    const int split = blockIdx.x, bh = blockIdx.y, b = bh / Hq, h = bh % Hq, hk = h / G;
    const int e0 = split * per_split, count = min(per_split, keep - e0);
    pdl_enter(q, K, V, delta, kept, partial, tickets, o, lse);
    for (int e = threadIdx.x; e < count; e += kAttnThreads) list[e] = kept[(size_t)bh * kept_stride + e0 + e];
    __syncthreads();
    decode_attend<T, D>(list, count, q, K, V, delta + (size_t)bh * ld, partial + ((size_t)bh * nsplit + split) * (D + 2), bh, b, hk, scale_log2,
                        ks_b, ks_l, ks_h, vs_b, vs_l, vs_h);
    if (last_of_row(tickets + bh, nsplit)) combine_row<T, D>(partial, o, lse, nsplit, bh);
}

// ---- incremental decoding: the kept set is carried from step to step --------------------------------------------------
// One key is appended per step, so the set of the w best keys changes by at most one member: the new key enters iff it
// beats the weakest kept key (or the set is not full yet), and that weakest key leaves. The state of a (batch, head) row:
//   int32 [0] count (<= w)   [1] position of the weakest kept key in the list   [2..3] its 64-bit sort key
//         [4..7] unused
//   int32 [8 .. 8 + w)       the kept key indices, in no particular order
// A step costs O(w), whatever the number of cached keys: no scan of the delta row.
constexpr int kListSplit = 256;                     // most kept keys per CTA of the list attention kernel (list_split)

__device__ __forceinline__ int state_stride(int w_cap) { return kStateHeader + ((w_cap + 3) & ~3); }

// what the appended key does to a row's set (hdr: count, position and order key of the weakest kept key): 0 nothing, 1 appended (set not full), 2 replaces the weakest
__device__ __forceinline__ int step_mode(const int4& hdr, int w_cap, unsigned long long kn) {
    if (hdr.x < w_cap) return 1;
    const unsigned long long kmin = ((unsigned long long)(unsigned)hdr.w << 32) | (unsigned)hdr.z;
    return kn > kmin ? 2 : 0;
}

// weakest key of the row's list (entry `skip_pos`, if >= 0, reads as key `skip_j`): written to the header by thread 0
__device__ __forceinline__ void store_weakest(int* hdr, const int* kept, int count, const float* dl, int skip_pos, int skip_j) {
    __shared__ unsigned long long s_key[32];
    __shared__ int s_pos[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    unsigned long long best = ~0ull;
    int pos = -1;
    for (int i = tid; i < count; i += blockDim.x) {
        const int j = i == skip_pos ? skip_j : kept[i];
        const unsigned long long k = key_of(dl[j], j);
        if (k < best) { best = k; pos = i; }
    }
    for (int o = 16; o; o >>= 1) {
        const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int p2 = __shfl_xor_sync(0xffffffffu, pos, o);
        if (k2 < best) { best = k2; pos = p2; }
    }
    if (lane == 0) { s_key[warp] = best; s_pos[warp] = pos; }
    __syncthreads();
    if (tid == 0) {
        for (int wq = 1; wq < nwarp; ++wq)
            if (s_key[wq] < best) { best = s_key[wq]; pos = s_pos[wq]; }
        hdr[1] = pos;
        hdr[2] = (int)(uint32_t)best;
        hdr[3] = (int)(uint32_t)(best >> 32);
    }
}

// The weakest key of one split's list: what the attention kernel's CTAs leave for the state's update (`pos`: its place in the row's list)
struct alignas(16) Weakest {
    unsigned long long key;
    int pos, unused;
};

// What the update of a row's state reads, requested before the row is combined
struct StepState {
    int4 hdr;                  // count, position and order key of the weakest kept key
    float delta_new;
    uint4 weak;                // lane s < 32: the weakest key of list s (Weakest)
    __device__ __forceinline__ void load(const float* dl, const int* row, const Weakest* w, int N, int nsplit) {
        hdr = *reinterpret_cast<const int4*>(row);
        delta_new = dl[N - 1];
        weak = w && (int)threadIdx.x < min(32, nsplit) ? *reinterpret_cast<const uint4*>(w + threadIdx.x) : make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0u, 0u);
    }
};

// brings a row's state up to date with the appended key N - 1 (every thread of the CTA takes part, and has loaded x before a barrier). weak: the weakest keys of the
// row's nsplit lists (NULL: the kept keys are scanned)
__device__ __forceinline__ void decode_state_update(const StepState& x, const float* dl, int N, int w_cap, int* hdr, const Weakest* weak, int nsplit) {
    int* kept = hdr + kStateHeader;
    const int newj = N - 1, count = x.hdr.x, weakest = x.hdr.y;
    const unsigned long long kn = key_of(x.delta_new, newj), kmin = ((unsigned long long)(unsigned)x.hdr.w << 32) | (unsigned)x.hdr.z;
    const int mode = step_mode(x.hdr, w_cap, kn);
    if (mode == 0) return;
    if (mode == 1) {                                   // the appended key has the largest index: on equal delta it is the weakest
        if (threadIdx.x == 0) {
            kept[count] = newj;
            hdr[0] = count + 1;
            if (count == 0 || kn < kmin) { hdr[1] = count; hdr[2] = (int)(uint32_t)kn; hdr[3] = (int)(uint32_t)(kn >> 32); }
        }
        return;
    }
    if (weak) {
        if (threadIdx.x < 32) {
            unsigned long long best = (unsigned long long)x.weak.y << 32 | x.weak.x;
            int pos = (int)x.weak.z;
            for (int s = threadIdx.x + 32; s < nsplit; s += 32)
                if (weak[s].key < best) { best = weak[s].key; pos = weak[s].pos; }
            for (int o = 16; o; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, best, o);
                const int p2 = __shfl_xor_sync(0xffffffffu, pos, o);
                if (k2 < best) { best = k2; pos = p2; }
            }
            if (threadIdx.x == 0) {
                hdr[1] = pos;
                hdr[2] = (int)(uint32_t)best;
                hdr[3] = (int)(uint32_t)(best >> 32);
            }
        }
    } else {
        store_weakest(hdr, kept, count, dl, weakest, newj);
    }
    if (threadIdx.x == 0) kept[weakest] = newj;
}

// attention over the row's kept list as it is AFTER the appended key N - 1 is taken into account (the stored state still
// describes the first N - 1 keys; decode_step_combine_kernel brings it up to date afterwards)
template <typename T, int D, int kSplit>
__global__ void __launch_bounds__(kAttnThreads, 2) decode_list_attn_kernel(const T* __restrict__ q, const T* __restrict__ K,
                                                                        const T* __restrict__ V, const float* __restrict__ delta,
                                                                        int64_t ld, const int* __restrict__ state, int w_cap,
                                                                        float* __restrict__ partial, int N, int Hq, int G,
                                                                        float scale_log2, int nsplit, int64_t ks_b, int64_t ks_l,
                                                                        int64_t ks_h, int64_t vs_b, int64_t vs_l, int64_t vs_h,
                                                                        Weakest* __restrict__ weak) {
    __shared__ int list[kSplit];
    __shared__ unsigned long long s_key[kSplit / 32];
    __shared__ int s_pos[kSplit / 32];
    const int split = blockIdx.x, bh = blockIdx.y, b = bh / Hq, h = bh % Hq, hk = h / G;
    const int tid = threadIdx.x;
    pdl_enter(q, K, V, delta, state, partial, weak);
    const float* dl = delta + (size_t)bh * ld;
    const int* hdr = state + (size_t)bh * state_stride(w_cap);
    const int* kept = hdr + kStateHeader;
    const int4 head = *reinterpret_cast<const int4*>(hdr);
    const int newj = N - 1, count = head.x;
    const int e = split * kSplit + tid;
    const int held = tid < kSplit && e < w_cap ? kept[e] : 0;          // (in flight together with the header)
    const int mode = step_mode(head, w_cap, key_of(dl[newj], newj));
    const int eff = count + (mode == 1 ? 1 : 0), weakest = head.y;
    const int mine = (e >= count || (mode == 2 && e == weakest)) ? newj : held;
    if (tid < kSplit && e < eff) list[tid] = mine;
    // When the appended key replaces the weakest one, the new weakest is found here, where the kept keys are read anyway: the combine kernel
    // scanned them again, two dependent loads at the end of the step (32 rows of 2048 kept keys, step of a captured loop 12.5 -> 11.4 us; 32 rows of 3000, 14.1 -> 11.8)
    if (weak && mode == 2 && tid < kSplit) {
        unsigned long long best = e < eff ? key_of(dl[mine], mine) : ~0ull;
        int pos = e;
        for (int o = 16; o; o >>= 1) {
            const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, best, o);
            const int p2 = __shfl_xor_sync(0xffffffffu, pos, o);
            if (k2 < best) { best = k2; pos = p2; }
        }
        if ((tid & 31) == 0) { s_key[tid >> 5] = best; s_pos[tid >> 5] = pos; }
    }
    __syncthreads();
    if (weak && mode == 2 && tid == 0) {
        Weakest x = {s_key[0], s_pos[0], 0};
        for (int g = 1; g < kSplit / 32; ++g)
            if (s_key[g] < x.key) { x.key = s_key[g]; x.pos = s_pos[g]; }
        weak[(size_t)bh * nsplit + split] = x;
    }
    decode_attend<T, D>(list, max(0, min(kSplit, eff - split * kSplit)), q, K, V, dl,
                        partial + ((size_t)bh * nsplit + split) * (D + 2), bh, b, hk, scale_log2, ks_b, ks_l, ks_h, vs_b, vs_l, vs_h);
}

// The step's second kernel, one CTA of 8 D threads per row: the splits' partials -> o, log-sum-exp, and then, every CTA of
// the attention kernel having read the row's state, the state takes in the appended key. (Doing this in the attention
// kernel's last CTA per row, as dma_decode does, was measured slower here, 16.5 -> 20.7 us per step: the state must then be
// writable in the attention kernel, whose loads of the kept list no longer take the read-only path, and the update, which
// scans the w kept keys, runs on 256 threads at the end of the row's critical path instead of 8 D.)
template <typename T, int D, int kBatch>
__global__ void __launch_bounds__(8 * D) decode_step_combine_kernel(const float* __restrict__ partial, T* __restrict__ o, float* __restrict__ lse,
                                                                    int nsplit, const float* __restrict__ delta, int64_t ld,
                                                                    int N, int w_cap, int* __restrict__ state, const Weakest* __restrict__ weak) {
    __shared__ float s_m[8], s_l[8], s_o[8][D];
    const int bh = blockIdx.x, c = threadIdx.x % D, g = threadIdx.x / D;     // group g takes the splits s = g, g + 8, ...
    pdl_enter(partial, o, lse, delta, state, weak);
    const float* p = partial + (size_t)bh * nsplit * (D + 2);
    const float* dl = delta + (size_t)bh * ld;
    int* hdr = state + (size_t)bh * state_stride(w_cap);
    const Weakest* wk = weak ? weak + (size_t)bh * nsplit : nullptr;
    // Everything the step needs is requested at once: the group's first kBatch splits, the header, the appended key's weight and the lists' weakest keys. (The maxima,
    // then the sums, then the state, each a round trip to L2 behind the one before: 16 captured steps of 32 rows of 2048 kept keys 147 -> 134 us, of one row 101 -> 91, of 16 rows of
    // 4973 164 -> 141.)
    StepState x;
    x.load(dl, hdr, wk, N, nsplit);
    float mx = -INFINITY, l = 0.0f, acc = 0.0f;
    for (int s0 = g; s0 < nsplit; s0 += 8 * kBatch) {
        float ms[kBatch], ls[kBatch], as[kBatch], m = mx;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float* ps = p + (size_t)(s0 + 8 * u) * (D + 2);
            const bool in = s0 + 8 * u < nsplit;
            ms[u] = in ? ps[D] : -INFINITY;
            ls[u] = in ? ps[D + 1] : 0.0f;
            as[u] = in ? ps[c] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) m = fmaxf(m, ms[u]);
        if (s0 != g && mx != -INFINITY) {
            const float f = exp2f(mx - m);
            l *= f;
            acc *= f;
        }
        mx = m;
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const float f = ms[u] == -INFINITY ? 0.0f : exp2f(ms[u] - mx);
            l += ls[u] * f;
            acc += as[u] * f;
        }
    }
    s_o[g][c] = acc;
    if (c == 0) { s_m[g] = mx; s_l[g] = l; }
    __syncthreads();
    if (g == 0) {
        float m_all = -INFINITY;
#pragma unroll
        for (int q = 0; q < 8; ++q) m_all = fmaxf(m_all, s_m[q]);
        float lt = 0.0f, at = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float f = s_m[q] == -INFINITY ? 0.0f : exp2f(s_m[q] - m_all);
            lt += s_l[q] * f;
            at += s_o[q][c] * f;
        }
        const float v = lt > 0.0f ? at / lt : 0.0f;
        if constexpr (sizeof(T) == 2) o[(size_t)bh * D + c] = __float2bfloat16_rn(v); else o[(size_t)bh * D + c] = v;
        if (c == 0) lse[bh] = lt > 0.0f ? 0.6931471805599453f * (m_all + log2f(lt)) : -INFINITY;
    }
    // incremental decoding: the attention kernel has read the row's state, which can now take in the appended key
    decode_state_update(x, dl, N, w_cap, hdr, wk, nsplit);
}



// Splits of a row's kept list: few enough that all CTAs are resident at once (two per SM), which matters when a step is
// short, but no longer than kMaxSplit keys, so that a large batch still comes in waves that balance.
constexpr int kResident = 2 * 148;
int split_keys(const Prob& P) {
    const int64_t bh = (int64_t)P.B * P.Hq;
    int per = kMinSplit;
    while (per < kMaxSplit && bh * ((P.w + per - 1) / per) > kResident) per += kMinSplit;
    return per;
}
// The kept keys per row that a workspace is sized for: the window, whatever the cached length, so that a loop may take its workspace
// at any step; a window beyond 2^20 (2^31 - 1: "keep all") stands for the cached length.
int held_keys(const Prob& P) { return P.w_cap <= 1 << 20 ? P.w_cap : P.w; }

// The most splits of all rows that a call with at most `keep` kept keys and at most P.B * P.Hq rows has. (The splits of one call
// fall where a longer list takes longer splits.)
size_t most_splits(const Prob& P, int keep) {
    const size_t bh = (size_t)P.B * P.Hq, few = bh * ((keep + kMinSplit - 1) / kMinSplit), many = bh * ((keep + kMaxSplit - 1) / kMaxSplit);
    return std::max(std::min(few, (size_t)kResident), many);
}

template <typename T, int D>
int launch_typed(const Prob& P, const void* q, const void* K, const void* V, const float* delta, int64_t ld, void* o, float* lse,
                 const int* kept, int64_t kept_stride, int* tickets, float* partial, cudaStream_t st) {
    const int per = split_keys(P), nsplit = (P.w + per - 1) / per;
    return launch_overlapped(decode_attn_kernel<T, D>, dim3(nsplit, P.B * P.Hq), dim3(kAttnThreads), 0, st, 1, (const T*)q, (const T*)K, (const T*)V,
                             delta, ld, kept, kept_stride, partial, P.w, per, P.Hq, P.G, P.scale * 1.4426950408889634f, nsplit, P.ks[0], P.ks[1],
                             P.ks[2], P.vs[0], P.vs[1], P.vs[2], tickets, (T*)o, lse);
}

}  // namespace

// Kept keys per CTA of a step with the carried state: 128 where all CTAs have an SM to themselves, else 256, two batches per warp.
// Eight captured steps, us, 128 / 256 keys: one row of w = 2048 70 / 74, 8 rows of 256 66 / 72, 16 rows of 1024 (128 CTAs) 72 /
// 76, but 16 rows of 2048 (256 CTAs) 96 / 96, one row of 32768 182 / 162, 32 rows of 2048 121 / 111, 256 rows of 4096 1127 / 926.
static int list_split(const Prob& P) {
    const int64_t ctas = (int64_t)P.B * P.Hq * ((held_keys(P) + kMinSplit - 1) / kMinSplit);
    return ctas <= 148 ? kMinSplit : kListSplit;
}
// the most splits of all rows that a step with at most `keep` kept keys and at most P.B * P.Hq rows has
static size_t most_list_splits(const Prob& P, int keep) {
    const size_t bh = (size_t)P.B * P.Hq;
    return std::max(std::min(bh * ((keep + kMinSplit - 1) / kMinSplit), (size_t)148), bh * ((keep + kListSplit - 1) / kListSplit));
}

// header | tickets | kept lists | partials of the larger of the two attention kernels' split counts
struct DecodeWs {
    int* tickets;
    int* kept;
    float* partial;
    size_t bytes;              // no fewer than for any shorter cache and smaller batch
};
static DecodeWs decode_ws(const Prob& P, void* ws) {
    const size_t bh = (size_t)P.B * P.Hq;
    const int keep = held_keys(P);
    const size_t splits = std::max(most_splits(P, keep), most_list_splits(P, keep));
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    DecodeWs w;
    size_t off = kWsHeaderBytes;
    char* base = (char*)ws;
    w.tickets = reinterpret_cast<int*>(base + off); off += up(bh * sizeof(int));
    w.kept = reinterpret_cast<int*>(base + off); off += up(bh * keep * sizeof(int));
    w.partial = reinterpret_cast<float*>(base + off); off += splits * (P.d + 2) * sizeof(float);
    w.bytes = off;
    return w;
}

size_t decode_ws_bytes(const Prob& P) {
    char dummy[1];
    return decode_ws(P, dummy).bytes;
}

size_t decode_state_bytes(const Prob& P) {
    return (size_t)P.B * P.Hq * (kStateHeader + ((P.w_cap + 3) & ~3)) * sizeof(int);
}

// The selection: kept indices of every row, ascending, to list (rows list_stride entries apart). `state`: list points into
// an incremental state, whose row headers are written too.
static int launch_select(const Prob& P, const float* delta, int64_t ld, int* list, int64_t list_stride, int* tickets, bool state, cudaStream_t st) {
    int nrank = 1;
    // the fewest CTAs whose registers hold a row; a row that needs a cluster gets more while all rows still run at once
    while (nrank < kSelectMaxCluster && ((int64_t)nrank * kCtaKeys < P.L || (nrank > 1 && 2ll * nrank * P.B * P.Hq <= 148))) nrank *= 2;
    // The kernel that streams a row: where the rows do not all have an SM's registers to themselves, or one CTA holds a row of more than 16384 keys. State taken up, us, registers / streamed, at w = 64, N / 16,
    // N / 4, N / 2, N - 1: 200 rows of 8192 keys 13.8 / 11.0 .. 14.3 / 11.9, 256 of 16384 15.1 / 13.0, 16.9 / 14.3, 17.4 / 15.9, 17.4 / 16.9, 15.7 / 14.7, 32 of 26000 12.4 / 10.2 .. 12.3 / 12.3, 512 of
    // 5000 26 / 18 .. 27 / 21; equal weights and ten values gain more (256 of 16384 15 / 12, 23 / 13), weights that rise along the row lose up to 8 % (32 of 32768 12.4 / 12.8). But 32 rows of 16384
    // 8.2 / 8.4 .. 9.8 / 10.7, rising 8.2 / 10.5; 32 of 65536 (clusters) 11.5 / 14.9 .. 14.8 / 22.5; 512 of 4096 (four keys to a thread, two CTAs per SM) 15.0 / 18.1 .. 15.9 / 20.7.
    const int64_t rows = (int64_t)P.B * P.Hq;
    if (P.w < P.L && P.L >= kStreamMinKeys && P.L <= kStreamMaxKeys && (rows * nrank > 148 || (P.L > 16384 && nrank == 1))) {
        auto stream = P.L > 65536 ? (state ? decode_select_stream_kernel<true, 8192> : decode_select_stream_kernel<false, 8192>)
                                  : (state ? decode_select_stream_kernel<true, 4096> : decode_select_stream_kernel<false, 4096>);
        // (state of the function, which other threads' calls share: always the limit)
        if (cudaFuncSetAttribute(stream, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stream_smem(kStreamMaxKeys)) != cudaSuccess) return DMA_ERR_CUDA;
        return launch_overlapped(stream, dim3((unsigned)rows), dim3(kSelectThreads), stream_smem(P.L), st, 1, delta, ld, P.L, P.w, list, list_stride, tickets);
    }
    const int slice = ((P.L + nrank - 1) / nrank + 31) / 32 * 32;
    auto pick = [&](auto st_tag) {
        constexpr bool kState = decltype(st_tag)::value;
        return slice <= 4 * kSelectThreads ? decode_select_kernel<4, kState> : slice <= 16 * kSelectThreads ? decode_select_kernel<16, kState>
               : slice <= kCtaKeys ? decode_select_kernel<32, kState> : decode_select_kernel<0, kState>;
    };
    auto kern = state ? pick(std::true_type{}) : pick(std::false_type{});
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SelectShared)) != cudaSuccess) return DMA_ERR_CUDA;
    return launch_overlapped(kern, dim3((unsigned)(P.B * P.Hq) * nrank), dim3(kSelectThreads), sizeof(SelectShared), st, nrank, delta, ld, P.L, P.w,
                             slice, list, list_stride, tickets);
}

int launch_decode(const Prob& P, const void* q, const void* K, const void* V, const float* delta, int64_t ld, void* o, float* lse,
                  int32_t* sel_idx, void* ws, cudaStream_t st) {
    const DecodeWs W = decode_ws(P, ws);
    int* kept = sel_idx ? sel_idx : W.kept;              // the caller's index output is the list the attention kernel reads
    int rc = launch_select(P, delta, ld, kept, P.w, W.tickets, false, st);
    if (rc) return rc;
    if (P.dtype == DMA_BF16)
        return P.d == 128 ? launch_typed<__nv_bfloat16, 128>(P, q, K, V, delta, ld, o, lse, kept, P.w, W.tickets, W.partial, st)
                          : launch_typed<__nv_bfloat16, 64>(P, q, K, V, delta, ld, o, lse, kept, P.w, W.tickets, W.partial, st);
    return P.d == 128 ? launch_typed<float, 128>(P, q, K, V, delta, ld, o, lse, kept, P.w, W.tickets, W.partial, st)
                      : launch_typed<float, 64>(P, q, K, V, delta, ld, o, lse, kept, P.w, W.tickets, W.partial, st);
}

// Builds the incremental state from the first N = P.L cached keys: the selection writes lists and headers in place.
int launch_decode_state_init(const Prob& P, const float* delta, int64_t ld, int* state, void* ws, cudaStream_t st) {
    (void)ws;
    const int stride = kStateHeader + ((P.w_cap + 3) & ~3);
    return launch_select(P, delta, ld, state + kStateHeader, stride, nullptr, true, st);
}

template <typename T, int D>
static int launch_step_typed(const Prob& P, const void* q, const void* K, const void* V, const float* delta, int64_t ld, int* state,
                             void* o, float* lse, float* partial, Weakest* weak, cudaStream_t st) {
    const int per = list_split(P), ns = (held_keys(P) + per - 1) / per;
    auto kern = per == kMinSplit ? decode_list_attn_kernel<T, D, kMinSplit> : decode_list_attn_kernel<T, D, kListSplit>;
    const int rc = launch_overlapped(kern, dim3(ns, P.B * P.Hq), dim3(kAttnThreads), 0, st, 1, (const T*)q, (const T*)K, (const T*)V,
                          delta, ld, (const int*)state, P.w_cap, partial, P.L, P.Hq, P.G, P.scale * 1.4426950408889634f, ns, P.ks[0], P.ks[1],
                          P.ks[2], P.vs[0], P.vs[1], P.vs[2], weak);
    if (rc) return rc;
    // Splits of a group in flight together: one where there are no more (480 rows of 5 kept keys, a step, 7.0 -> 6.5 us, with the maxima first 6.6; 32 of 2048 8.2 -> 7.9), else four, and eight of more than 32 of a
    // row (combine kernel: 4 rows of 66141 kept keys, 259 splits, 11.5 -> 8.4 us, two of 16384, 64 splits, 3.55 -> 2.9, but 8 of 4096 2.85 -> 3.07)
    auto combine = ns > 32 ? decode_step_combine_kernel<T, D, 8> : ns > 8 ? decode_step_combine_kernel<T, D, 4> : decode_step_combine_kernel<T, D, 1>;
    return launch_overlapped(combine, dim3(P.B * P.Hq), dim3(8 * D), 0, st, 1, (const float*)partial, (T*)o, lse, ns, delta,
                             ld, P.L, P.w_cap, state, (const Weakest*)weak);
}

// One decoding step with the carried state: P.L counts the cached keys INCLUDING the one appended for this step.
int launch_decode_step(const Prob& P, const void* q, const void* K, const void* V, const float* delta, int64_t ld, int* state,
                       void* o, float* lse, void* ws, cudaStream_t st) {
    const DecodeWs W = decode_ws(P, ws);
    float* partial = W.partial;
    // (the kept lists' part of the workspace, which a step does not use otherwise: 16 bytes per 128 kept keys of the row)
    Weakest* weak = held_keys(P) >= (int)(sizeof(Weakest) / sizeof(int)) ? reinterpret_cast<Weakest*>(W.kept) : nullptr;
    if (P.dtype == DMA_BF16)
        return P.d == 128 ? launch_step_typed<__nv_bfloat16, 128>(P, q, K, V, delta, ld, state, o, lse, partial, weak, st)
                          : launch_step_typed<__nv_bfloat16, 64>(P, q, K, V, delta, ld, state, o, lse, partial, weak, st);
    return P.d == 128 ? launch_step_typed<float, 128>(P, q, K, V, delta, ld, state, o, lse, partial, weak, st)
                      : launch_step_typed<float, 64>(P, q, K, V, delta, ld, state, o, lse, partial, weak, st);
}

}  // namespace dma
