// Shared declarations of the DMA CUDA library: resolved problem view, launch accounting, small device helpers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dma.h"

namespace dma {

constexpr int kWsHeaderBytes = 256;   // every workspace starts with this header; int32 word 0 = status

// dma_problem_t with defaults resolved and derived sizes filled in.
struct Prob {
    int B, Hq, Hkv, L, d, G;
    int w;                 // min(w, L)
    int w_cap;             // w as given (the capacity of an incremental decoding state)
    int dtype, flags;      // flags: the caller's and what they imply (DMA_FLAG_COMPACT_KV also where the library chose it)
    bool chose_compact;    // token-compacted execution is the library's choice: a shorter sequence may walk tiles
    int causal;            // 1: key j visible to rows i >= j; 0: to every row (the key's first row is 0 instead of j)
    int bm, bn, Tr, Tc, Wd;   // bitmap tile sizes, tile counts, uint32 words per bitmap row
    int bwd_split;            // CTAs that share a KV head in the tile-mode backward (0: tc_bwd_splits chooses)
    int bwd_heads;            // (batch, query head) pairs by which the token-compacted backward cuts its walks (0: B Hq)
    int Lq, q_off;            // forward over a chunk of query rows: Q, O, lse hold the rows q_off .. q_off + Lq - 1 (Lq = L, q_off = 0: all)
    float scale;
    int64_t qs[3], ks[3], vs[3], os[3];   // batch, seq, head strides in elements
};

int resolve(const dma_problem_t* p, Prob* out);          // validation + defaults; returns dma_status
void count_launch(int n = 1);
// measurement hook (dma_kernel_timing): brackets a stage's main kernel with a pair of CUDA events while recording is on
void timing_mark(int which, bool after, cudaStream_t st);
int check_launch();                                       // cudaGetLastError -> dma_status

// stage launchers (each returns a dma_status); defined in the stage's .cu file
size_t mask_ws_bytes(const Prob& P);
size_t mask_bwd_need(const Prob& P);       // as tc_bwd_need, tc_bwd_ws_bytes
size_t mask_bwd_ws_bytes(const Prob& P);
int launch_delta_range(const Prob& P, const void* V, const float* W, const float* A, float* delta, int64_t ld, int j_begin,
                       int j_end, cudaStream_t st);
size_t decode_ws_bytes(const Prob& P);
size_t decode_state_bytes(const Prob& P);
int launch_decode_state_init(const Prob& P, const float* delta, int64_t ld, int* state, void* ws, cudaStream_t st);
int launch_decode_step(const Prob& P, const void* q, const void* K, const void* V, const float* delta, int64_t ld, int* state,
                       void* o, float* lse, void* ws, cudaStream_t st);
int launch_decode(const Prob& P, const void* q, const void* K, const void* V, const float* delta, int64_t ld, void* o, float* lse,
                  int32_t* sel_idx, void* ws, cudaStream_t st);
int launch_mask_bwd(const Prob& P, const void* V, const float* W, const float* A, const float* delta, const float* dM,
                    void* dV, float* dW, float* dA, void* ws, cudaStream_t st);
int launch_mask_build(const Prob& P, const void* V, const float* W, const float* A, float* bias, int32_t* expiry,
                      uint32_t* bitmap, void* ws, cudaStream_t st, const int32_t* cu_seqlens = nullptr, int nseq = 0);

size_t simt_bwd_ws_bytes(const Prob& P);
int launch_simt_fwd(const Prob& P, const void* Q, const void* K, const void* V, const float* bias,
                    const int32_t* expiry, const uint32_t* bitmap, void* O, float* lse, void* ws, cudaStream_t st);
int launch_simt_bwd(const Prob& P, const void* Q, const void* K, const void* V, const void* O, const void* dO,
                    const float* lse, const float* bias, const int32_t* expiry, const uint32_t* bitmap, void* dQ,
                    void* dK, void* dV, float* dM, void* ws, cudaStream_t st);

size_t tc_fwd_ws_bytes(const Prob& P);
int launch_tc_fwd(const Prob& P, const void* Q, const void* K, const void* V, const float* bias,
                  const int32_t* expiry, const uint32_t* bitmap, void* O, float* lse, void* ws, cudaStream_t st);
size_t tc_bwd_need(const Prob& P);         // what the call uses
size_t tc_bwd_ws_bytes(const Prob& P);     // what is asked for: at least the need of every shorter sequence and smaller batch
int tc_bwd_splits(const Prob& P);
// dma_attn_bwd on a part of a problem: with the split and the walks of the whole one, so that the parts' results are the whole's
int attn_bwd_part(const dma_problem_t* p, int split, int heads, const void* Q, const void* K, const void* V, const void* O, const void* dO,
                  const float* lse, const float* bias, const int32_t* expiry, const uint32_t* bitmap, void* dQ, void* dK, void* dV,
                  float* dM, void* ws, size_t ws_bytes, cudaStream_t st);
int launch_tc_bwd(const Prob& P, const void* Q, const void* K, const void* V, const void* O, const void* dO,
                  const float* lse, const float* bias, const int32_t* expiry, const uint32_t* bitmap, void* dQ,
                  void* dK, void* dV, float* dM, void* ws, cudaStream_t st);

// ---------------------------------------------------------------------------------------------
// launches that overlap the tail of the kernel before them (programmatic dependent launch)
// ---------------------------------------------------------------------------------------------
// A kernel launched this way may become resident once every CTA of the previous kernel of the stream has left the chip or is
// about to, instead of after that kernel's completion has been reported. Every such kernel calls pdl_enter() (or
// pdl_enter_restrict()) with ALL its global pointers before its first access to global memory: it returns once the previous
// kernel has completed and its writes are visible. What is saved is the launch latency between dependent kernels, about 1 to 2 us
// each, which short kernels are made of: step of 2 x 1000 rows, d = 64: 112 -> 103 us, prefill of 4096 keys 123 -> 107 us.
// (Letting the next kernel in early, with griddepcontrol.launch_dependents at the top, was slower everywhere: its waiting CTAs
// take the places that the running kernel's CTAs leave unevenly, 218 -> 239 us for 2048 rows of a 16384-key prefill, 2998 ->
// 3071 us for its training step.)
// Returns a dma_status; a caller that gets an error launches nothing more, since the later kernels read what this one writes.
template <typename... KArgs, typename... Args>
inline int launch_config(bool overlapped, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = overlapped ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    if (cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...) != cudaSuccess) {
        cudaGetLastError();              // (consumed here: it is not the next call's error)
        return DMA_ERR_CUDA;
    }
    count_launch();
    return DMA_OK;
}
template <typename... KArgs, typename... Args>
inline int launch_overlapped(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, Args... args) {
    return launch_config(true, kernel, grid, block, smem, st, cluster, args...);
}
// the launch of a kernel that does not wait itself
template <typename... KArgs, typename... Args>
inline int launch_plain(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    return launch_config(false, kernel, grid, block, smem, st, 1, args...);
}

// ---------------------------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------------------------
// Waits for the previous kernel. The pointers pass through an empty asm statement behind the
// wait, so that no load through them (a read-only load of a const __restrict__ parameter is free to move) comes before it.
template <typename... Ts>
__device__ __forceinline__ void pdl_enter(Ts&... ptrs) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    auto pin = [](auto& p) { asm volatile("" : "+l"(p) :: "memory"); };
    (pin(ptrs), ...);
}

// The same wait for kernels that its pins slow down. A pointer that has passed through asm is no longer __restrict__: the loads
// through it wait for every store before them, those to shared memory included. Here the pointers move by a zero that only the
// asm statement knows, so that the addresses depend on the wait and the pointers stay __restrict__. For the kernels of
// mask_build.cu; us with pdl_enter / this (without overlap or pins before): full sampling weights of 32 heads, 1024 channels, mask
// build of 16384 keys 204 / 163 (165), of 8192 keys 131 / 91 (91), delta of 8 x 65536 keys, 32 heads 574 / 566 (558), mask build
// of 32 heads, 16384 keys 76 / 73 (76). The kernels of the other files gain and lose by it (fp32 forward of two heads, 256 rows
// 12.3 / 14.2, mask backward of 4096 keys 13.8 / 14.2) and keep the pins.
template <typename... Ts>
__device__ __forceinline__ void pdl_enter_restrict(Ts&... ptrs) {
    int64_t zero;
    asm volatile("griddepcontrol.wait;\n\tmov.s64 %0, 0;" : "=l"(zero) :: "memory");
    ((ptrs += zero), ...);
}

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void store_as(float* p, float x) { *p = x; }
__device__ __forceinline__ void store_as(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }

// bit (kt % 32) of word [bh, qt, kt / 32]
__device__ __forceinline__ bool bitmap_test(const uint32_t* bitmap, int Tr, int Wd, int bh, int qt, int kt) {
    return (bitmap[((size_t)bh * Tr + qt) * Wd + (kt >> 5)] >> (kt & 31)) & 1u;
}

}  // namespace dma
