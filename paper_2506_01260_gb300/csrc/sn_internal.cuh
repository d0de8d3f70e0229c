// sn_internal.cuh — types shared by the library's translation units.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sn.h"

// Bits of the per-basis device error word.
enum : unsigned int {
    SN_EBIT_BAD_ID = 1u,    // an id or position was out of range (row zeroed)
    SN_EBIT_TIMEOUT = 2u,   // a bounded wait expired; the kernel gave up
    SN_EBIT_NUMERIC = 4u,   // a factorisation met a non-positive pivot
};

// Padded copies of U kept by a basis handle.
//   u32  [d, k]      fp32, as given (CUDA-core paths, row i = U[i, :])
//   u32t [k, d]      fp32 transpose (CUDA-core reconstruction, coalesced in d)
//   u32p [d32/2, kp, 2]  fp32, rows of U in pairs, zero past k and d (d32 = d rounded
//                    up to 32; CUDA-core compress and projection)
//   ut16 [n_pad, d]  bf16 U^T, rows >= k zero: B operand of the d -> k contraction
//   up16 [d, k64]    bf16 U, columns >= k zero: operand of the k -> d expansion
struct sn_basis {
    int device;
    int d, k;
    int n_pad;   // k rounded up to 16 (MMA N of the compress contraction)
    int k64;     // k rounded up to 64 (whole 128-byte swizzle atoms)
    int kp;      // k rounded up to the CUDA-core compress's columns (u32p)
    void *mem;   // the one device allocation that every buffer below lies in
    float *u32;
    float *u32t;
    float *u32p;
    __nv_bfloat16 *ut16;
    __nv_bfloat16 *up16;
    unsigned int *err;
    // fp32 partial rows of the compress contractions' split last-round tiles:
    // [0] forward (X and projected-table modes), [1] backward; tail_cap row
    // tiles of 128 x n_pad each (one per SM of the device)
    float *tail[2];
    int tail_cap;
};

namespace sn {

// Counts every kernel the library launches (reported by sn_launch_count).
void count_launch(int n = 1);

// ---- dependent launches ----------------------------------------------------------
// A kernel launched with programmatic stream serialization may be set up before the
// previous kernel of its stream has ended: griddep_wait blocks until that one has
// completed and its writes are visible (a no-op after a normal launch or any
// other kind of predecessor).  The library's kernels call it before their first
// access to global memory, so a launch overlaps the end of whatever ran before it, and
// none completes before its predecessor has.
//
// griddep_launch_dependents lets the next such kernel start as soon as every CTA of
// this one has called it, instead of when they end.  Only grids of at most kFewCtas
// call it: their successor finds idle SMs.  Called by every kernel, the
// successor's first CTAs crowd onto the SMs that happen to be free, and the four
// boundary calls took 76 us instead of 67 (1B class, 128 CTAs a grid), 192 instead of
// 182 (8B class), in fp32 153 instead of 137.
constexpr unsigned kFewCtas = 64;

__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void griddep_start()
{
    if (gridDim.x <= kFewCtas)
        griddep_launch_dependents();
    griddep_wait();
}

// ---- clusters ----------------------------------------------------------------------
__device__ __forceinline__ void cluster_arrive()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}
// the fp32 at shared address `a` of the cluster's CTA `rank`
__device__ __forceinline__ float ld_cluster(uint32_t a, uint32_t rank)
{
    uint32_t r;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r) : "memory");
    return v;
}

// Launch `kernel` in clusters of `cluster` CTAs along x, as a dependent of the
// previous kernel of the stream.
template <typename... KArgs, typename... Args>
cudaError_t launch_clusters(void (*kernel)(KArgs...), int cluster, dim3 grid, dim3 block, size_t smem,
                            cudaStream_t s, const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t s, const Args &...args)
{
    return launch_clusters(kernel, 1, grid, block, smem, s, args...);
}

// ---- CUDA-core kernels (fp32 path) -------------------------------------------
cudaError_t simt_compress(const sn_basis &b, const float *X, const int32_t *ids, const int32_t *pos,
                          int64_t T, int seq_len, const float *tok, int64_t vocab, const float *pe,
                          float *C, bool gather, cudaStream_t s);
cudaError_t simt_decompress(const sn_basis &b, const float *C, const int32_t *ids,
                            const int32_t *pos, int64_t T, int seq_len, const float *tok,
                            int64_t vocab, const float *pe, float *X, bool gather, cudaStream_t s);
cudaError_t simt_project(const sn_basis &b, const float *W, int64_t cols, int64_t ld, float *W_out,
                         float *A, cudaStream_t s);
int simt_padded_columns(int k);   // sn_basis::kp

// SMs available to kernels on a stream (fewer than the device's in a green context)
int stream_sms(cudaStream_t s);

cudaError_t prepare_basis(sn_basis &b, const float *U, cudaStream_t s);

// ---- tensor-core kernels (bf16 path, tcgen05 + TMA) -----------------------------
struct TcArgs {
    const __nv_bfloat16 *X;     // compress: X or G [T, d]; decompress: output X or G
    const int32_t *ids;
    const int32_t *pos;
    const __nv_bfloat16 *tok;
    const __nv_bfloat16 *pe;
    __nv_bfloat16 *C;           // compress: output [T, k]; decompress: input
    int64_t T;
    int64_t vocab;
    int seq_len;
    bool gather;                // subtract / add the embeddings
};
cudaError_t tc_compress(const sn_basis &b, const TcArgs &a, cudaStream_t s);
cudaError_t tc_decompress(const sn_basis &b, const TcArgs &a, __nv_bfloat16 *X_out,
                          cudaStream_t s);
cudaError_t tc_project(const sn_basis &b, const __nv_bfloat16 *W, int64_t cols, int64_t ld,
                       __nv_bfloat16 *W_out, void *workspace, cudaStream_t s);
size_t tc_project_workspace(const sn_basis &b, int64_t cols);
// out[r, :] = A[r, :] U in fp32 (projected tables: T_fixed U, P U)
cudaError_t tc_contract_f32(const sn_basis &b, const __nv_bfloat16 *A, int64_t rows, float *out,
                            cudaStream_t s);
// Grassmann accumulation M += G^T Cg (M fp32 [d, k]); workspace bytes for T tokens
size_t tc_grassmann_workspace(const sn_basis &b, int64_t T);
cudaError_t tc_grassmann_accumulate(const sn_basis &b, const __nv_bfloat16 *G,
                                    const __nv_bfloat16 *Cg, int64_t T, float *M, void *workspace,
                                    cudaStream_t s);
// ||G||^2 - ||Cg||^2 added to *acc (fp64); the Grassmann step (CUDA cores)
cudaError_t grassmann_residual(const sn_basis &b, const __nv_bfloat16 *G,
                               const __nv_bfloat16 *Cg, int64_t T, double *acc, cudaStream_t s);
size_t grassmann_step_workspace(const sn_basis &b);
cudaError_t grassmann_step(const sn_basis &b, const float *M, int K, float eta, float *U_new,
                           void *workspace, cudaStream_t s);
// Row-constant AdamW step (fp32 W, M, V; grad bf16 or fp32); colsum: [cols] fp32 scratch
cudaError_t adamw_rowconst(bool grad_bf16, float *W, const void *g, float *M, float *V,
                           int64_t rows, int64_t cols, int64_t t, float lr, float b1, float b2,
                           float eps, float lam, float *colsum, cudaStream_t s);
// Lossy comparators (bf16 batches [T, d])
cudaError_t lossy_topk(const void *X, int64_t T, int d, int kk, void *vals, uint16_t *cols,
                       cudaStream_t s);
cudaError_t lossy_topk_restore(const void *vals, const uint16_t *cols, int64_t T, int d, int kk,
                               void *out, cudaStream_t s);
cudaError_t lossy_sign(const void *X, int64_t T, int d, uint32_t *bits, float *scale,
                       cudaStream_t s);
cudaError_t lossy_sign_restore(const uint32_t *bits, const float *scale, int64_t T, int d,
                               void *out, cudaStream_t s);
cudaError_t lossy_quant(const void *X, int64_t T, int d, int format, uint8_t *codes, float *scale,
                        cudaStream_t s);
cudaError_t lossy_quant_restore(const uint8_t *codes, const float *scale, int64_t T, int d,
                                int format, void *out, cudaStream_t s);
// C = X U - TU[ids] - PU[pos] (PU may be null)
cudaError_t tc_compress_projected(const sn_basis &b, const __nv_bfloat16 *X, const int32_t *ids,
                                  const int32_t *pos, int64_t T, int seq_len, const float *TU,
                                  int64_t vocab, const float *PU, __nv_bfloat16 *C,
                                  cudaStream_t s);

}  // namespace sn
