// sn_adamw.cu — the row-constant AdamW step that keeps W_p2 inside the
// subspace (Sec. 5), memory-bound, on the CUDA cores.
//
// W is the torch weight [rows = d, cols = n]; its columns are the paper's rows
// of W_p2 (the d-vectors that live in S).  One step t >= 1:
//   M = b1 M + (1 - b1) g,  V = b2 V + (1 - b2) g^2          (in place, fp32)
//   mu[c] = mean over the column of V / (1 - b2^t)             (the paper's row mean)
//   W = W - lr (M / (1 - b1^t)) / (sqrt(mu[c]) + eps) - lambda W
// Pass 1 updates V and adds each block's column sums of V^ to a zeroed [cols]
// fp32 workspace with one atomic per column and block; pass 2 updates M (it
// reads g again, 2 bytes, instead of reading back an updated M, 4 bytes) and
// W: 28 bytes moved per element with a bf16 gradient.  Each thread owns four
// adjacent columns (16-byte accesses, rows unrolled by four) of a block of rows
// when the column count is a multiple of 4, else one column; every access is
// coalesced along the columns.
#include <algorithm>

#include "sn_internal.cuh"

namespace sn {
namespace {

constexpr int kThreads = 256;
constexpr int kCols = 256;   // columns per block of the second pass (one per thread)
constexpr int kRows = 16;    // rows per thread

// The first pass's blocks: kLanes threads along the columns, kGroups groups of them along
// the rows, each thread kRows rows.  A block's column sums meet in shared memory, so
// a column takes one atomic for kGroups * kRows = 64 rows: the rounding of the atomic
// chain is what the sums' error consists of.  One atomic for 16 rows (blocks of 256 x 16)
// took as long, but its error against 64 bits was 1.6 to 1.8 times as large ([8192, 1024], W = 0:
// 1.88e-7 of W instead of 1.15e-7).
constexpr int kLanes = 64, kGroups = kThreads / kLanes;

__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float4 add(float4 a, float4 b)
{
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// The sum of `s` over the block's row groups, for the threads of the first one
template <typename T>
__device__ __forceinline__ T sum_groups(T s)
{
    __shared__ T red[kThreads];
    red[threadIdx.x] = s;
#pragma unroll
    for (int o = kThreads / 2; o >= kLanes; o /= 2) {
        __syncthreads();
        if ((int)threadIdx.x < o)
            red[threadIdx.x] = s = add(s, red[threadIdx.x + o]);
    }
    return s;
}

__global__ void __launch_bounds__(kCols) k_zero(float *__restrict__ p, int64_t n)
{
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * kCols + threadIdx.x; i < n; i += (int64_t)gridDim.x * kCols)
        p[i] = 0.f;
}

template <typename GT>
__device__ __forceinline__ float load_grad(const GT *g, int64_t e);
template <>
__device__ __forceinline__ float load_grad<float>(const float *g, int64_t e)
{
    return __ldg(g + e);
}
template <>
__device__ __forceinline__ float load_grad<__nv_bfloat16>(const __nv_bfloat16 *g, int64_t e)
{
    return __bfloat162float(g[e]);
}

template <typename GT>
__global__ void __launch_bounds__(kThreads) k_adamw_moments(const GT *__restrict__ g,
                                                             float *__restrict__ M,
                                                             float *__restrict__ V, int64_t rows,
                                                             int64_t cols, float b1, float b2,
                                                             float vcorr, float *__restrict__ colsum)
{
    griddep_wait();
    const int64_t c = (int64_t)blockIdx.x * kLanes + threadIdx.x % kLanes;
    const int64_t r0 = ((int64_t)blockIdx.y * kGroups + threadIdx.x / kLanes) * kRows;
    const int64_t r1 = c < cols ? (r0 + kRows < rows ? r0 + kRows : rows) : 0;
    float s = 0.f;
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t e = r * cols + c;
        const float gv = load_grad(g, e);
        const float m = b1 * M[e] + (1.f - b1) * gv;
        const float v = b2 * V[e] + (1.f - b2) * gv * gv;
        M[e] = m;
        V[e] = v;
        s += v * vcorr;
    }
    s = sum_groups(s);
    if (threadIdx.x < kLanes && c < cols)
        atomicAdd(colsum + c, s);
}

__global__ void __launch_bounds__(kCols) k_adamw_apply(float *__restrict__ W,
                                                        const float *__restrict__ M, int64_t rows,
                                                        int64_t cols, float lr, float mcorr,
                                                        float eps, float lam, float inv_rows,
                                                        const float *__restrict__ colsum)
{
    griddep_wait();
    const int64_t c = (int64_t)blockIdx.x * kCols + threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.y * kRows;
    if (c >= cols)
        return;
    const float alpha = 1.f / (sqrtf(colsum[c] * inv_rows) + eps);
    const float step = lr * mcorr * alpha;
    const int64_t r1 = r0 + kRows < rows ? r0 + kRows : rows;
    for (int64_t r = r0; r < r1; ++r) {
        const int64_t e = r * cols + c;
        const float w = W[e];
        W[e] = w - step * M[e] - lam * w;
    }
}

// ---- four columns per thread ------------------------------------------------

template <typename GT>
__device__ __forceinline__ float4 load_grad4(const GT *g, int64_t e);
template <>
__device__ __forceinline__ float4 load_grad4<float>(const float *g, int64_t e)
{
    return __ldg((const float4 *)(g + e));
}
template <>
__device__ __forceinline__ float4 load_grad4<__nv_bfloat16>(const __nv_bfloat16 *g, int64_t e)
{
    const uint2 u = __ldg((const uint2 *)(g + e));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
}

// Rows per thread and rows in flight of the two passes.  Blocks run column-major over a
// few rows, so the GPU as a whole sweeps the arrays in order of address.  [4096, 14336],
// bf16 gradient: threads of
// 64 / 32 / 16 + 8 rows take 259 / 251 / 240 us (6.9 TB/s on 28 bytes an element), 8 + 8
// rows 241, 4 + 4 rows 267; [1024, 1024]: 30 us with 64 rows (64 blocks), 13 with 16 + 8.
// Evict-first hints on V, M and W or a reversed second pass, to find g in L2, made it
// slower (262-271 us), and so did a single kernel of clusters that own 128 columns
// (339), or a loop over several runs of rows in a block (263).
constexpr int kRows2 = 8;   // second pass (the first: kRows)
constexpr int kUnroll1 = 4, kUnroll2 = 8;

template <typename GT>
__global__ void __launch_bounds__(kThreads) k_adamw_v4(const GT *__restrict__ g, float *__restrict__ V,
                                                        int64_t rows, int64_t cols, float b2, float vcorr,
                                                        float *__restrict__ colsum)
{
    griddep_wait();
    const int64_t c = 4 * ((int64_t)blockIdx.x * kLanes + threadIdx.x % kLanes);
    const int64_t r0 = ((int64_t)blockIdx.y * kGroups + threadIdx.x / kLanes) * kRows;
    const int64_t r1 = c < cols ? (r0 + kRows < rows ? r0 + kRows : rows) : 0;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t rb = r0; rb < r1; rb += kUnroll1) {
        float4 gv[kUnroll1], vv[kUnroll1];
#pragma unroll
        for (int u = 0; u < kUnroll1; ++u)
            if (rb + u < r1) {
                gv[u] = load_grad4(g, (rb + u) * cols + c);
                vv[u] = *(const float4 *)(V + (rb + u) * cols + c);
            }
#pragma unroll
        for (int u = 0; u < kUnroll1; ++u)
            if (rb + u < r1) {
                float4 v;
                v.x = b2 * vv[u].x + (1.f - b2) * gv[u].x * gv[u].x;
                v.y = b2 * vv[u].y + (1.f - b2) * gv[u].y * gv[u].y;
                v.z = b2 * vv[u].z + (1.f - b2) * gv[u].z * gv[u].z;
                v.w = b2 * vv[u].w + (1.f - b2) * gv[u].w * gv[u].w;
                *(float4 *)(V + (rb + u) * cols + c) = v;
                s.x += v.x * vcorr;
                s.y += v.y * vcorr;
                s.z += v.z * vcorr;
                s.w += v.w * vcorr;
            }
    }
    s = sum_groups(s);
    if (threadIdx.x >= kLanes || c >= cols)
        return;
    atomicAdd(colsum + c, s.x);
    atomicAdd(colsum + c + 1, s.y);
    atomicAdd(colsum + c + 2, s.z);
    atomicAdd(colsum + c + 3, s.w);
}

template <typename GT>
__global__ void __launch_bounds__(kCols) k_adamw_mw4(const GT *__restrict__ g, float *__restrict__ W,
                                                      float *__restrict__ M, int64_t rows,
                                                      int64_t cols, float b1, float lr, float mcorr,
                                                      float eps, float lam, float inv_rows,
                                                      const float *__restrict__ colsum)
{
    griddep_wait();
    const int64_t c = 4 * ((int64_t)blockIdx.x * kCols + threadIdx.x);
    const int64_t r0 = (int64_t)blockIdx.y * kRows2;
    if (c >= cols)
        return;
    const float4 cs = *(const float4 *)(colsum + c);
    const float4 st = make_float4(lr * mcorr / (sqrtf(cs.x * inv_rows) + eps),
                                  lr * mcorr / (sqrtf(cs.y * inv_rows) + eps),
                                  lr * mcorr / (sqrtf(cs.z * inv_rows) + eps),
                                  lr * mcorr / (sqrtf(cs.w * inv_rows) + eps));
    const int64_t r1 = r0 + kRows2 < rows ? r0 + kRows2 : rows;
    for (int64_t rb = r0; rb < r1; rb += kUnroll2) {
        float4 gv[kUnroll2], mv[kUnroll2], wv[kUnroll2];
#pragma unroll
        for (int u = 0; u < kUnroll2; ++u)
            if (rb + u < r1) {
                const int64_t e = (rb + u) * cols + c;
                gv[u] = load_grad4(g, e);
                mv[u] = *(const float4 *)(M + e);
                wv[u] = *(const float4 *)(W + e);
            }
#pragma unroll
        for (int u = 0; u < kUnroll2; ++u)
            if (rb + u < r1) {
                const int64_t e = (rb + u) * cols + c;
                float4 m, w;
                m.x = b1 * mv[u].x + (1.f - b1) * gv[u].x;
                m.y = b1 * mv[u].y + (1.f - b1) * gv[u].y;
                m.z = b1 * mv[u].z + (1.f - b1) * gv[u].z;
                m.w = b1 * mv[u].w + (1.f - b1) * gv[u].w;
                w.x = wv[u].x - st.x * m.x - lam * wv[u].x;
                w.y = wv[u].y - st.y * m.y - lam * wv[u].y;
                w.z = wv[u].z - st.z * m.z - lam * wv[u].z;
                w.w = wv[u].w - st.w * m.w - lam * wv[u].w;
                *(float4 *)(M + e) = m;
                *(float4 *)(W + e) = w;
            }
    }
}

// The first pass over `rows` rows: V (and M, where the columns are taken singly)
template <typename GT>
cudaError_t moments(const GT *g, float *M, float *V, int64_t rows, int64_t cols, float b1, float b2,
                    float vcorr, float *colsum, cudaStream_t s)
{
    const unsigned y = (unsigned)((rows + kGroups * kRows - 1) / (kGroups * kRows));
    count_launch();
    if (cols % 4 != 0)
        return launch_dependent(k_adamw_moments<GT>,
                                dim3((unsigned)((cols + kLanes - 1) / kLanes), y), dim3(kThreads), 0, s, g, M,
                                V, rows, cols, b1, b2, vcorr, colsum);
    return launch_dependent(k_adamw_v4<GT>, dim3((unsigned)((cols / 4 + kLanes - 1) / kLanes), y),
                            dim3(kThreads), 0, s, g, V, rows, cols, b2, vcorr, colsum);
}

// The second pass: W (and M)
template <typename GT>
cudaError_t apply(const GT *g, float *W, float *M, int64_t rows, int64_t cols, float b1, float lr, float mcorr,
                  float eps, float lam, float inv_rows, const float *colsum, cudaStream_t s)
{
    count_launch();
    if (cols % 4 != 0)
        return launch_dependent(k_adamw_apply,
                                dim3((unsigned)((cols + kCols - 1) / kCols), (unsigned)((rows + kRows - 1) / kRows)),
                                dim3(kCols), 0, s, W, M, rows, cols, lr, mcorr, eps, lam, inv_rows, colsum);
    return launch_dependent(k_adamw_mw4<GT>,
                            dim3((unsigned)((cols / 4 + kCols - 1) / kCols), (unsigned)((rows + kRows2 - 1) / kRows2)),
                            dim3(kCols), 0, s, g, W, M, rows, cols, b1, lr, mcorr, eps, lam, inv_rows, colsum);
}

}  // namespace

cudaError_t adamw_rowconst(bool grad_bf16, float *W, const void *g, float *M, float *V,
                           int64_t rows, int64_t cols, int64_t t, float lr, float b1, float b2,
                           float eps, float lam, float *colsum, cudaStream_t s)
{
    // three dependent launches: a memset between two kernels would end the overlap
    cudaError_t e = launch_dependent(k_zero, dim3((unsigned)std::min<int64_t>((cols + kCols - 1) / kCols, 152)),
                                     dim3(kCols), 0, s, colsum, cols);
    count_launch();
    // bias corrections of step t, in double before rounding to fp32
    const float vcorr = (float)(1.0 / (1.0 - pow((double)b2, (double)t)));
    const float mcorr = (float)(1.0 / (1.0 - pow((double)b1, (double)t)));
    const float inv_rows = (float)(1.0 / (double)rows);
    // a grid's y extent holds 65535 blocks: more rows go in several launches per pass
    const int64_t most = (int64_t)65535 * (cols % 4 == 0 ? kRows2 : kRows);
    for (int64_t r = 0; r < rows && e == cudaSuccess; r += most) {
        const int64_t n = std::min(rows - r, most), o = r * cols;
        e = grad_bf16 ? moments((const __nv_bfloat16 *)g + o, M + o, V + o, n, cols, b1, b2, vcorr, colsum, s)
                      : moments((const float *)g + o, M + o, V + o, n, cols, b1, b2, vcorr, colsum, s);
    }
    for (int64_t r = 0; r < rows && e == cudaSuccess; r += most) {
        const int64_t n = std::min(rows - r, most), o = r * cols;
        e = grad_bf16 ? apply((const __nv_bfloat16 *)g + o, W + o, M + o, n, cols, b1, lr, mcorr, eps, lam,
                              inv_rows, colsum, s)
                      : apply((const float *)g + o, W + o, M + o, n, cols, b1, lr, mcorr, eps, lam, inv_rows,
                              colsum, s);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace sn
