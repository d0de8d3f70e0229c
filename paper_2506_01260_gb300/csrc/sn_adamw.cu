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
// adjacent columns (16-byte accesses; four rows in flight in the first pass, eight in
// the second) when the column count is a multiple of 4, else one column.
#include <algorithm>

#include "sn_internal.cuh"

namespace sn {
namespace {

constexpr int kThreads = 256;
constexpr int kRows = 16;    // rows per thread
constexpr int kRows2 = 8;    // rows per thread, second pass with four columns a thread

// A block is `lanes` threads along the columns times kThreads / lanes row groups.  First
// pass: at most 64 lanes.  A block's column sums meet in shared memory, so a column takes
// one atomic for at least 4 * kRows = 64 rows: the rounding of the atomic chain is what the
// sums' error consists of.  One atomic for 16 rows (256 lanes) took as long, but its error
// against 64 bits was 1.6 to 1.8 times as large ([8192, 1024], W = 0: 1.88e-7 of W
// instead of 1.15e-7).  Second pass: at most 256 lanes, the whole block along one row.
// Weights with fewer columns take the power of two of lanes that covers them, and a
// group then every (kThreads / lanes)-th row of its block's run, so that a block's
// accesses stay contiguous: [2^20, 4] takes 22 us and [65536, 64] 18 (894 and 114 with 256
// lanes throughout, of which 1 and 16 had a column; 287 and 62 with 64 rows a block as well).
constexpr int kLanes1 = 64, kLanes2 = 256;

__host__ __device__ constexpr int rows_per_block(int lanes, int rows) { return kThreads / lanes * rows; }

// log2 of the lanes for `units` columns (or groups of four)
int lanes_log2(int64_t units, int most)
{
    int l = 0;
    while ((1 << l) < most && ((int64_t)1 << l) < units)
        ++l;
    return l;
}

// This thread's column unit, its first row, the step to its next row and the end of its
// run.  LANES > 0, the widest form: consecutive rows, every step a constant (left to run
// time, the addresses cost the wide kernels their loads in flight: 278 us for 237 at
// [4096, 14336]).
struct Place {
    int64_t unit, r, r1;
    int step;
};
template <int ROWS, int LANES>
__device__ __forceinline__ Place place(int lx, int64_t rows)
{
    Place p;
    if (LANES > 0) {
        p.unit = (int64_t)blockIdx.x * LANES + threadIdx.x % LANES;
        p.step = 1;
        p.r = ((int64_t)blockIdx.y * (kThreads / LANES) + threadIdx.x / LANES) * ROWS;
        p.r1 = p.r + ROWS < rows ? p.r + ROWS : rows;
    } else {
        p.unit = ((int64_t)blockIdx.x << lx) + (threadIdx.x & ((1 << lx) - 1));
        p.step = kThreads >> lx;
        const int64_t r0 = (int64_t)blockIdx.y * p.step * ROWS;
        p.r = r0 + (threadIdx.x >> lx);
        p.r1 = r0 + p.step * ROWS < rows ? r0 + p.step * ROWS : rows;
    }
    return p;
}

__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float4 add(float4 a, float4 b)
{
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// The sum of `s` over the block's row groups, for the threads of the first one
template <typename T>
__device__ __forceinline__ T sum_groups(T s, int lx)
{
    __shared__ T red[kThreads];
    red[threadIdx.x] = s;
    for (int o = kThreads / 2; o >= 1 << lx; o /= 2) {
        __syncthreads();
        if ((int)threadIdx.x < o)
            red[threadIdx.x] = s = add(s, red[threadIdx.x + o]);
    }
    return s;
}

__global__ void __launch_bounds__(kThreads) k_zero(float *__restrict__ p, int64_t n)
{
    griddep_wait();
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
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
                                                             float vcorr, float *__restrict__ colsum,
                                                             int lx)
{
    griddep_wait();
    const Place at = place<kRows, 0>(lx, rows);
    const int64_t c = at.unit;
    float s = 0.f;
    for (int64_t r = at.r; r < at.r1 && c < cols; r += at.step) {
        const int64_t e = r * cols + c;
        const float gv = load_grad(g, e);
        const float m = b1 * M[e] + (1.f - b1) * gv;
        const float v = b2 * V[e] + (1.f - b2) * gv * gv;
        M[e] = m;
        V[e] = v;
        s += v * vcorr;
    }
    s = sum_groups(s, lx);
    if (threadIdx.x < 1 << lx && c < cols)
        atomicAdd(colsum + c, s);
}

__global__ void __launch_bounds__(kThreads) k_adamw_apply(float *__restrict__ W,
                                                           const float *__restrict__ M, int64_t rows,
                                                           int64_t cols, float lr, float mcorr,
                                                           float eps, float lam, float inv_rows,
                                                           const float *__restrict__ colsum, int lx)
{
    griddep_wait();
    const Place at = place<kRows, 0>(lx, rows);
    const int64_t c = at.unit;
    if (c >= cols)
        return;
    const float alpha = 1.f / (sqrtf(colsum[c] * inv_rows) + eps);
    const float step = lr * mcorr * alpha;
    for (int64_t r = at.r; r < at.r1; r += at.step) {
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
// bf16 gradient: threads of 64 / 32 / 16 + 8 rows take 259 / 251 / 240 us (6.9 TB/s on 28
// bytes an element), 8 + 8 rows 241, 4 + 4 rows 267; [1024, 1024]: 30 us with 64 rows (64
// blocks), 13 with 16 + 8.  Evict-first hints on V, M and W or a reversed second pass, to
// find g in L2, made it slower (262-271 us), and so did a single kernel of clusters that
// own 128 columns (339), or a loop over several runs of rows in a block (263).
constexpr int kUnroll1 = 4, kUnroll2 = 8;

template <typename GT, bool WIDE>
__global__ void __launch_bounds__(kThreads) k_adamw_v4(const GT *__restrict__ g, float *__restrict__ V,
                                                        int64_t rows, int64_t cols, float b2, float vcorr,
                                                        float *__restrict__ colsum, int lx)
{
    griddep_wait();
    const Place at = place<kRows, WIDE ? kLanes1 : 0>(lx, rows);
    const int64_t c = 4 * at.unit;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t r1 = c < cols ? at.r1 : 0;
    for (int64_t r = at.r; r < r1; r += kUnroll1 * at.step) {
        float4 gv[kUnroll1], vv[kUnroll1];
#pragma unroll
        for (int u = 0; u < kUnroll1; ++u)
            if (r + u * at.step < r1) {
                gv[u] = load_grad4(g, (r + u * at.step) * cols + c);
                vv[u] = *(const float4 *)(V + (r + u * at.step) * cols + c);
            }
#pragma unroll
        for (int u = 0; u < kUnroll1; ++u)
            if (r + u * at.step < r1) {
                float4 v;
                v.x = b2 * vv[u].x + (1.f - b2) * gv[u].x * gv[u].x;
                v.y = b2 * vv[u].y + (1.f - b2) * gv[u].y * gv[u].y;
                v.z = b2 * vv[u].z + (1.f - b2) * gv[u].z * gv[u].z;
                v.w = b2 * vv[u].w + (1.f - b2) * gv[u].w * gv[u].w;
                *(float4 *)(V + (r + u * at.step) * cols + c) = v;
                s.x += v.x * vcorr;
                s.y += v.y * vcorr;
                s.z += v.z * vcorr;
                s.w += v.w * vcorr;
            }
    }
    s = sum_groups(s, lx);
    if (threadIdx.x >= 1 << lx || c >= cols)
        return;
    atomicAdd(colsum + c, s.x);
    atomicAdd(colsum + c + 1, s.y);
    atomicAdd(colsum + c + 2, s.z);
    atomicAdd(colsum + c + 3, s.w);
}

template <typename GT, bool WIDE>
__global__ void __launch_bounds__(kThreads, 2) k_adamw_mw4(const GT *__restrict__ g, float *__restrict__ W,
                                                      float *__restrict__ M, int64_t rows,
                                                      int64_t cols, float b1, float lr, float mcorr,
                                                      float eps, float lam, float inv_rows,
                                                      const float *__restrict__ colsum, int lx)
{
    griddep_wait();
    const Place at = place<kRows2, WIDE ? kLanes2 : 0>(lx, rows);
    const int64_t c = 4 * at.unit;
    if (c >= cols)
        return;
    const float4 cs = *(const float4 *)(colsum + c);
    const float4 st = make_float4(lr * mcorr / (sqrtf(cs.x * inv_rows) + eps),
                                  lr * mcorr / (sqrtf(cs.y * inv_rows) + eps),
                                  lr * mcorr / (sqrtf(cs.z * inv_rows) + eps),
                                  lr * mcorr / (sqrtf(cs.w * inv_rows) + eps));
    for (int64_t r = at.r; r < at.r1; r += kUnroll2 * at.step) {
        float4 gv[kUnroll2], mv[kUnroll2], wv[kUnroll2];
#pragma unroll
        for (int u = 0; u < kUnroll2; ++u)
            if (r + u * at.step < at.r1) {
                const int64_t e = (r + u * at.step) * cols + c;
                gv[u] = load_grad4(g, e);
                mv[u] = *(const float4 *)(M + e);
                wv[u] = *(const float4 *)(W + e);
            }
#pragma unroll
        for (int u = 0; u < kUnroll2; ++u)
            if (r + u * at.step < at.r1) {
                const int64_t e = (r + u * at.step) * cols + c;
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
    const bool four = cols % 4 == 0;
    const int64_t units = four ? cols / 4 : cols;
    const int lx = lanes_log2(units, kLanes1), per = rows_per_block(1 << lx, kRows);
    const dim3 grid((unsigned)(((units - 1) >> lx) + 1), (unsigned)((rows + per - 1) / per));
    count_launch();
    if (!four)
        return launch_dependent(k_adamw_moments<GT>, grid, dim3(kThreads), 0, s, g, M, V, rows, cols, b1, b2,
                                vcorr, colsum, lx);
    return launch_dependent(1 << lx == kLanes1 ? k_adamw_v4<GT, true> : k_adamw_v4<GT, false>, grid,
                            dim3(kThreads), 0, s, g, V, rows, cols, b2, vcorr, colsum, lx);
}

// The second pass: W (and M)
template <typename GT>
cudaError_t apply(const GT *g, float *W, float *M, int64_t rows, int64_t cols, float b1, float lr, float mcorr,
                  float eps, float lam, float inv_rows, const float *colsum, cudaStream_t s)
{
    const bool four = cols % 4 == 0;
    const int64_t units = four ? cols / 4 : cols;
    const int lx = lanes_log2(units, kLanes2), per = rows_per_block(1 << lx, four ? kRows2 : kRows);
    const dim3 grid((unsigned)(((units - 1) >> lx) + 1), (unsigned)((rows + per - 1) / per));
    count_launch();
    if (!four)
        return launch_dependent(k_adamw_apply, grid, dim3(kThreads), 0, s, W, M, rows, cols, lr, mcorr, eps,
                                lam, inv_rows, colsum, lx);
    return launch_dependent(1 << lx == kLanes2 ? k_adamw_mw4<GT, true> : k_adamw_mw4<GT, false>, grid,
                            dim3(kThreads), 0, s, g, W, M, rows, cols, b1, lr, mcorr, eps, lam, inv_rows,
                            colsum, lx);
}

}  // namespace

cudaError_t adamw_rowconst(bool grad_bf16, float *W, const void *g, float *M, float *V,
                           int64_t rows, int64_t cols, int64_t t, float lr, float b1, float b2,
                           float eps, float lam, float *colsum, cudaStream_t s)
{
    // three dependent launches: a memset between two kernels would end the overlap
    cudaError_t e = launch_dependent(k_zero, dim3((unsigned)std::min<int64_t>((cols + kThreads - 1) / kThreads, 152)),
                                     dim3(kThreads), 0, s, colsum, cols);
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
