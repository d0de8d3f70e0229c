// sn_grassmann.cu — the subspace update on the Grassmann manifold (Sec. 4.5,
// closed-form gradient of Sec. 6), on the CUDA cores.
//
// With S = (1/K) sum_t G_t^T G_t accumulated as M = sum_t G_t^T (G_t U) = K S U
// (the tensor-core accumulation lives with the contraction kernels), one step is
//   grad    = -2 S U = -(2/K) M                         Euclidean gradient
//   tangent = grad - U (U^T grad)                        Riemannian gradient
//   A       = U - eta * tangent
//   U_new   = Q of A = Q R with diag(R) > 0               retraction
// The retraction is CholeskyQR2: R1 = chol(A^T A), Q1 = A R1^-1, then the
// same once more on Q1 (the Cholesky factor has a positive diagonal, so Q is
// the unique QR factor with diag(R) > 0).  The O(d k^2) products run in fp32
// on the CUDA cores (Gram matrices as per-64-row partial products summed with
// their rounding errors, without atomics; A R^-1 as a row-by-matrix product), the O(k^3)
// Cholesky factor and its triangular inverse in fp32 (this GPU's fp64 rate is a
// small fraction of its fp32 rate).  A is within a small step
// of orthonormal, so its Gram matrix is near the identity and the second pass
// removes what the first leaves; it all runs once every K iterations.
//
// The whole step is one cooperative kernel, a CTA per 64 rows: its products take a
// microsecond or two each, so what counts is the chain of dependent stages.  A CTA
// keeps its rows in shared memory from U and M to U_new and meets the others only
// in the three Gram matrices, each two grid barriers: partial products out, every
// CTA sums a slice of the elements, the sums back in.  Each CTA then factors the
// k x k matrix for itself, which costs less than a third barrier would.  The
// stages are functions, not inlined, so that the second use of each finds its
// instructions cached (inlined, the step took 62 us).  At d = 4096, k = 41 it takes 54
// us, about 20 of them in the two factorisations and 11 in the six barriers; as
// twelve kernels (the factorisation a chain of k two-barrier steps and a serial
// substitution in one block, 47 us each) it took 164 us.
#include <algorithm>

#include "sn_tc.cuh"

namespace sn {
namespace {

constexpr int kRows = 64;       // rows of U per CTA (and per Gram partial)
constexpr int kStepThreads = 512;
constexpr int kStepWarps = kStepThreads / 32;

struct StepParams {
    const float *U, *M;
    float *Y, *G1, *G2;         // k x k sums of the three Gram matrices
    float *A, *Q;               // [d, k]: rows of a CTA that owns several blocks
    float *part;                // [nblk, k, k] partial products
    unsigned int *bar;          // barrier arrivals, and a flag that a wait gave up (both zeroed)
    float *U_new;
    unsigned int *err;
    int d, k, nblk;
    float beta, gamma;          // A = U + beta M + gamma U Y
};

// dst[r][c] = src[row0 + r, c] for the block's rows, zero past d and k (pitch k4 <=
// 128).  A warp takes four rows, all its loads in flight before the first store.
__device__ __forceinline__ void load_rows(float *dst, const float *src, int row0, int d, int k, int k4)
{
    constexpr int N = kRows / kStepWarps;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float v[N][4];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int r = row0 + N * warp + i;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = lane + 32 * q;
            v[i][q] = r < d && c < k ? __ldcg(src + (size_t)r * k + c) : 0.f;
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (lane + 32 * q < k4)
                dst[(N * warp + i) * k4 + lane + 32 * q] = v[i][q];
}
__device__ __forceinline__ void store_rows(float *dst, const float *src, int row0, int d, int k, int k4)
{
    constexpr int N = kRows / kStepWarps;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int r = N * warp + i;
        if (row0 + r < d)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (lane + 32 * q < k)
                    dst[(size_t)(row0 + r) * k + lane + 32 * q] = src[r * k4 + lane + 32 * q];
    }
}

// out[a, b] = sum over the 64 staged rows of sa[r][a] sb[r][b].  A thread owns a
// 4 x 4 tile of (a, b): per row two 16-byte shared loads feed 16 FMAs.  Where the tiles
// are fewer than the threads, groups of threads take every rg-th row and their
// sums meet in `red`.
__device__ __noinline__ void gram(const float *sa, const float *sb, int k, int k4, float *red, float *out)
{
    const int nt = k4 / 4, ntile = nt * nt;
    const int rg = max(1, min(8, kStepThreads / ntile));
    for (int t0 = 0; t0 < ntile; t0 += kStepThreads) {      // one turn unless k > 88
        const int tl = t0 + (rg > 1 ? threadIdx.x % ntile : threadIdx.x);
        const int g = rg > 1 ? threadIdx.x / ntile : 0;
        const bool mine = tl < ntile && g < rg;
        const int ta = 4 * (tl / nt), tb = 4 * (tl % nt);
        float acc[4][4] = {};
        if (mine)
#pragma unroll 4
            for (int r = g; r < kRows; r += rg) {
                const float4 x = *(const float4 *)(sa + r * k4 + ta);
                const float4 y = *(const float4 *)(sb + r * k4 + tb);
                const float xa[4] = {x.x, x.y, x.z, x.w}, yb[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        acc[i][j] = fmaf(xa[i], yb[j], acc[i][j]);
            }
        if (rg > 1) {
            if (mine && g > 0)
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    red[((g - 1) * 16 + i) * ntile + tl] = acc[i / 4][i % 4];
            __syncthreads();
            if (mine && g == 0)
                for (int h = 0; h < rg - 1; ++h)
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        acc[i / 4][i % 4] += red[(h * 16 + i) * ntile + tl];
        }
        if (mine && g == 0)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (ta + i < k && tb + j < k)
                        out[(ta + i) * k + tb + j] = acc[i][j];
    }
    __syncthreads();
}

// s + v as s (rounded) plus the rounding error added to e
__device__ __forceinline__ void two_sum(float &s, float &e, float v)
{
    const float t = __fadd_rn(s, v), w = __fsub_rn(t, s);
    e += __fadd_rn(__fsub_rn(s, __fsub_rn(t, w)), __fsub_rn(v, w));
    s = t;
}

// This CTA's slice of out[e] = sum over the blocks of part[blk, e]: 32 elements a warp,
// the warps that are left over sharing out the blocks.  The sums carry their
// rounding errors along (Knuth's two-sum), so they are as good as fp64 ones rounded
// once; a chain of fp64 additions took 3 us a slice on this GPU.  Where fp32 overflows, the
// pair says nothing and the element is summed again in fp64.
__device__ __noinline__ void sum_slice(const StepParams &p, float *out, float2 *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int kk = p.k * p.k, per = (kk + gridDim.x - 1) / gridDim.x;
    const int e0 = blockIdx.x * per, n = min(per, kk - e0);
    const int nch = (n + 31) / 32;
    const int G = nch > 0 ? max(1, kStepWarps / nch) : 1;
    for (int c0 = 0; c0 < nch; c0 += kStepWarps / G) {
        const int ch = c0 + warp / G, g = warp % G, e = 32 * ch + lane;
        const bool mine = warp / G < kStepWarps / G && e < n;
        float s = 0.f, err = 0.f;
        if (mine)
            for (int b0 = g; b0 < p.nblk; b0 += 8 * G) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)          // eight loads in flight
                    v[u] = b0 + u * G < p.nblk ? __ldcg(p.part + (size_t)(b0 + u * G) * kk + e0 + e)
                                               : 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    two_sum(s, err, v[u]);
            }
        red[warp * 32 + lane] = make_float2(s, err);
        __syncthreads();
        if (mine && g == 0) {
            for (int h = 1; h < G; ++h) {
                const float2 v = red[(warp + h) * 32 + lane];
                two_sum(s, err, v.x);
                err += v.y;
            }
            s += err;
            if (!isfinite(s)) {
                double t = 0.0;
                for (int b = 0; b < p.nblk; ++b)
                    t += (double)__ldcg(p.part + (size_t)b * kk + e0 + e);
                s = (float)t;
            }
            out[e0 + e] = s;
        }
        __syncthreads();
    }
}

// sa[r][:] = alpha sa[r][:] + beta sb[r][:] + gamma (sa[r][:] W) for the 64 staged
// rows, W [k4][k4] zero-padded; a thread owns RM rows x 4 columns.
template <int RM>
__device__ __forceinline__ void row_mix(float *sa, const float *sb, const float *W, int k4, bool whole,
                                        float beta, float gamma)
{
    const int nc = k4 / 4, t = threadIdx.x;
    const int r = RM * (t / nc), c = 4 * (t % nc);
    const bool mine = r < kRows;
    float acc[RM][4] = {};
    if (mine) {
        for (int l = 0; l < k4; l += 4) {
            float a[RM][4];
#pragma unroll
            for (int i = 0; i < RM; ++i) {
                const float4 v = *(const float4 *)(sa + (r + i) * k4 + l);
                a[i][0] = v.x, a[i][1] = v.y, a[i][2] = v.z, a[i][3] = v.w;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = *(const float4 *)(W + (l + q) * k4 + c);
#pragma unroll
                for (int i = 0; i < RM; ++i) {
                    acc[i][0] = fmaf(a[i][q], w.x, acc[i][0]);
                    acc[i][1] = fmaf(a[i][q], w.y, acc[i][1]);
                    acc[i][2] = fmaf(a[i][q], w.z, acc[i][2]);
                    acc[i][3] = fmaf(a[i][q], w.w, acc[i][3]);
                }
            }
        }
        if (whole)
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc[i][j] = sa[(r + i) * k4 + c + j] + beta * sb[(r + i) * k4 + c + j] +
                                gamma * acc[i][j];
    }
    __syncthreads();                                 // every row has been read
    if (mine)
#pragma unroll
        for (int i = 0; i < RM; ++i)
            *(float4 *)(sa + (r + i) * k4 + c) =
                make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    __syncthreads();
}
__device__ __noinline__ void mix(float *sa, const float *sb, const float *W, int k4, bool whole,
                                    float beta, float gamma)
{
    if (k4 <= 64)                                    // 32 x 16 threads at most
        row_mix<2>(sa, sb, W, k4, whole, beta, gamma);
    else
        row_mix<4>(sa, sb, W, k4, whole, beta, gamma);
}

// W[r][c] = G[r, c], zero-padded to [k4][k4]
__device__ __noinline__ void load_square(float *W, const float *G, int k, int k4)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float v[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = warp + kStepWarps * i, c = lane + 32 * q;
            v[i][q] = r < k && c < k ? __ldcg(G + r * k + c) : 0.f;
        }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int r = warp + kStepWarps * i, c = lane + 32 * q;
            if (r < k4 && c < k4)
                W[r * k4 + c] = v[i][q];
        }
    __syncthreads();
}

// W = R^-1 for R the upper Cholesky factor of the symmetric positive-definite G
// (k x k), G = R^T R, in fp32: elimination without square roots, G = L D L^T, with
// L^-1 collected in the columns already eliminated.  Step j takes m = G[j, i] / G[j, j]
// times row j from every later row i, in the columns c > j of G (both triangles, so
// the rule is the same for all) and c < j of L^-1, whose own column j becomes -m.
// R^-1 = (D^-1/2 L^-1)^T.  Warp w holds rows 8 w .. 8 w + 7 in registers, lane l the
// columns l + 32 q.  The chain of k dependent steps is what this costs, so a warp
// eliminates its eight rows by itself, with shuffles, publishes them (`rows`, 2 x 8 x
// 128 floats, and 1 / D in `inv`), and the later warps then take all eight from their
// rows at once: one barrier per eight steps.  Flags a pivot that is not positive
// and goes on with 1.
template <int KQ>
__device__ __noinline__ void cholesky_inverse(const float *G, int k, int k4, float *rows,
                                                 float *inv, float *W, unsigned int *err)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int np = (k + 7) / 8;                      // panels, one per warp
    float v[8][KQ];                                  // rows past k are the identity's
    float dinv = 1.f;                                // lane i < 8: 1 / sqrt(D) of row 8 warp + i
    bool bad = false;
    if (warp < np) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int q = 0; q < KQ; ++q) {
                const int r = 8 * warp + i, c = lane + 32 * q;
                v[i][q] = r < k && c < k ? __ldcg(G + r * k + c) : (r == c ? 1.f : 0.f);
            }
    }
    for (int t = 0; t < np; ++t) {
        float *rt = rows + (t & 1) * 8 * 128;        // two buffers: one barrier per panel
        float *it = inv + (t & 1) * 8;
        if (warp == t) {
            const int l0 = 8 * (t & 3);              // its columns: lanes l0 .. l0 + 7, q = t / 4
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float x = v[j][0];
#pragma unroll
                for (int q = 1; q < KQ; ++q)
                    x = t / 4 == q ? v[j][q] : x;
                float pv = __shfl_sync(0xffffffffu, x, l0 + j);
                bad = bad || !(pv > 0.f);
                pv = pv > 0.f ? pv : 1.f;
                const float r = __frcp_rn(pv);
                if (lane == j)
                    dinv = pv;
                x *= r;
#pragma unroll
                for (int i = j + 1; i < 8; ++i) {
                    const float m = __shfl_sync(0xffffffffu, x, l0 + i);
#pragma unroll
                    for (int q = 0; q < KQ; ++q)
                        v[i][q] = lane + 32 * q == 8 * t + j ? -m : fmaf(-m, v[j][q], v[i][q]);
                }
                if (lane == 0)
                    it[j] = r;
#pragma unroll
                for (int q = 0; q < KQ; ++q)
                    rt[j * 128 + lane + 32 * q] = v[j][q];
            }
            dinv = 1.f / sqrtf(dinv);
        }
        __syncthreads();
        if (warp > t && warp < np) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float r = it[j];
                float s[KQ];
#pragma unroll
                for (int q = 0; q < KQ; ++q)
                    s[q] = rt[j * 128 + lane + 32 * q];
                const float4 a = *(const float4 *)(rt + j * 128 + 8 * warp);
                const float4 b = *(const float4 *)(rt + j * 128 + 8 * warp + 4);
                const float m[8] = {a.x * r, a.y * r, a.z * r, a.w * r, b.x * r, b.y * r, b.z * r, b.w * r};
#pragma unroll
                for (int q = 0; q < KQ; ++q) {
                    const bool own = lane + 32 * q == 8 * t + j;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        v[i][q] = own ? -m[i] : fmaf(-m[i], s[q], v[i][q]);
                }
            }
        }
    }
    if (bad && lane == 0 && blockIdx.x == 0)
        atomicOr(err, SN_EBIT_NUMERIC);
    __syncthreads();
    // W[l][c] = L^-1[c][l] / sqrt(D[c]), zero-padded: row r of L^-1 is column r of W
    for (int e = threadIdx.x; e < k4 * (k4 - k); e += kStepThreads)
        W[(e / (k4 - k)) * k4 + k + e % (k4 - k)] = 0.f;
    if (warp < np)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = 8 * warp + i;
            const float f = __shfl_sync(0xffffffffu, dinv, i);
            if (r < k)
#pragma unroll
                for (int q = 0; q < KQ; ++q) {
                    const int l = lane + 32 * q;
                    if (l < k4)
                        W[l * k4 + r] = l <= r ? (l < r ? v[i][q] : 1.f) * f : 0.f;
                }
        }
    __syncthreads();
}

template <int KQ>                                    // ceil(k / 32)
__global__ void __launch_bounds__(kStepThreads, 1) k_grassmann_step(StepParams p)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(16) float rows[2 * 8 * 128];
    __shared__ float inv[2 * 8];
    const int k = p.k, k4 = (k + 3) & ~3, kk = k * k;
    float *sa = sm, *sb = sa + kRows * k4, *W = sb + kRows * k4;
    float *red = W + k4 * k4;                        // sums of the Gram groups and of the slices
    const bool one = p.nblk <= (int)gridDim.x;       // a block of rows per CTA, kept in sa
    unsigned int nbar = 0;
    auto reduce = [&](float *out) {                  // out = the sum of all partial products
        if (!tc::grid_barrier(p.bar, ++nbar, p.err))
            return false;
        sum_slice(p, out, (float2 *)red);
        return tc::grid_barrier(p.bar, ++nbar, p.err);
    };
    // Y = U^T M
    for (int blk = blockIdx.x; blk < p.nblk; blk += gridDim.x) {
        load_rows(sa, p.U, blk * kRows, p.d, k, k4);
        load_rows(sb, p.M, blk * kRows, p.d, k, k4);
        __syncthreads();
        gram(sa, sb, k, k4, red, p.part + (size_t)blk * kk);
    }
    if (!reduce(p.Y))
        return;
    // A = U + beta M + gamma U Y, and A^T A
    load_square(W, p.Y, k, k4);
    for (int blk = blockIdx.x; blk < p.nblk; blk += gridDim.x) {
        if (!one) {
            load_rows(sa, p.U, blk * kRows, p.d, k, k4);
            load_rows(sb, p.M, blk * kRows, p.d, k, k4);
            __syncthreads();
        }
        mix(sa, sb, W, k4, true, p.beta, p.gamma);
        if (!one)
            store_rows(p.A, sa, blk * kRows, p.d, k, k4);
        gram(sa, sa, k, k4, red, p.part + (size_t)blk * kk);
    }
    if (!reduce(p.G1))
        return;
    // Q1 = A R1^-1, and Q1^T Q1
    cholesky_inverse<KQ>(p.G1, k, k4, rows, inv, W, p.err);
    for (int blk = blockIdx.x; blk < p.nblk; blk += gridDim.x) {
        if (!one) {
            load_rows(sa, p.A, blk * kRows, p.d, k, k4);
            __syncthreads();
        }
        mix(sa, sb, W, k4, false, 0.f, 1.f);
        if (!one)
            store_rows(p.Q, sa, blk * kRows, p.d, k, k4);
        gram(sa, sa, k, k4, red, p.part + (size_t)blk * kk);
    }
    if (!reduce(p.G2))
        return;
    // U_new = Q1 R2^-1
    cholesky_inverse<KQ>(p.G2, k, k4, rows, inv, W, p.err);
    for (int blk = blockIdx.x; blk < p.nblk; blk += gridDim.x) {
        if (!one) {
            load_rows(sa, p.Q, blk * kRows, p.d, k, k4);
            __syncthreads();
        }
        mix(sa, sb, W, k4, false, 0.f, 1.f);
        store_rows(p.U_new, sa, blk * kRows, p.d, k, k4);
    }
}

// acc += sum(G^2) - sum(Cg^2) over bf16 G [T, d] and Cg [T, k].  Bound by the read of
// G: eight 16-byte loads in flight per thread, four CTAs per SM (T = 16384, d = 4096:
// 25 us, 5.3 TB/s; with four loads in flight 35 us).  The squares (128 positive terms at
// a time) are summed in fp32 and then added up in fp64, since this GPU's fp64 rate
// could not keep up with one fp64 operation per element.
constexpr int kResLoads = 8;

__global__ void __launch_bounds__(256, 4) k_residual(const __nv_bfloat16 *__restrict__ G, int64_t ng,
                                                     const __nv_bfloat16 *__restrict__ Cg, int64_t nc,
                                                     double *acc)
{
    griddep_wait();
    double s = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n8 = ng / 8;
    for (int64_t e0 = t0; e0 < n8; e0 += 2 * kResLoads * stride) {
        float f = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t e1 = e0 + h * kResLoads * stride;
            uint4 w[kResLoads];
#pragma unroll
            for (int u = 0; u < kResLoads; ++u)
                w[u] = e1 + u * stride < n8 ? __ldg((const uint4 *)G + e1 + u * stride)
                                            : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < kResLoads; ++u) {
                const uint32_t ws[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float lo = __uint_as_float(ws[q] << 16);
                    const float hi = __uint_as_float(ws[q] & 0xFFFF0000u);
                    f = fmaf(lo, lo, fmaf(hi, hi, f));
                }
            }
        }
        s += (double)f;
    }
    for (int64_t e = (ng / 8) * 8 + t0; e < ng; e += stride) {
        const float v = __bfloat162float(G[e]);
        s += (double)v * v;
    }
    for (int64_t e = t0; e < nc; e += stride) {
        const float v = __bfloat162float(Cg[e]);
        s -= (double)v * v;
    }
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
            t += red[w];
        atomicAdd(acc, t);
    }
}

int sm_count()
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

cudaError_t grassmann_residual(const sn_basis &b, const __nv_bfloat16 *G,
                               const __nv_bfloat16 *Cg, int64_t T, double *acc, cudaStream_t s)
{
    const int64_t want = (T * b.d / 8 + 255) / 256;
    const int grid = (int)std::min<int64_t>(std::max<int64_t>(want, 1), 4 * sm_count());
    const cudaError_t e =
        launch_dependent(k_residual, dim3(grid), dim3(256), 0, s, G, T * b.d, Cg, T * b.k, acc);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// workspace: Y, G1, G2 and the barrier (k x k fp32 each, two spare ones) | A, Q1
// (d x k fp32 each) | Gram partials (one k x k fp32 block per kRows rows)
size_t grassmann_step_workspace(const sn_basis &b)
{
    const size_t kk = align256(sizeof(float) * (size_t)b.k * b.k);
    const size_t dk = align256(sizeof(float) * (size_t)b.d * b.k);
    const size_t parts = align256(sizeof(float) * (size_t)((b.d + kRows - 1) / kRows) * b.k * b.k);
    return 5 * kk + 2 * dk + parts;
}

cudaError_t grassmann_step(const sn_basis &b, const float *M, int K, float eta, float *U_new,
                           void *workspace, cudaStream_t s)
{
    const int d = b.d, k = b.k, k4 = (k + 3) & ~3;
    const size_t kk = align256(sizeof(float) * (size_t)k * k);
    const size_t dk = align256(sizeof(float) * (size_t)d * k);
    char *w = (char *)workspace;
    // A = U - eta * (c M - U (c Y)) with c = -2 / K
    const double c = -2.0 / K;
    StepParams p;
    p.U = b.u32;
    p.M = M;
    p.Y = (float *)w;
    p.G1 = (float *)(w + kk);
    p.G2 = (float *)(w + 2 * kk);
    p.bar = (unsigned int *)(w + 3 * kk);
    p.A = (float *)(w + 5 * kk);
    p.Q = (float *)(w + 5 * kk + dk);
    p.part = (float *)(w + 5 * kk + 2 * dk);
    p.U_new = U_new;
    p.err = b.err;
    p.d = d;
    p.k = k;
    p.nblk = (d + kRows - 1) / kRows;
    p.beta = (float)(-eta * c);
    p.gamma = (float)(eta * c);
    // rows of U (A, Q1) and M, a k x k matrix, the Gram groups' sums
    const size_t smem = sizeof(float) * (2 * (size_t)kRows * k4 + (size_t)k4 * k4 + 16 * kStepThreads);
    void (*const kernels[4])(StepParams) = {k_grassmann_step<1>, k_grassmann_step<2>,
                                            k_grassmann_step<3>, k_grassmann_step<4>};
    void (*const kernel)(StepParams) = kernels[(k - 1) / 32];
    cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(p.bar, 0, 2 * sizeof(unsigned int), s);
    if (e != cudaSuccess)
        return e;
    // cooperative: the CTAs wait for one another, so all are resident, one on each SM
    // that the stream's context has
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(p.nblk, stream_sms(s)));
    cfg.blockDim = dim3(kStepThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, p);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace sn
