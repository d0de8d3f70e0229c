// sn_simt.cu — CUDA-core kernels: the fp32 path of every boundary operation
// and the one-off preparation of a basis handle's padded copies of U.
//
// fp32 inputs must match the fp64 definition to ~1e-5 relative, which rules
// out TF32/bf16 tensor-core inputs; these kernels use fp32 FMA with fp32
// accumulation.  At k = 20 they do 5-10 flops per byte read, so both the FMA
// pipe (74 TFLOP/s) and HBM bound them: every kernel keeps a register tile per
// thread (an operand read from shared memory feeds 4-32 FMAs), issues packed
// two-wide FMAs (fma.rn.f32x2: half the issue slots, each half an ordinary
// fp32 FMA) and splits the long reduction over d between warps and over a
// thread-block cluster, whose partial sums meet in shared memory.
#include <algorithm>

#include "sn_internal.cuh"

namespace sn {
namespace {

// Row state of a token inside a block: skip (t >= T), compute, or zero (bad id).
enum : int { ROW_SKIP = 0, ROW_OK = 1, ROW_BAD = 2 };

// Validate token t's id and position; returns the row state and the element
// offsets of its token-table and positional-table rows.
__device__ __forceinline__ int token_rows(int64_t t, int64_t T, bool gather,
                                          const int32_t *ids, const int32_t *pos,
                                          int seq_len, int64_t vocab, bool has_pe, int d,
                                          int64_t *tok_off, int64_t *pe_off,
                                          unsigned int *err)
{
    *tok_off = 0;
    *pe_off = 0;
    if (t >= T)
        return ROW_SKIP;
    if (!gather)
        return ROW_OK;
    int64_t id = ids[t];
    int64_t p = 0;
    bool bad = id < 0 || id >= vocab;
    if (has_pe) {
        p = pos ? (int64_t)pos[t] : t % seq_len;
        bad = bad || p < 0 || p >= seq_len;
    }
    if (bad) {
        atomicOr(err, SN_EBIT_BAD_ID);
        return ROW_BAD;
    }
    *tok_off = id * d;
    *pe_off = p * d;
    return ROW_OK;
}

// ---- packed fp32 pairs, shared memory, clusters ---------------------------------
typedef unsigned long long f32x2;   // two fp32, the lower-indexed one in the low half

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_4(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
// `bytes` (0 to 16) of the 16, the rest zeros
__device__ __forceinline__ void cp_async_part(uint32_t dst, const void *src, unsigned bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.wait_all;" ::: "memory");
}
// CTAs per cluster that share one output tile's reduction: 1 where the stream's context
// has not all of the SMs (a cluster might find no place in it), else the power of two up
// to 8 with the least (rounds of the grid) x (steps per CTA + 3 for its start + one
// for each CTA whose partial sums meet), every CTA keeping at least one step.  Among
// equal costs, the fewest CTAs.  Measured on whole calls, with 1 / 2 / 4 / 8 CTAs:
// compress of 8192 x 2048 (256 tiles) 31 / 34 / 35 / 43 us; projection at k = 20, when its
// first pass still loaded W a single step ahead, of [2048, 2048] (16 tiles) 74 / 48 / 33 / 37 us, of
// [2048, 8192] (64 tiles) 92 / 67 / 72 / 90 us.
int cluster_split(int64_t tiles, int steps, int sms, int per_sm, cudaStream_t s)
{
    const int64_t slots = (int64_t)sms * per_sm;
    int best = 1;
    int64_t best_cost = -1;
    for (int c = 1; c <= 8 && c <= steps; c *= 2) {
        const int64_t rounds = (tiles * c + slots - 1) / slots;
        const int64_t cost = rounds * ((steps + c - 1) / c + 3 + c);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best > 1 && stream_sms(s) < sms ? 1 : best;
}

// ---- C[t, :] = (X[t, :] - tok[id] - pe[p]) U  (or G U when !GATHER) -----------
// A CTA of four warps owns 32 tokens.  WN warps (1, 2 or 4: k <= 32, 64, 128)
// form a group that covers all k columns of a run of 32-column chunks of d; the
// groups of a CTA and the CTAs of a cluster take the chunks in turn and add up
// their partial sums at the end, so even a few tokens occupy many warps.  Per
// chunk a group loads the 32 x 32 pieces of X, tok and pe (128-byte row
// segments) into registers a chunk ahead, stores their fp32 difference to
// shared memory and multiplies it by 32 rows of U (paired copy u32p, by
// cp.async).  A thread owns 4 tokens x TN columns, each sum kept as two halves
// (even and odd columns of d) so that both operands of a packed FMA are pairs
// as they lie in shared memory.  At T = 8192, d = 2048, k = 20 (134 and 67 MB read):
// 42 us with embeddings (3.3 TB/s) and 30 us without, where one output per thread
// and one pair of shared loads per FMA took 271 and 239 us.  What bounds it is the
// latency of the 7 warps that the registers leave on an SM, on shared loads for the
// most part: 0.36 instructions a cycle and scheduler, the shared-memory pipe 37 and 49% busy,
// the FMA pipe 30 and 36%.  Tiles of 8 tokens a thread need 255 registers and were
// slower (48 and 30 us), so were chunks of 16 columns at twice the warps (45 us).
constexpr int CTM = 4;          // tokens per thread
constexpr int CTOK = 8 * CTM;   // tokens per CTA
constexpr int CCH = 32;         // columns of d per chunk
constexpr int CPITCH = CCH + 4; // floats per staged row: a column's rows fall in distinct banks
constexpr int CTHREADS = 128;

struct SimtCompress {
    const float *up;            // paired copy of U
    const float *X, *tok, *pe;
    const int32_t *ids, *pos;
    float *C;
    unsigned int *err;
    int64_t T, vocab;
    int d, k, seq_len, split;   // split: CTAs per cluster
};

template <int WN, int TN, bool GATHER>
__global__ void __launch_bounds__(CTHREADS) k_simt_compress(const SimtCompress p)
{
    constexpr int G = CTHREADS / 32 / WN;        // groups per CTA
    constexpr int GS = 32 * WN;                   // threads per group
    constexpr int KP = 4 * TN * WN;               // padded columns of U
    constexpr int NL = CTOK * CCH / 4 / GS;       // 16-byte pieces per thread and operand
    constexpr int LR = CTOK / NL;                 // rows that one load of the group covers
    extern __shared__ __align__(16) float sm[];
    __shared__ int64_t rtok[CTOK], rpe[CTOK];
    __shared__ int rstate[CTOK];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int group = warp / WN, wcol = warp % WN, gl = tid % GS;
    const int rank = (int)(blockIdx.x % p.split);
    const int64_t t0 = (int64_t)(blockIdx.x / p.split) * CTOK;
    const bool has_pe = GATHER && p.pe != nullptr;
    griddep_wait();
    if (tid < CTOK)
        rstate[tid] = token_rows(t0 + tid, p.T, GATHER, p.ids, p.pos, p.seq_len, p.vocab, has_pe,
                                 p.d, &rtok[tid], &rpe[tid], p.err);
    __syncthreads();

    float *rb = sm + group * (2 * CTOK * CPITCH);
    float *ub = sm + G * (2 * CTOK * CPITCH) + group * (2 * CCH * KP);
    const int lrow = gl / (CCH / 4), lcol = 4 * (gl % (CCH / 4));
    unsigned rows_ok = 0;                          // this thread's rows that are read
#pragma unroll
    for (int u = 0; u < NL; ++u)
        rows_ok |= (rstate[lrow + LR * u] == ROW_OK ? 1u : 0u) << u;

    float4 xv[NL], tv[GATHER ? NL : 1], pv[GATHER ? NL : 1];
    auto load = [&](int c) {
        const int col = c * CCH + lcol;
        const bool in = col < p.d;                  // d is a multiple of 8
        const float *x = p.X + (t0 + lrow) * p.d + col;
#pragma unroll
        for (int u = 0; u < NL; ++u) {
            const int row = lrow + LR * u;
            const bool ok = in && ((rows_ok >> u) & 1u);
            xv[u] = ok ? __ldcs((const float4 *)(x + (int64_t)(LR * u) * p.d))
                       : make_float4(0.f, 0.f, 0.f, 0.f);
            if (GATHER) {
                tv[u] = ok ? __ldg((const float4 *)(p.tok + rtok[row] + col))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
                if (has_pe)
                    pv[u] = ok ? __ldg((const float4 *)(p.pe + rpe[row] + col))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    };
    auto load_u = [&](int c, int b) {
        const float *src = p.up + (int64_t)c * CCH * KP;
        const uint32_t dst = smem_addr(ub + b * CCH * KP);
        for (int f = gl; f < CCH * KP / 4; f += GS)
            cp_async_16(dst + 16 * f, src + 4 * f);
    };

    f32x2 acc[CTM][TN];
#pragma unroll
    for (int m = 0; m < CTM; ++m)
#pragma unroll
        for (int n = 0; n < TN; ++n)
            acc[m][n] = 0ull;
    // Token lane, column lane.  A pass of the shared memory serves equal addresses where
    // neighbouring lanes share them: wide tiles, whose reads of U outweigh those of the
    // rows, put the lanes of one column side by side (k = 128: 112 us instead of 174).
    constexpr bool kWide = TN >= 6;
    const int tg = kWide ? lane & 7 : lane >> 2, cg = kWide ? lane >> 3 : lane & 3;
    const int nch = (p.d + CCH - 1) / CCH, step = p.split * G;
    int c = rank * G + group;
    if (c < nch) {
        load(c);
        load_u(c, 0);
    }
    for (int it = 0; c < nch; ++it, c += step) {
        const int b = it & 1;
#pragma unroll
        for (int u = 0; u < NL; ++u) {
            float4 r = xv[u];
            if (GATHER) {
                r.x -= tv[u].x;
                r.y -= tv[u].y;
                r.z -= tv[u].z;
                r.w -= tv[u].w;
                if (has_pe) {
                    r.x -= pv[u].x;
                    r.y -= pv[u].y;
                    r.z -= pv[u].z;
                    r.w -= pv[u].w;
                }
            }
            *(float4 *)(rb + b * CTOK * CPITCH + (lrow + LR * u) * CPITCH + lcol) = r;
        }
        cp_async_wait_all();
        if (WN == 1)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(GS) : "memory");
        if (c + step < nch) {
            load(c + step);
            load_u(c + step, b ^ 1);
        }
        const float *rt = rb + b * CTOK * CPITCH + tg * CPITCH;
        const f32x2 *ut = (const f32x2 *)(ub + b * CCH * KP) + (4 * wcol + cg) * TN;
#pragma unroll
        for (int q = 0; q < CCH / 4; ++q) {
            ulonglong2 r[CTM];
#pragma unroll
            for (int m = 0; m < CTM; ++m)
                r[m] = *(const ulonglong2 *)(rt + 8 * m * CPITCH + 4 * q);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                f32x2 u[TN];
                const f32x2 *us = ut + (2 * q + h) * KP;
                if (TN % 2 == 0) {
#pragma unroll
                    for (int n = 0; n < TN / 2; ++n) {
                        const ulonglong2 w = ((const ulonglong2 *)us)[n];
                        u[2 * n] = w.x;
                        u[2 * n + 1] = w.y;
                    }
                } else {
#pragma unroll
                    for (int n = 0; n < TN; ++n)
                        u[n] = us[n];
                }
#pragma unroll
                for (int m = 0; m < CTM; ++m)
#pragma unroll
                    for (int n = 0; n < TN; ++n)
                        acc[m][n] = fma2(h ? r[m].y : r[m].x, u[n], acc[m][n]);
            }
        }
    }

    // partial sums of the CTA's groups, then of the cluster's CTAs
    constexpr int RP = KP + 1;
    __syncthreads();                                // every group is done with its stages
#pragma unroll
    for (int m = 0; m < CTM; ++m)
#pragma unroll
        for (int n = 0; n < TN; ++n) {
            const float2 v = unpack2(acc[m][n]);
            sm[(group * CTOK + tg + 8 * m) * RP + (4 * wcol + cg) * TN + n] = v.x + v.y;
        }
    __syncthreads();
    const int nout = CTOK * p.k;
    const int per = (nout + p.split - 1) / p.split;
    if (p.split > 1) {
        for (int e = tid; e < nout; e += CTHREADS) {
            const int o = e / p.k * RP + e % p.k;
            float v = sm[o];
#pragma unroll
            for (int g = 1; g < G; ++g)
                v += sm[g * CTOK * RP + o];
            sm[o] = v;
        }
        cluster_sync();
    }
    for (int e = rank * per + tid; e < min(nout, (rank + 1) * per); e += CTHREADS) {
        const int tl = e / p.k, o = tl * RP + e % p.k;
        float v = 0.f;
        if (p.split > 1) {
            for (int r = 0; r < p.split; ++r)
                v += ld_cluster(smem_addr(sm + o), r);
        } else {
#pragma unroll
            for (int g = 0; g < G; ++g)
                v += sm[g * CTOK * RP + o];
        }
        if (rstate[tl] != ROW_SKIP)
            p.C[t0 * p.k + e] = rstate[tl] == ROW_OK ? v : 0.f;
    }
    if (p.split > 1)
        cluster_sync();                             // no CTA leaves while its sums are read
}

// ---- out[r, c] = sum_j L[r, j] R[j, c] (+ pe[p, c] + tok[id, c]) -----------------
// The reconstruction (L = C, R = U^T) and the projection's second pass
// (L = U, R = U^T W).  A CTA keeps 128 columns of R in shared memory and walks down
// the rows; its warps share nothing else, each taking 16 rows at a time (copied to
// its own piece of shared memory), a thread 8 rows x 8 columns (two 16-byte runs
// 64 columns apart).  j goes up in order in one fp32 FMA chain per output; a
// packed FMA takes two adjacent columns and an element of L twice.  At T = 8192,
// d = 2048, k = 20: 28 us without and 45 us with embeddings (one column and 8 tokens a
// thread: 40 and 72 us); the projection's second pass to [2048, 8192] 28 us (98).  The
// FMA pipe is half busy; the rest is the stores and, with embeddings, the T_fixed rows
// (whose form spills 40 bytes a thread to stay at two CTAs an SM).
constexpr int ETILE = 128;      // columns per CTA, rows per step of its eight warps
constexpr int EROWS = 16;       // rows per warp and step
constexpr int ETHREADS = 256;

struct SimtExpand {
    const float *L, *R;
    const float *tok, *pe;
    const int32_t *ids, *pos;
    float *out;
    unsigned int *err;
    int64_t rows, cols, ldr, ldo, vocab;
    int k, seq_len;
};

template <bool EMB>
__global__ void __launch_bounds__(ETHREADS, 2) k_simt_expand(const SimtExpand p)
{
    extern __shared__ __align__(16) float smx[];
    const int kq = (p.k + 1) & ~1;                  // j in pairs: odd k gets a zero column
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *rs = smx;                                // [kq][ETILE]
    float *ls = smx + kq * ETILE + warp * 2 * EROWS * kq;   // [2][EROWS][kq]
    __shared__ int64_t rtok[EMB ? 2 * ETILE : 1], rpe[EMB ? 2 * ETILE : 1];
    __shared__ int rstate[2 * ETILE];
    const int64_t c0 = (int64_t)blockIdx.x * ETILE;
    const bool has_pe = EMB && p.pe != nullptr;
    griddep_wait();
    if (p.ldr % 4 == 0) {
        for (int e = tid; e < p.k * (ETILE / 4); e += ETHREADS) {
            const int j = e / (ETILE / 4), q = 4 * (e % (ETILE / 4));
            if (c0 + q < p.cols)                    // cols = ldr here: whole 16 bytes
                *(float4 *)(rs + j * ETILE + q) =
                    __ldg((const float4 *)(p.R + (int64_t)j * p.ldr + c0 + q));
        }
    } else {
        for (int e = tid; e < p.k * ETILE; e += ETHREADS) {
            const int j = e / ETILE, q = e % ETILE;
            if (c0 + q < p.cols)
                rs[e] = __ldg(p.R + (int64_t)j * p.ldr + c0 + q);
        }
    }
    if (kq > p.k) {
        if (tid < ETILE)
            rs[p.k * ETILE + tid] = 0.f;
        ls[lane * kq + p.k] = 0.f;
    }
    __syncthreads();

    const int rg = lane >> 4, cl = lane & 15;
    const int64_t ntiles = (p.rows + ETILE - 1) / ETILE;
    // the next rows of L (4-byte copies: k may be odd) and their table rows, a step ahead
    auto fetch = [&](int64_t tile, int b) {
        const int64_t r0 = tile * ETILE + EROWS * warp;
        const int nrow = (int)max((int64_t)0, min((int64_t)EROWS, p.rows - r0));
        const float *src = p.L + r0 * p.k;
        float *dst = ls + b * EROWS * kq;
        if (kq == p.k) {
            for (int e = lane; e < nrow * kq; e += 32)
                cp_async_4(smem_addr(dst + e), src + e);
        } else {
            for (int r = 0; r < nrow; ++r)
                for (int j = lane; j < p.k; j += 32)
                    cp_async_4(smem_addr(dst + r * kq + j), src + r * p.k + j);
        }
        if (lane < EROWS) {
            const int w = (b * 8 + warp) * EROWS + lane;
            if (EMB)
                rstate[w] = token_rows(r0 + lane, p.rows, true, p.ids, p.pos, p.seq_len, p.vocab,
                                       has_pe, (int)p.cols, &rtok[w], &rpe[w], p.err);
            else
                rstate[w] = lane < nrow ? ROW_OK : ROW_SKIP;
        }
    };
    fetch(blockIdx.y, 0);
    int b = 0;
    for (int64_t tile = blockIdx.y; tile < ntiles; tile += gridDim.y, b ^= 1) {
        const int64_t r0 = tile * ETILE + EROWS * warp;
        const int w0 = (b * 8 + warp) * EROWS;
        cp_async_wait_all();
        __syncwarp();                               // this step's rows are staged
        if (tile + gridDim.y < ntiles)
            fetch(tile + gridDim.y, b ^ 1);
        const float *lt = ls + (b * EROWS + 8 * rg) * kq;
        // With embeddings the 128 columns are taken 64 at a time, so that the T_fixed rows
        // can be loaded before the products and still fit the registers.
#pragma unroll
        for (int h0 = 0; h0 < (EMB ? 2 : 1); ++h0) {
            constexpr int NH = EMB ? 1 : 2;         // 64-column runs per turn
            const float *rt = rs + 64 * h0 + 4 * cl;
            float4 tv[EMB ? 8 : 1];
            if (EMB) {                              // p.cols = d is a multiple of 8 here
                const int64_t c = c0 + 64 * h0 + 4 * cl;
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int r = w0 + 8 * rg + m;
                    tv[m] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (c + 4 <= p.cols && rstate[r] == ROW_OK)
                        tv[m] = __ldg((const float4 *)(p.tok + rtok[r] + c));
                }
            }
            f32x2 acc[8][2 * NH];
#pragma unroll
            for (int m = 0; m < 8; ++m)
#pragma unroll
                for (int n = 0; n < 2 * NH; ++n)
                    acc[m][n] = 0ull;
#pragma unroll 2
            for (int j = 0; j < kq; j += 2) {
                float2 l[8];
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    l[m] = *(const float2 *)(lt + m * kq + j);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    ulonglong2 r[NH];
#pragma unroll
                    for (int h = 0; h < NH; ++h)
                        r[h] = *(const ulonglong2 *)(rt + (j + i) * ETILE + 64 * h);
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const float v = i ? l[m].y : l[m].x;
                        const f32x2 vv = pack2(v, v);
#pragma unroll
                        for (int h = 0; h < NH; ++h) {
                            acc[m][2 * h] = fma2(vv, r[h].x, acc[m][2 * h]);
                            acc[m][2 * h + 1] = fma2(vv, r[h].y, acc[m][2 * h + 1]);
                        }
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                const int64_t c = c0 + 64 * (h0 + h) + 4 * cl;
                const bool whole = c + 4 <= p.cols;
                float4 ev[EMB ? 8 : 1];
                if (EMB && has_pe) {
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const int r = w0 + 8 * rg + m;
                        if (whole && rstate[r] == ROW_OK)
                            ev[m] = __ldg((const float4 *)(p.pe + rpe[r] + c));
                    }
                }
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int st = rstate[w0 + 8 * rg + m];
                    if (st == ROW_SKIP)
                        continue;
                    const float2 x = unpack2(acc[m][2 * h]), y = unpack2(acc[m][2 * h + 1]);
                    float4 v = make_float4(x.x, x.y, y.x, y.y);
                    if (EMB) {
                        if (has_pe) {
                            v.x += ev[m].x;
                            v.y += ev[m].y;
                            v.z += ev[m].z;
                            v.w += ev[m].w;
                        }
                        v.x += tv[m].x;
                        v.y += tv[m].y;
                        v.z += tv[m].z;
                        v.w += tv[m].w;
                        if (st == ROW_BAD)
                            v = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    float *o = p.out + (r0 + 8 * rg + m) * p.ldo + c;
                    if (whole) {
                        __stcs((float4 *)o, v);
                    } else {
                        if (c < p.cols) o[0] = v.x;
                        if (c + 1 < p.cols) o[1] = v.y;
                        if (c + 2 < p.cols) o[2] = v.z;
                    }
                }
            }
        }
    }
}

// The same for few rows: a thread owns one column and 8 rows and reads its column of R from
// L2, so that a CTA starts without a copy of R and a small output is spread over eight times
// as many threads.  Bound by that chain of loads, eight in flight.  The sums' chains are the
// same, and so are the bits.  65 rows, d = 1000, k = 128: 9.4 us without and 11.4 us with
// embeddings, by the tile kernel 15.9 and 24.7; 1024 rows (512 CTAs) 15.2 and 17.2 against
// 17.1 and 26.0; 2048 rows (1024 CTAs) 29.9 and 33.4 against 17.2 and 26.2.
constexpr int FROWS = 8;        // rows per CTA
constexpr int FTHREADS = 256;   // columns per CTA
constexpr int FK = 128;         // largest k
static_assert(FTHREADS / 32 == FROWS, "a warp copies a row");

template <bool EMB>
__global__ void __launch_bounds__(FTHREADS) k_simt_expand_few(const SimtExpand p)
{
    __shared__ __align__(16) float ls[FROWS][FK];
    __shared__ int64_t rtok[FROWS], rpe[FROWS];
    __shared__ int rstate[FROWS];
    const int tid = threadIdx.x;
    const int64_t c = (int64_t)blockIdx.x * FTHREADS + tid, r0 = (int64_t)blockIdx.y * FROWS;
    const bool has_pe = EMB && p.pe != nullptr;
    griddep_wait();
    if (tid < FROWS)
        rstate[tid] = token_rows(r0 + tid, p.rows, EMB, p.ids, p.pos, p.seq_len, p.vocab, has_pe,
                                 (int)p.cols, &rtok[tid], &rpe[tid], p.err);
    for (int j = tid & 31; j < p.k; j += 32) {       // a row per warp
        const int m = tid >> 5;
        ls[m][j] = r0 + m < p.rows ? p.L[(r0 + m) * p.k + j] : 0.f;
    }
    __syncthreads();
    if (c >= p.cols)
        return;
    float acc[FROWS] = {};
#pragma unroll 8
    for (int j = 0; j < p.k; ++j) {
        const float u = __ldg(p.R + (int64_t)j * p.ldr + c);
#pragma unroll
        for (int m = 0; m < FROWS; ++m)
            acc[m] = fmaf(ls[m][j], u, acc[m]);
    }
#pragma unroll
    for (int m = 0; m < FROWS; ++m) {
        if (rstate[m] == ROW_SKIP)
            continue;
        float v = acc[m];
        if (EMB && rstate[m] == ROW_OK) {
            if (has_pe)
                v += __ldg(p.pe + rpe[m] + c);
            v += __ldg(p.tok + rtok[m] + c);
        }
        p.out[(r0 + m) * p.ldo + c] = rstate[m] == ROW_OK ? v : 0.f;
    }
}

// ---- A = U^T W (fp32 [k, cols]), the projection's first pass ---------------------
// A warp owns 128 columns of W (a thread four, as two pairs) and JT columns of U;
// WN warps form a group that covers all k, and the groups of a CTA and the CTAs of
// a cluster take blocks of eight rows of W in turn.  W and U (paired copy u32p) come
// through a ring of four steps by cp.async: a thread copies and reads its own
// 16-byte pieces of W, U is shared and read by broadcast, two rows x two columns a
// load for 8 packed FMAs.  [2048, 2048] and [2048, 8192] at k = 20: 18 and 29 us (HBM
// 2.5 and 10, FMA pipe 2.3 and 9 on all SMs), 20 and 35 with W a single step ahead in
// registers, and 1297 and 1339 with a thread per column that walked all of d with one
// load of U per FMA.  The FMA pipe is 38 and 42% busy: two warps a scheduler issue 0.36
// and 0.39 a cycle.  Three CTAs of four warps on an SM were slower (18 and 33 us).
constexpr int PROWS = 8;        // rows of W per group and step
constexpr int PTHREADS = 256;
constexpr int PSTEPS = 4;       // steps in the ring

struct SimtProject {
    const float *up, *W;
    float *A;
    int64_t cols, ld;
    int d, k, split;
};

template <int WN, int JT>
__global__ void __launch_bounds__(PTHREADS) k_simt_project_a(const SimtProject p)
{
    constexpr int G = PTHREADS / 32 / WN, KP = WN * JT;
    constexpr int BROWS = PROWS * G;                // rows of W per CTA and step
    extern __shared__ __align__(16) float smp[];    // U [PSTEPS][BROWS / 2][KP][2], then W
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int group = warp / WN, jg = warp % WN;
    const int rank = (int)(blockIdx.x % p.split);
    const int64_t c0 = (int64_t)(blockIdx.x / p.split) * 128, c = c0 + 4 * lane;
    float *ws = smp + PSTEPS * BROWS * KP + 4 * tid;    // [PSTEPS][PROWS][PTHREADS][4]

    // this thread's 16 bytes of a row of W, zero-filled past the last column
    const unsigned wbytes = (unsigned)(4 * max((int64_t)0, min((int64_t)4, p.cols - c)));
    const float *wsrc = p.W + (wbytes ? c : 0);
    const int stride = BROWS * p.split;
    auto fetch = [&](int step) {
        const int row0 = rank * BROWS + step * stride, b = step % PSTEPS;
        if (row0 < p.d) {
            const int r = row0 + PROWS * group;
            if (r < p.d)                            // d is a multiple of 8: all rows or none
#pragma unroll
                for (int i = 0; i < PROWS; ++i)
                    cp_async_part(smem_addr(ws + (b * PROWS + i) * 4 * PTHREADS),
                                  wsrc + (int64_t)(r + i) * p.ld, wbytes);
            // u32p is padded to 32 rows past d
            const int n = min(BROWS, (p.d + 31) / 32 * 32 - row0) * KP / 4;
            const float *src = p.up + (int64_t)row0 * KP;
            const uint32_t dst = smem_addr(smp + b * BROWS * KP);
            for (int f = tid; f < n; f += PTHREADS)
                cp_async_16(dst + 16 * f, src + 4 * f);
        }
        cp_async_commit();
    };
    f32x2 acc[JT][2];
#pragma unroll
    for (int j = 0; j < JT; ++j)
        acc[j][0] = acc[j][1] = 0ull;
    griddep_wait();
#pragma unroll
    for (int s = 0; s < PSTEPS - 1; ++s)
        fetch(s);
    for (int it = 0, row = rank * BROWS; row < p.d; ++it, row += stride) {
        const int b = it % PSTEPS;
        cp_async_wait<PSTEPS - 2>();
        __syncthreads();                            // this step has landed, the last one is used up
        fetch(it + PSTEPS - 1);
        if (row + PROWS * group >= p.d)             // past the end: no rows were fetched
            continue;
        const float *ut = smp + b * BROWS * KP + PROWS * group * KP + 2 * jg * JT;
        const float *wt = ws + b * PROWS * 4 * PTHREADS;
#pragma unroll
        for (int i = 0; i < PROWS / 2; ++i) {
            const ulonglong2 w0 = *(const ulonglong2 *)(wt + 2 * i * 4 * PTHREADS);
            const ulonglong2 w1 = *(const ulonglong2 *)(wt + (2 * i + 1) * 4 * PTHREADS);
#pragma unroll
            for (int j = 0; j < JT; j += 2) {
                // (U[2i, j], U[2i + 1, j], U[2i, j + 1], U[2i + 1, j + 1])
                const float4 u = *(const float4 *)(ut + 2 * i * KP + 2 * j);
                const f32x2 a0 = pack2(u.x, u.x), a1 = pack2(u.y, u.y);
                const f32x2 b0 = pack2(u.z, u.z), b1 = pack2(u.w, u.w);
                acc[j][0] = fma2(a0, w0.x, acc[j][0]);
                acc[j][1] = fma2(a0, w0.y, acc[j][1]);
                acc[j + 1][0] = fma2(b0, w0.x, acc[j + 1][0]);
                acc[j + 1][1] = fma2(b0, w0.y, acc[j + 1][1]);
                acc[j][0] = fma2(a1, w1.x, acc[j][0]);
                acc[j][1] = fma2(a1, w1.y, acc[j][1]);
                acc[j + 1][0] = fma2(b1, w1.x, acc[j + 1][0]);
                acc[j + 1][1] = fma2(b1, w1.y, acc[j + 1][1]);
            }
        }
    }
    cp_async_wait_all();                            // (empty groups only)
    // partial sums [G][KP][128] of the groups, then of the cluster's CTAs
    float *red = smp;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < JT; ++j)
        *(ulonglong2 *)(red + ((size_t)group * KP + jg * JT + j) * 128 + 4 * lane) =
            make_ulonglong2(acc[j][0], acc[j][1]);
    __syncthreads();
    const int nout = p.k * 128;
    for (int e = tid; e < nout; e += PTHREADS) {
        float v = red[e];
#pragma unroll
        for (int g = 1; g < G; ++g)
            v += red[(size_t)g * KP * 128 + e];
        if (p.split > 1)
            red[e] = v;
        else if (c0 + (e & 127) < p.cols)
            p.A[(int64_t)(e >> 7) * p.cols + c0 + (e & 127)] = v;
    }
    if (p.split > 1) {
        cluster_sync();
        const int per = (nout + p.split - 1) / p.split;
        for (int e = rank * per + tid; e < min(nout, (rank + 1) * per); e += PTHREADS) {
            float v = 0.f;
            for (int r = 0; r < p.split; ++r)
                v += ld_cluster(smem_addr(red + e), r);
            if (c0 + (e & 127) < p.cols)
                p.A[(int64_t)(e >> 7) * p.cols + c0 + (e & 127)] = v;
        }
        cluster_sync();                             // no CTA leaves while its sums are read
    }
}

// ---- padded copies of U ---------------------------------------------------------
__global__ void k_prepare_basis(const float *__restrict__ U, int d, int k, int n_pad, int k64, int kp,
                                float *__restrict__ u32t, float *__restrict__ u32p,
                                __nv_bfloat16 *__restrict__ ut16, __nv_bfloat16 *__restrict__ up16)
{
    const int64_t n_t = (int64_t)k * d, n_ut = (int64_t)n_pad * d, n_up = (int64_t)d * k64;
    const int64_t n_p = (int64_t)((d + 31) / 32 * 32) * kp;
    const int64_t n = max(max(n_t, n_p), max(n_ut, n_up));
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (e < n_t) {            // u32t[j, i] = U[i, j]
            const int64_t j = e / d, i = e % d;
            u32t[e] = U[i * k + j];
        }
        if (e < n_p) {            // u32p[i / 2, j, i % 2] = U[i, j], zero for j >= k and i >= d
            const int64_t q = e >> 1, j = q % kp, i = 2 * (q / kp) + (e & 1);
            u32p[e] = j < k && i < d ? U[i * k + j] : 0.f;
        }
        if (e < n_ut) {           // ut16[j, i] = U[i, j], zero rows j >= k
            const int64_t j = e / d, i = e % d;
            ut16[e] = __float2bfloat16_rn(j < k ? U[i * k + j] : 0.f);
        }
        if (e < n_up) {           // up16[i, j] = U[i, j], zero columns j >= k
            const int64_t i = e / k64, j = e % k64;
            up16[e] = __float2bfloat16_rn(j < k ? U[i * k + j] : 0.f);
        }
    }
}

// Warps per group and columns per thread of the compress, and (times four) of the
// projection's first pass: the widths they are built for (at k = 20, 41 and 82
// the padded columns kp = 4 wn tn are 20, 48 and 96).
void compress_shape(int k, int *wn, int *tn)
{
    *wn = k <= 32 ? 1 : k <= 64 ? 2 : 4;
    const int t = (k + 4 * *wn - 1) / (4 * *wn);
    *tn = *wn == 1 ? (t == 7 ? 8 : t) : (t <= 6 ? 6 : 8);
}

template <int WN, int TN>
cudaError_t launch_compress_f32(SimtCompress p, bool gather, int sms, cudaStream_t s)
{
    constexpr int G = CTHREADS / 32 / WN, KP = 4 * TN * WN;
    constexpr size_t stage = sizeof(float) * G * (2 * CTOK * CPITCH + 2 * CCH * KP);
    constexpr size_t red = sizeof(float) * G * CTOK * (KP + 1);
    constexpr size_t smem = stage > red ? stage : red;
    const int64_t tiles = (p.T + CTOK - 1) / CTOK;
    const int steps = ((p.d + CCH - 1) / CCH + G - 1) / G;
    // registers let two (gather) or three CTAs share an SM for k = 13 .. 32; three or four
    // fit at other widths, where the split may come out larger than it need be
    p.split = cluster_split(tiles, steps, sms, gather ? 2 : 3, s);
    const unsigned grid = (unsigned)(tiles * p.split);
    void (*const kernel)(SimtCompress) =
        gather ? k_simt_compress<WN, TN, true> : k_simt_compress<WN, TN, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = launch_clusters(kernel, p.split, dim3(grid), dim3(CTHREADS), smem, s, p);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <bool EMB>
cudaError_t launch_expand_f32(const SimtExpand &p, int sms, cudaStream_t s)
{
    const int kq = (p.k + 1) & ~1;
    const int smem = (int)(sizeof(float) * 3 * ETILE * kq);
    cudaError_t e = cudaFuncSetAttribute(k_simt_expand<EMB>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess)
        return e;
    // CTAs per column tile: the least (rounds of the grid) x (row tiles per CTA + 1 for its
    // copy of R)
    const int64_t ctiles = (p.cols + ETILE - 1) / ETILE, rtiles = (p.rows + ETILE - 1) / ETILE;
    const int64_t slots = (int64_t)sms * (smem <= 110 << 10 ? 2 : 1);
    int64_t best = -1, gy = 1;
    for (int64_t y = 1; y <= rtiles && y <= 2 * slots; ++y) {
        const int64_t cost = (ctiles * y + slots - 1) / slots * ((rtiles + y - 1) / y + 1);
        if (best < 0 || cost < best) {
            best = cost;
            gy = y;
        }
    }
    e = launch_dependent(k_simt_expand<EMB>, dim3((unsigned)ctiles, (unsigned)gy), dim3(ETHREADS), smem,
                         s, p);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <bool EMB>
cudaError_t launch_expand_few(const SimtExpand &p, cudaStream_t s)
{
    const dim3 grid((unsigned)((p.cols + FTHREADS - 1) / FTHREADS), (unsigned)((p.rows + FROWS - 1) / FROWS));
    const cudaError_t e = launch_dependent(k_simt_expand_few<EMB>, grid, dim3(FTHREADS), 0, s, p);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int WN, int JT>
cudaError_t launch_project_a(SimtProject p, int sms, cudaStream_t s)
{
    constexpr int G = PTHREADS / 32 / WN, KP = WN * JT;
    constexpr size_t stage = sizeof(float) * PSTEPS * (PROWS * G * KP + PROWS * 4 * PTHREADS);
    constexpr size_t red = sizeof(float) * G * KP * 128;
    const int64_t tiles = (p.cols + 127) / 128;
    const int steps = (p.d + PROWS * G - 1) / (PROWS * G);
    p.split = cluster_split(tiles, steps, sms, 1, s);
    constexpr size_t smem = stage > red ? stage : red;
    cudaError_t e = cudaFuncSetAttribute(k_simt_project_a<WN, JT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = launch_clusters(k_simt_project_a<WN, JT>, p.split, dim3((unsigned)(tiles * p.split)),
                            dim3(PTHREADS), smem, s, p);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Where the kernel for few rows is the faster one.  Five of its CTAs fit an SM.  Without
// embeddings, as long as all are there at once (counted by their columns, four an SM: they
// are bound by their FMAs then): 1024 rows of d = 1000, k = 41 take 6.9 us, 9.4 with tiles;
// 2048 rows 11.8 and 9.5.  With embeddings the tile kernel takes its 128 columns in two
// halves and runs in rounds: of one tile an SM while there are no more, in the time of one
// round of the other's CTAs; else of two tiles an SM, in the time of 1.8 (2.05 for k > 32); for
// k > 72, whose shared memory leaves no room for a second tile, of one, in 1.3.  6001 rows
// of d = 1000, k = 41 take 33.7 us and 37.7 with tiles (3004 CTAs, two rounds), 2048 rows
// 16.4 and 15.1; 12000 rows of d = 200, k = 128 32.9 and 49.2, 2048 of 1000 33.4 and 26.1.
bool few_rows(const SimtExpand &p, bool emb, int sms)
{
    const int64_t ctas = (p.cols + FTHREADS - 1) / FTHREADS * ((p.rows + FROWS - 1) / FROWS);
    if (!emb)
        return ctas <= 5 * (int64_t)sms && std::min<int64_t>(p.cols, FTHREADS) * ctas <= 4 * FTHREADS * (int64_t)sms;
    const int64_t tiles = (p.cols + ETILE - 1) / ETILE * ((p.rows + ETILE - 1) / ETILE);
    const int64_t slots = p.k > 72 ? sms : 2 * sms, rounds = (tiles + slots - 1) / slots;
    const int64_t percent = tiles <= sms ? 100 : (p.k > 72 ? 130 : p.k > 32 ? 205 : 180) * rounds;
    return 100 * ctas <= 5 * sms * percent && (p.rows + FROWS - 1) / FROWS <= 65535;
}

int sm_count_f32(int device)
{
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n <= 0)
        n = 148;
    return n;
}

}  // namespace

int simt_padded_columns(int k)
{
    int wn, tn;
    compress_shape(k, &wn, &tn);
    return 4 * wn * tn;
}

cudaError_t simt_compress(const sn_basis &b, const float *X, const int32_t *ids, const int32_t *pos,
                          int64_t T, int seq_len, const float *tok, int64_t vocab, const float *pe,
                          float *C, bool gather, cudaStream_t s)
{
    SimtCompress p{b.u32p, X, tok, pe, ids, pos, C, b.err, T, vocab, b.d, b.k, seq_len, 1};
    const int sms = sm_count_f32(b.device);
    int wn, tn;
    compress_shape(b.k, &wn, &tn);
    switch (10 * wn + tn) {
    case 11: return launch_compress_f32<1, 1>(p, gather, sms, s);
    case 12: return launch_compress_f32<1, 2>(p, gather, sms, s);
    case 13: return launch_compress_f32<1, 3>(p, gather, sms, s);
    case 14: return launch_compress_f32<1, 4>(p, gather, sms, s);
    case 15: return launch_compress_f32<1, 5>(p, gather, sms, s);
    case 16: return launch_compress_f32<1, 6>(p, gather, sms, s);
    case 18: return launch_compress_f32<1, 8>(p, gather, sms, s);
    case 26: return launch_compress_f32<2, 6>(p, gather, sms, s);
    case 28: return launch_compress_f32<2, 8>(p, gather, sms, s);
    case 46: return launch_compress_f32<4, 6>(p, gather, sms, s);
    default: return launch_compress_f32<4, 8>(p, gather, sms, s);
    }
}

cudaError_t simt_decompress(const sn_basis &b, const float *C, const int32_t *ids,
                            const int32_t *pos, int64_t T, int seq_len, const float *tok,
                            int64_t vocab, const float *pe, float *X, bool gather, cudaStream_t s)
{
    const SimtExpand p{C, b.u32t, tok, pe, ids, pos, X, b.err, T, b.d, b.d, b.d, vocab, b.k, seq_len};
    const int sms = sm_count_f32(b.device);
    if (few_rows(p, gather, sms))
        return gather ? launch_expand_few<true>(p, s) : launch_expand_few<false>(p, s);
    return gather ? launch_expand_f32<true>(p, sms, s) : launch_expand_f32<false>(p, sms, s);
}

cudaError_t simt_project(const sn_basis &b, const float *W, int64_t cols, int64_t ld, float *W_out,
                         float *A, cudaStream_t s)
{
    const SimtProject a{b.u32p, W, A, cols, ld, b.d, b.k, 1};
    const int sms = sm_count_f32(b.device);
    int wn, tn;
    compress_shape(b.k, &wn, &tn);
    cudaError_t e;
    switch (10 * wn + tn) {
    case 11: e = launch_project_a<1, 4>(a, sms, s); break;
    case 12: e = launch_project_a<1, 8>(a, sms, s); break;
    case 13: e = launch_project_a<1, 12>(a, sms, s); break;
    case 14: e = launch_project_a<1, 16>(a, sms, s); break;
    case 15: e = launch_project_a<1, 20>(a, sms, s); break;
    case 16: e = launch_project_a<1, 24>(a, sms, s); break;
    case 18: e = launch_project_a<1, 32>(a, sms, s); break;
    case 26: e = launch_project_a<2, 24>(a, sms, s); break;
    case 28: e = launch_project_a<2, 32>(a, sms, s); break;
    case 46: e = launch_project_a<4, 24>(a, sms, s); break;
    default: e = launch_project_a<4, 32>(a, sms, s); break;
    }
    if (e != cudaSuccess)
        return e;
    const SimtExpand p{b.u32, A, nullptr, nullptr, nullptr, nullptr, W_out, b.err, b.d, cols, cols,
                       ld, 1, b.k, 1};
    return launch_expand_f32<false>(p, sms, s);
}

cudaError_t prepare_basis(sn_basis &b, const float *U, cudaStream_t s)
{
    cudaError_t e = cudaMemcpyAsync(b.u32, U, sizeof(float) * (size_t)b.d * b.k,
                                    cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess)
        return e;
    k_prepare_basis<<<304, 256, 0, s>>>(U, b.d, b.k, b.n_pad, b.k64, b.kp, b.u32t, b.u32p, b.ut16,
                                        b.up16);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sn
