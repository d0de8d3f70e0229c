// sn_lossy.cu — the lossy comparators of the paper's comparison at equal wire
// size (Sec. 8, "Comparison against lossy compressions"): per-row top-k, 1-bit
// sign quantization and row-scaled 8-bit quantization (int8, fp8 e4m3) of a
// bf16 batch, with their restores.
//
// Top-k keeps the kk entries of largest magnitude of each row, ties towards the
// lower column, and writes them in ascending column order.  One warp per row
// (grid-stride over rows, 8 warps a CTA, no block barriers); selection works
// on the 15-bit bf16 magnitude ("key"), lane l owning chunks l, l + 32, ... of
// 8 entries (16 bytes).
//
//   bound   Lane l keeps the M largest maxima of its chunks; the bound is the
//           q-th largest, over the lanes, of each lane's M-th (q = ceil(kk/M)).
//           q lanes then vouch for M distinct chunks each whose maximum
//           reaches the bound, so at least kk entries do: the kk-th largest
//           key is >= bound.  M = ceil(kk / 24), at most 4.
//   select  The chunks whose maximum reaches the bound are re-read (they are
//           still in L2) and their entries at or above it appended in column
//           order (about 2 kk of them on continuous data); the kk-th largest
//           key among those is found by a bit-by-bit search with warp counts,
//           and the kept entries are placed by ballot prefixes, the lowest
//           columns first among those equal to it.
//   exact   When more than kWCap chunks or entries reach the bound (many
//           equal keys, kk > 128) the same search and placement run over the
//           whole row, re-read from L2, skipping chunks whose maximum cannot
//           matter.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "sn_tc.cuh"

namespace sn {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kWCap = 256;                // candidate chunks and entries per warp
constexpr int kLoadBatch = 8;             // 16-byte loads in flight per lane (top-k)
constexpr int kSignUnroll = 8;            // 16-byte loads in flight per lane (sign)
constexpr int kQuantUnroll = 8;           // 16-byte loads in flight per lane (8-bit)

__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Largest magnitude key among the 8 bf16 of a chunk.
__device__ __forceinline__ int max_key8(uint4 v)
{
    const uint32_t c = max_u16x2(max_u16x2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu),
                                 max_u16x2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu));
    return (int)max(c & 0xFFFFu, c >> 16);
}

__device__ __forceinline__ int key_of(uint4 v, int e)
{
    const uint32_t w = e < 2 ? v.x : e < 4 ? v.y : e < 6 ? v.z : v.w;
    return (int)((w >> (16 * (e & 1))) & 0x7FFFu);
}

__device__ __forceinline__ uint32_t bits_of(uint4 v, int e)
{
    const uint32_t w = e < 2 ? v.x : e < 4 ? v.y : e < 6 ? v.z : v.w;
    return (w >> (16 * (e & 1))) & 0xFFFFu;
}

__device__ __forceinline__ int warp_count(bool p) { return __popc(__ballot_sync(0xffffffffu, p)); }

__device__ __forceinline__ uint32_t lanes_below()
{
    return (1u << (threadIdx.x & 31)) - 1u;
}

// Inclusive prefix sum over the warp.
__device__ __forceinline__ int warp_incl_scan(int n)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, n, o);
        n += lane >= o ? y : 0;
    }
    return n;
}

// Count of the chunk's entries whose key is >= thr.
__device__ __forceinline__ int count_ge8(uint4 v, int thr)
{
    int n = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
        n += key_of(v, e) >= thr;
    return n;
}

// Shared memory of one warp: chunk maxima, candidate chunks, candidate
// entries (bf16 bits | column << 16).
struct TopkWarpSmem {
    uint16_t *smax;
    uint16_t *clist;
    uint32_t *cand;
};

__host__ __device__ __forceinline__ int topk_region_bytes(int nch)
{
    return ((nch * 2 + 15) & ~15) + kWCap * 2 + kWCap * 4;
}

// Exact path: the kk-th largest key of the whole row and the placement of
// the kept entries in column order.
__device__ void topk_row_exact(const uint4 *src, int nch, int kk, const uint16_t *smax,
                               uint16_t *vo, uint16_t *co)
{
    const int lane = threadIdx.x & 31;
    int thr = 0;
    for (int bit = 14; bit >= 0; --bit) {
        const int trial = thr | (1 << bit);
        int cnt = 0;
        for (int c = lane; c < nch; c += 32)
            if ((int)smax[c] >= trial)
                cnt += count_ge8(__ldg(src + c), trial);
        if (__reduce_add_sync(0xffffffffu, cnt) >= kk)
            thr = trial;
    }
    int above = 0;
    for (int c = lane; c < nch; c += 32)
        if ((int)smax[c] > thr)
            above += count_ge8(__ldg(src + c), thr + 1);
    const int need = kk - __reduce_add_sync(0xffffffffu, above);
    int eq_before = 0, kept_before = 0;
    for (int c0 = 0; c0 < nch; c0 += 32) {                    // warp-uniform
        const int c = c0 + lane;
        const bool live = c < nch && (int)smax[c] >= thr;
        const uint4 v = live ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
        uint32_t eqf = 0, gtf = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = live ? key_of(v, e) : -1;
            eqf |= (k == thr ? 1u : 0u) << e;
            gtf |= (k > thr ? 1u : 0u) << e;
        }
        const int neq = __popc(eqf);
        const int eq_incl = warp_incl_scan(neq);
        int allowed = need - (eq_before + eq_incl - neq);     // ties this lane may still take
        uint32_t keep = gtf, rest = eqf;
        while (allowed > 0 && rest) {
            const uint32_t low = rest & (0u - rest);
            keep |= low;
            rest ^= low;
            --allowed;
        }
        const int nk = __popc(keep);
        const int k_incl = warp_incl_scan(nk);
        int p = kept_before + k_incl - nk;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if ((keep >> e) & 1u) {
                vo[p] = (uint16_t)bits_of(v, e);
                co[p] = (uint16_t)(8 * c + e);
                ++p;
            }
        eq_before += __shfl_sync(0xffffffffu, eq_incl, 31);
        kept_before += __shfl_sync(0xffffffffu, k_incl, 31);
    }
}

template <int M>
__global__ void __launch_bounds__(kThreads) k_topk(const uint16_t *__restrict__ X, int64_t T,
                                                    int d, int kk, uint16_t *__restrict__ vals,
                                                    uint16_t *__restrict__ cols)
{
    griddep_wait();
    extern __shared__ __align__(16) uint8_t tk_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nch = d / 8, per_lane = (nch + 31) / 32;
    uint8_t *base = tk_smem + warp * topk_region_bytes(nch);
    uint16_t *smax = (uint16_t *)base;
    uint16_t *clist = (uint16_t *)(base + ((nch * 2 + 15) & ~15));
    uint32_t *cand = (uint32_t *)(base + ((nch * 2 + 15) & ~15) + kWCap * 2);
    const int q = M > 0 ? (kk + M - 1) / M : 33;
    const int64_t nwarps = (int64_t)gridDim.x * kWarps;
    for (int64_t t = (int64_t)blockIdx.x * kWarps + warp; t < T; t += nwarps) {
        const uint4 *src = (const uint4 *)(X + t * (int64_t)d);
        uint16_t *vo = vals + t * kk;
        uint16_t *co = cols + t * kk;
        __syncwarp();                         // the previous row is done with smax, clist, cand
        // pass 1: chunk maxima, and each lane's M largest
        int top[M > 0 ? M : 1];
#pragma unroll
        for (int j = 0; j < (M > 0 ? M : 1); ++j)
            top[j] = -1;
        for (int i0 = 0; i0 < per_lane; i0 += kLoadBatch) {
            uint4 v[kLoadBatch];
#pragma unroll
            for (int u = 0; u < kLoadBatch; ++u) {
                const int c = lane + 32 * (i0 + u);
                v[u] = c < nch ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kLoadBatch; ++u) {
                const int c = lane + 32 * (i0 + u);
                if (c < nch) {
                    int x = max_key8(v[u]);
                    smax[c] = (uint16_t)x;
#pragma unroll
                    for (int j = 0; j < M; ++j) {
                        const int hi = max(top[j], x);
                        x = min(top[j], x);
                        top[j] = hi;
                    }
                }
            }
        }
        int bound = -1;
        if (M > 0 && q <= 32) {
            // (the lanes' values agree above their first differing bit, and a bound
            // up to 3 keys low only admits a few more candidates; for M = 4, where those
            // few can be more than a warp holds, it is searched to the last bit: T = 16384,
            // d = 4096, kk = 96 took 81 us with the low bound, now 53)
            const int vl = top[M > 0 ? M - 1 : 0];
            const int hi = max(__reduce_max_sync(0xffffffffu, vl), 0);
            const int lo = max(__reduce_min_sync(0xffffffffu, vl), 0);
            int bit = 31 - __clz(lo ^ hi);
            int b = hi & ~((1 << (bit + 1)) - 1);
            for (; bit >= (M < 4 ? 2 : 0); --bit)
                if (warp_count(vl >= (b | (1 << bit))) >= q)
                    b |= 1 << bit;
            bound = warp_count(vl >= b) >= q ? b : -1;
        }
        __syncwarp();                         // smax visible to the whole warp
        // candidate chunks, in column order
        int nchk = 0;
        for (int i = 0; i < per_lane; ++i) {
            const int c = lane + 32 * i;
            const bool hit = c < nch && (int)smax[c] >= bound;
            const uint32_t bal = __ballot_sync(0xffffffffu, hit);
            const int p = nchk + __popc(bal & lanes_below());
            if (hit && p < kWCap)
                clist[p] = (uint16_t)c;
            nchk += __popc(bal);
        }
        bool exact = nchk > kWCap;
        int nc = 0;
        if (!exact) {
            __syncwarp();
            for (int r0 = 0; r0 < nchk; r0 += 32) {           // warp-uniform
                const int j = r0 + lane;
                const int c = j < nchk ? (int)clist[j] : 0;
                const uint4 v = j < nchk ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
                uint32_t f = 0;
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    f |= (j < nchk && key_of(v, e) >= bound ? 1u : 0u) << e;
                const int n = __popc(f);
                const int incl = warp_incl_scan(n);
                int p = nc + incl - n;
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if ((f >> e) & 1u) {
                        if (p < kWCap)
                            cand[p] = bits_of(v, e) | ((uint32_t)(8 * c + e) << 16);
                        ++p;
                    }
                nc += __shfl_sync(0xffffffffu, incl, 31);
            }
            exact = nc > kWCap;
        }
        if (exact) {
            topk_row_exact(src, nch, kk, smax, vo, co);
            continue;
        }
        __syncwarp();                         // cand visible to the whole warp
        // every entry at or above the bound is a candidate, so for any trial
        // the candidate count decides "at least kk entries reach it" as the
        // whole row would
        // (the candidates' keys stay in registers; thr lies between the bound and the row's
        // largest key, so their common bits are not searched.  T = 16384, d = 4096, kk = 20:
        // 45 -> 33 us with the same shortcut for the bound above.  Up to 64 candidates
        // two votes count them, past that the lanes' own counts and one sum: with a vote
        // per 32 candidates read from shared memory, T = 30000, d = 1024, kk = 64 took 82
        // us instead of 63)
        constexpr int kKeys = kWCap / 32;
        int key[kKeys];
#pragma unroll
        for (int i = 0; i < kKeys; ++i)
            key[i] = lane + 32 * i < nc ? (int)(cand[lane + 32 * i] & 0x7FFFu) : -1;
        auto reach = [&](int trial) {
            if (nc <= 64)                                                  // warp-uniform
                return warp_count(key[0] >= trial) + warp_count(key[1] >= trial);
            int cnt = 0;
#pragma unroll
            for (int i = 0; i < kKeys; ++i)
                cnt += key[i] >= trial;
            return (int)__reduce_add_sync(0xffffffffu, cnt);
        };
        int rmax = key[0];
#pragma unroll
        for (int i = 1; i < kKeys; ++i)
            rmax = max(rmax, key[i]);
        rmax = __reduce_max_sync(0xffffffffu, rmax);
        int bit = 31 - __clz(rmax ^ max(bound, 0));
        int thr = rmax & ~((1 << (bit + 1)) - 1);
        for (; bit >= 0; --bit)
            if (reach(thr | (1 << bit)) >= kk)
                thr |= 1 << bit;
        const int need = kk - reach(thr + 1);
        int eq_before = 0, kept_before = 0;
        for (int r0 = 0; r0 < nc; r0 += 32) {                 // warp-uniform
            const int j = r0 + lane;
            const uint32_t cj = j < nc ? cand[j] : 0u;
            const int k = j < nc ? (int)(cj & 0x7FFFu) : -1;
            const uint32_t be = __ballot_sync(0xffffffffu, k == thr);
            const bool keep = k > thr || (k == thr && eq_before + __popc(be & lanes_below()) < need);
            const uint32_t bk = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int p = kept_before + __popc(bk & lanes_below());
                vo[p] = (uint16_t)(cj & 0xFFFFu);
                co[p] = (uint16_t)(cj >> 16);
            }
            eq_before += __popc(be);
            kept_before += __popc(bk);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_topk_restore(const uint16_t *__restrict__ vals,
                                                            const uint16_t *__restrict__ cols,
                                                            int64_t T, int d, int kk,
                                                            uint16_t *__restrict__ out)
{
    griddep_wait();
    for (int64_t t = blockIdx.x; t < T; t += gridDim.x) {
        uint16_t *dst = out + t * (int64_t)d;
        __syncthreads();
        for (int c = threadIdx.x; c < d / 8; c += kThreads)
            ((uint4 *)dst)[c] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        for (int j = threadIdx.x; j < kk; j += kThreads)
            dst[cols[t * kk + j]] = vals[t * kk + j];
    }
}

// Sign quantization: one warp per row; lane l of a 256-column slab reads its
// 8 entries as one 16-byte load, forms their 8 sign bits (1 for a negative
// nonzero entry; NaN inputs are outside the comparator's domain), and 4 lanes
// merge their bytes into one 32-bit word.  The row scale is the mean
// magnitude, summed per chunk, then per lane, then across the warp in fp32.
__global__ void __launch_bounds__(kThreads) k_sign(const uint16_t *__restrict__ X, int64_t T, int d,
                                                    uint32_t *__restrict__ bits,
                                                    float *__restrict__ scale)
{
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    const int nch = d / 8, words = (d + 31) / 32;
    for (int64_t t = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; t < T; t += nwarps) {
        const uint4 *src = (const uint4 *)(X + t * (int64_t)d);
        uint32_t *dst = bits + t * words;
        float s = 0.f;
        for (int base = 0; base < nch; base += kSignUnroll * 32) {     // warp-uniform
            uint4 v[kSignUnroll];
#pragma unroll
            for (int u = 0; u < kSignUnroll; ++u) {
                const int c = base + 32 * u + lane;
                v[u] = c < nch ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kSignUnroll; ++u) {
                const int c = base + 32 * u + lane;
                const uint32_t wd[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                // per 32-bit word: sign AND "magnitude nonzero" (adding 0x7FFF
                // to a 15-bit magnitude carries into bit 15 exactly when it is
                // not 0), moved so word e's two bits land on 2e and 16 + 2e
                uint32_t x = 0;
                float cs = 0.f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t w = wd[e];
                    x |= (w & ((w & 0x7FFF7FFFu) + 0x7FFF7FFFu) & 0x80008000u) >> (15 - 2 * e);
                    cs += fabsf(__uint_as_float(w << 16)) + fabsf(__uint_as_float(w & 0xFFFF0000u));
                }
                const uint32_t byte = (x | (x >> 15)) & 0xFFu;
                s += cs;
                uint32_t wv = byte << (8 * (lane & 3));
                wv |= __shfl_xor_sync(0xffffffffu, wv, 1);
                wv |= __shfl_xor_sync(0xffffffffu, wv, 2);
                if ((lane & 3) == 0 && (c >> 2) < words)
                    dst[c >> 2] = wv;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0)
            scale[t] = s / (float)d;
    }
}

// Restore: one warp per row, one 16-byte store of 8 entries per lane.
__global__ void __launch_bounds__(kThreads) k_sign_restore(const uint32_t *__restrict__ bits,
                                                            const float *__restrict__ scale,
                                                            int64_t T, int d,
                                                            uint16_t *__restrict__ out)
{
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    const int nch = d / 8, words = (d + 31) / 32;
    for (int64_t t = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; t < T; t += nwarps) {
        const __nv_bfloat16 pos = __float2bfloat16_rn(scale[t]);
        const __nv_bfloat16 neg = __float2bfloat16_rn(-scale[t]);
        const uint32_t p = *(const uint16_t *)&pos, n = *(const uint16_t *)&neg;
        uint4 *dst = (uint4 *)(out + t * (int64_t)d);
        for (int c = lane; c < nch; c += 32) {
            const uint32_t byte = (bits[t * words + (c >> 2)] >> (8 * (c & 3))) & 0xFFu;
            uint32_t wd[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                wd[e] = ((byte >> (2 * e)) & 1u ? n : p) | (((byte >> (2 * e + 1)) & 1u ? n : p) << 16);
            dst[c] = make_uint4(wd[0], wd[1], wd[2], wd[3]);
        }
    }
}

// ---- Row-scaled 8-bit quantization -------------------------------------------
// a = max |x| of the row, scale = a / qmax, code = Q(x * r) with r = qmax / a
// (0 for a zero row): int8 rounds half to even and clamps to +-127, fp8 e4m3
// rounds to nearest even and saturates at +-448.  The code is decided in fp32
// from one rounded division per row and one rounded product per entry.

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// the four codes of one packed word pair of bf16 (entries 0..3 in bytes 0..3)
template <int FMT>
__device__ __forceinline__ uint32_t quant4(uint32_t w0, uint32_t w1, float r)
{
    const float x0 = __fmul_rn(bf16_lo(w0), r), x1 = __fmul_rn(bf16_hi(w0), r);
    const float x2 = __fmul_rn(bf16_lo(w1), r), x3 = __fmul_rn(bf16_hi(w1), r);
    if (FMT == SN_Q_INT8) {
        // |x| <= 127 (1 + 2^-23), so rint(x) already lies in [-127, 127].  Adding
        // 1.5 * 2^23 rounds x to an integer (the fp32 addition rounds to nearest
        // even at unit spacing) held in the low mantissa bits, whose low byte is
        // rint(x) in two's complement; byte permutes gather the four low bytes.
        constexpr float kRound = 12582912.0f;
        const uint32_t q0 = __float_as_uint(__fadd_rn(x0, kRound));
        const uint32_t q1 = __float_as_uint(__fadd_rn(x1, kRound));
        const uint32_t q2 = __float_as_uint(__fadd_rn(x2, kRound));
        const uint32_t q3 = __float_as_uint(__fadd_rn(x3, kRound));
        return __byte_perm(__byte_perm(q0, q1, 0x0040), __byte_perm(q2, q3, 0x0040), 0x5410);
    }
    const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(x0, x1), __NV_SATFINITE, __NV_E4M3);
    const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(x2, x3), __NV_SATFINITE, __NV_E4M3);
    return lo | (hi << 16);
}

// One warp per row.  Pass 1 takes the largest magnitude from the low 15 bits
// of every bf16 (they order the magnitudes of finite values); pass 2 reads
// the row again (from L2) and writes each 16-byte chunk's 8 codes with one
// 8-byte store, the warp's 32 stores one contiguous 256-byte run.
template <int FMT>
__global__ void __launch_bounds__(kThreads) k_quant(const uint16_t *__restrict__ X, int64_t T, int d,
                                                     uint8_t *__restrict__ codes,
                                                     float *__restrict__ scale)
{
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    const int nch = d / 8;
    const float qmax = FMT == SN_Q_INT8 ? 127.f : 448.f;
    for (int64_t t = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; t < T; t += nwarps) {
        const uint4 *src = (const uint4 *)(X + t * (int64_t)d);
        uint32_t m = 0;
        for (int base = 0; base < nch; base += kQuantUnroll * 32) {
            uint4 v[kQuantUnroll];
#pragma unroll
            for (int u = 0; u < kQuantUnroll; ++u) {
                const int c = base + 32 * u + lane;
                v[u] = c < nch ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kQuantUnroll; ++u)
                m = max_u16x2(m, max_u16x2(max_u16x2(v[u].x & 0x7FFF7FFFu, v[u].y & 0x7FFF7FFFu),
                                           max_u16x2(v[u].z & 0x7FFF7FFFu, v[u].w & 0x7FFF7FFFu)));
        }
        m = __reduce_max_sync(0xffffffffu, max(m & 0xFFFFu, m >> 16));
        const float a = __uint_as_float(m << 16);
        const float r = a > 0.f ? qmax / a : 0.f;
        uint2 *dst = (uint2 *)(codes + t * (int64_t)d);
        for (int base = 0; base < nch; base += kQuantUnroll * 32) {
            uint4 v[kQuantUnroll];
#pragma unroll
            for (int u = 0; u < kQuantUnroll; ++u) {
                const int c = base + 32 * u + lane;
                v[u] = c < nch ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < kQuantUnroll; ++u) {
                const int c = base + 32 * u + lane;
                if (c < nch)
                    dst[c] = make_uint2(quant4<FMT>(v[u].x, v[u].y, r), quant4<FMT>(v[u].z, v[u].w, r));
            }
        }
        if (lane == 0)
            scale[t] = a / qmax;
    }
}

// the values of four codes (bytes 0..3 of q)
template <int FMT>
__device__ __forceinline__ void dequant4(uint32_t q, float (&f)[4])
{
    if (FMT == SN_Q_INT8) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            f[e] = (float)(int8_t)(q >> (8 * e));
        return;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const __half2_raw raw =
            __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(q >> (16 * h)), __NV_E4M3);
        const float2 v = __half22float2(__half2(raw));
        f[2 * h] = v.x;
        f[2 * h + 1] = v.y;
    }
}

__device__ __forceinline__ uint32_t bf16x2_rn(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *(const uint32_t *)&v;
}

// Restore: one warp per row; per lane 8 codes in, decode(code) * scale in
// fp32, one rounding to bf16, one 16-byte store.
template <int FMT>
__global__ void __launch_bounds__(kThreads) k_quant_restore(const uint8_t *__restrict__ codes,
                                                             const float *__restrict__ scale,
                                                             int64_t T, int d,
                                                             uint16_t *__restrict__ out)
{
    griddep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    const int nch = d / 8;
    for (int64_t t = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; t < T; t += nwarps) {
        const float s = scale[t];
        const uint2 *src = (const uint2 *)(codes + t * (int64_t)d);
        uint4 *dst = (uint4 *)(out + t * (int64_t)d);
        for (int c = lane; c < nch; c += 32) {
            const uint2 q = __ldg(src + c);
            float f[8];
            dequant4<FMT>(q.x, *(float(*)[4])f);
            dequant4<FMT>(q.y, *(float(*)[4])(f + 4));
            dst[c] = make_uint4(bf16x2_rn(f[0] * s, f[1] * s), bf16x2_rn(f[2] * s, f[3] * s),
                                bf16x2_rn(f[4] * s, f[5] * s), bf16x2_rn(f[6] * s, f[7] * s));
        }
    }
}

int row_grid(int64_t T)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int)(T < 8 * (int64_t)sms ? T : 8 * (int64_t)sms);
}

// One warp per row: at most 8 resident CTAs of 8 warps per SM.
int warp_grid(int64_t T)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t need = (T + kWarps - 1) / kWarps;
    return (int)(need < 8 * (int64_t)sms ? need : 8 * (int64_t)sms);
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), int grid, size_t smem, cudaStream_t s, const Args &...args)
{
    const cudaError_t e = launch_dependent(kernel, dim3(grid), dim3(kThreads), smem, s, args...);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int M>
cudaError_t launch_topk(const void *X, int64_t T, int d, int kk, void *vals, uint16_t *cols,
                        cudaStream_t s)
{
    const size_t smem = (size_t)kWarps * topk_region_bytes(d / 8);
    cudaError_t e = cudaFuncSetAttribute(k_topk<M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess)
        return e;
    int dev = 0, sms = 148, per_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_topk<M>, kThreads, smem);
    if (e != cudaSuccess)
        return e;
    const int64_t resident = (int64_t)sms * (per_sm > 0 ? per_sm : 1);   // one wave
    const int64_t need = (T + kWarps - 1) / kWarps;
    return launch(k_topk<M>, (int)(need < resident ? need : resident), smem, s, (const uint16_t *)X, T, d,
                  kk, (uint16_t *)vals, cols);
}

}  // namespace

cudaError_t lossy_topk(const void *X, int64_t T, int d, int kk, void *vals, uint16_t *cols,
                       cudaStream_t s)
{
    // M = ceil(kk / 24) chunk maxima vouched for per lane; past 4 the bound
    // is too loose to pay and every row takes the exact path
    const int m = (kk + 23) / 24;
    switch (m) {
    case 1: return launch_topk<1>(X, T, d, kk, vals, cols, s);
    case 2: return launch_topk<2>(X, T, d, kk, vals, cols, s);
    case 3: return launch_topk<3>(X, T, d, kk, vals, cols, s);
    case 4: return launch_topk<4>(X, T, d, kk, vals, cols, s);
    default: return launch_topk<0>(X, T, d, kk, vals, cols, s);
    }
}

cudaError_t lossy_topk_restore(const void *vals, const uint16_t *cols, int64_t T, int d, int kk,
                               void *out, cudaStream_t s)
{
    return launch(k_topk_restore, row_grid(T), 0, s, (const uint16_t *)vals, cols, T, d, kk,
                  (uint16_t *)out);
}

cudaError_t lossy_sign(const void *X, int64_t T, int d, uint32_t *bits, float *scale,
                       cudaStream_t s)
{
    return launch(k_sign, warp_grid(T), 0, s, (const uint16_t *)X, T, d, bits, scale);
}

// The 8-bit quantizer reads every row twice; the second read hits L2 only if
// the rows in flight (one per warp) stay well inside it, so the grid keeps
// them under 48 MiB: 2 CTAs of 8 warps per SM at d = 8192, up to 8 for short
// rows.
int quant_grid(int64_t T, int d)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t per_sm = ((int64_t)48 << 20) / ((int64_t)sms * kWarps * 2 * d);
    const int64_t ctas = (per_sm < 1 ? 1 : per_sm > 8 ? 8 : per_sm) * sms;
    const int64_t need = (T + kWarps - 1) / kWarps;
    return (int)(need < ctas ? need : ctas);
}

cudaError_t lossy_quant(const void *X, int64_t T, int d, int format, uint8_t *codes, float *scale,
                        cudaStream_t s)
{
    const int grid = quant_grid(T, d);
    return launch(format == SN_Q_INT8 ? k_quant<SN_Q_INT8> : k_quant<SN_Q_E4M3>, grid, 0, s,
                  (const uint16_t *)X, T, d, codes, scale);
}

cudaError_t lossy_quant_restore(const uint8_t *codes, const float *scale, int64_t T, int d,
                                int format, void *out, cudaStream_t s)
{
    return launch(format == SN_Q_INT8 ? k_quant_restore<SN_Q_INT8> : k_quant_restore<SN_Q_E4M3>,
                  warp_grid(T), 0, s, codes, scale, T, d, (uint16_t *)out);
}

cudaError_t lossy_sign_restore(const uint32_t *bits, const float *scale, int64_t T, int d,
                               void *out, cudaStream_t s)
{
    return launch(k_sign_restore, warp_grid(T), 0, s, bits, scale, T, d, (uint16_t *)out);
}

}  // namespace sn
