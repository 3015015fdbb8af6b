// ptf.cu -- Power-of-Two Factor calibration (Sec. 3.2, Eqs. 8-10) and the
// PTF quantizer (Eq. 7) on sm_103a.
//
// Calibration runs in two launches on the caller's stream (a calibration
// batch split by rows over several ranks runs each per rank, with the range and
// the sums exchanged in between; see fqvit_calibrate_minmax / _sse_partial /
// _combine); with more than four factors a third takes the argmin:
//   1. per-block min / max of the calibration batch (exact fp32 compares);
//   2. every block folds the partials into s, zp (Eqs. 8-9), then a warp per
//      (channel, factor) sums the squared quantization error of Eq. 10 over
//      the rows, in ascending row order, in fp64, and the block's channels
//      take the smallest factor with the least error.  Few rows (the rule is at launch_sse): a
//      thread per sum.
//
// The fp64 sums.  The order fixes the rounding of every step, and fp64 is slow
// on this GPU (one thread per sum took 1.0 ms for 6304 rows of 384 channels,
// about 300 cycles a row).  But the terms are squares of fp32 numbers: exact
// integers m 2^k with m < 2^48.  While the accumulator M 2^u (2^52 <= M < 2^53)
// stays in its binade, adding a term is M += n with n the term in units of 2^u
// rounded to nearest, which does not depend on M, except that a tie goes to the
// even sum.  So a warp takes 32 rows at a time: every lane rounds its row's
// term, the lanes with a tie look up the parity of the sum before them (a tie
// leaves it even, so it is the parity of the terms since the last tie: two
// ballots), and one reduction adds the 32 integers.  When the sum leaves the
// binade (at most a few dozen times per sum, and at the start) the rows before
// the one that crosses are added, that one with a real fp64 addition, and the
// rest rounded anew.  The same bits as the sequential sum.
// Measured: the calibration of 6304 x 384 (K = 3) 1000 -> 84 us; with its quantization and the read
// back of s and zp between them 1036 -> 160 us.
#include "fqvit_internal.cuh"

#include <cfloat>

namespace fqvit {

namespace {

constexpr int kMaxPartials = 1024;  // blocks of the min/max pass
constexpr int kWsHeader = 64;       // s0, zp, flags

__device__ __forceinline__ float pow2f(int e)  // 2^e for -126 <= e <= 127, exact
{
    return __int_as_float((e + 127) << 23);
}

__global__ void __launch_bounds__(256) minmax_partial_kernel(const float *__restrict__ x, int64_t rows, int C,
                                                             int64_t ld, float2 *__restrict__ part)
{
    pdl_release();
    pdl_wait();
    float mn = FLT_MAX, mx = -FLT_MAX;
    auto take = [&](float v) {
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
    };
    if (C % 4 == 0 && ld % 4 == 0 && ((uintptr_t)x % 16) == 0) {  // 16-byte loads, four rows' in flight
        const int cv = C >> 2, tr = min(cv, (int)blockDim.x), rpb = blockDim.x / tr;
        const int rl = threadIdx.x / tr, cl = threadIdx.x - rl * tr;
        const int64_t step = (int64_t)gridDim.x * rpb;
        if (rl < rpb)
            for (int c = cl; c < cv; c += tr) {
                const float4 *col = reinterpret_cast<const float4 *>(x) + c;
                const int64_t l4 = ld >> 2;
                for (int64_t r = (int64_t)blockIdx.x * rpb + rl; r < rows; r += 4 * step) {
                    float4 v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = __ldg(col + (r + i * step < rows ? r + i * step : r) * l4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) take(v[i].x), take(v[i].y), take(v[i].z), take(v[i].w);
                }
            }
    } else {
        for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
            const float *xr = x + r * ld;
            for (int c = threadIdx.x; c < C; c += blockDim.x) take(__ldg(xr + c));
        }
    }
    __shared__ float smn[32], smx[32];
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        smn[w] = mn;
        smx[w] = mx;
    }
    __syncthreads();
    if (w == 0) {
        int nw = blockDim.x >> 5;
        mn = l < nw ? smn[l] : FLT_MAX;
        mx = l < nw ? smx[l] : -FLT_MAX;
        for (int o = 16; o > 0; o >>= 1) {
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (l == 0) part[blockIdx.x] = make_float2(mn, mx);
    }
}

// Folds the min / max partials of one shard into mnmx[2].
__global__ void minmax_final_kernel(const float2 *__restrict__ part, int nparts, float *__restrict__ mnmx)
{
    float mn = FLT_MAX, mx = -FLT_MAX;
    for (int i = threadIdx.x; i < nparts; i += 32) {
        float2 p = part[i];
        mn = fminf(mn, p.x);
        mx = fmaxf(mx, p.y);
    }
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (threadIdx.x == 0) {
        mnmx[0] = mn;
        mnmx[1] = mx;
    }
}

// One (channel, factor) sum of Eq. 10, held by a whole warp: acc = M 2^u, 2^52 <= M < 2^53, or M = 0
struct SeqSum {
    unsigned long long M = 0;
    int u = 0;

    __device__ __forceinline__ void set(double acc)  // acc > 0, normal (squares of fp32 are at least 2^-298)
    {
        const unsigned long long b = (unsigned long long)__double_as_longlong(acc);
        M = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
        u = (int)(b >> 52) - 1075;
    }
    __device__ __forceinline__ double value() const
    {
        return M == 0 ? 0.0
                      : __longlong_as_double((long long)(((unsigned long long)(u + 1075) << 52) |
                                                         (M & 0xFFFFFFFFFFFFFull)));
    }
    // d^2 = m 2^k
    static __device__ __forceinline__ void square(float d, unsigned long long &m, int &k)
    {
        const uint32_t b = __float_as_uint(d) & 0x7FFFFFFFu, ef = b >> 23;
        const uint32_t mant = ef ? (b & 0x7FFFFFu) | 0x800000u : b;
        m = (unsigned long long)mant * mant;
        k = 2 * ((int)(ef ? ef : 1) - 150);
    }

    // adds d[g]^2 of the lanes of groups 0 .. 3, in that order, where the sum stays in its binade (the usual
    // case: four groups' roundings side by side, one reduction); else (an infinity or a NaN among them too) does
    // nothing and returns false
    __device__ __forceinline__ bool add128(const float (&d)[4])
    {
        constexpr unsigned long long kTop = 1ull << 53;
        const uint32_t full = 0xffffffffu;
        const uint32_t below = (1u << (threadIdx.x & 31)) - 1u;
        // terms of k <= u + 10 can be rounded in 64 bits: the bits of |d| below those of the first exponent past it
        const int last = min(((u + 10) >> 1) + 150, 254);
        const uint32_t top = last >= 1 ? (uint32_t)(last + 1) << 23 : 1u;
        unsigned long long n[4];
        bool tie[4], fits = M != 0;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            unsigned long long m;
            int k;
            square(d[g], m, k);
            const int r = min(u - k, 50);  // 50: the term rounds to 0
            fits = fits && (__float_as_uint(d[g]) & 0x7FFFFFFFu) < top;
            const unsigned long long t = m + ((1ull << (r & 63)) >> 1);  // (r > 0)
            n[g] = r > 0 ? t >> (r & 63) : m << (-r & 63);  // rounded to nearest, a tie up; or exact
            tie[g] = r > 0 && (n[g] << (r & 63)) == t;
        }
        if (!__all_sync(full, fits)) return false;
        uint32_t par = (uint32_t)M;  // parity of the sum before the group
        unsigned long long nn = 0;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint32_t ties = __ballot_sync(full, tie[g]), odd = __ballot_sync(full, !tie[g] && (n[g] & 1));
            if (ties) {  // warp-uniform
                const uint32_t prev = ties & below;
                const uint32_t since = prev ? below & ~((2u << (31 - __clz(prev))) - 1u) : below;
                const uint32_t before = __popc(odd & since) + (prev ? 0u : par);
                if (tie[g]) n[g] -= (before + (uint32_t)n[g]) & 1u;  // up if that makes the sum even, else down
                par = __popc(odd & ~((2u << (31 - __clz(ties))) - 1u));
            } else {
                par += __popc(odd);
            }
            nn += n[g];
        }
        nn = min(nn, kTop);
        const unsigned long long lo = __reduce_add_sync(full, (uint32_t)(nn & 0x7FFFFFFu));
        const unsigned long long hi = __reduce_add_sync(full, (uint32_t)(nn >> 27));
        const unsigned long long tot = lo + (hi << 27);
        if (M + tot >= kTop) return false;
        M += tot;
        return true;
    }

    // adds d^2 of lanes 0 .. 31, in that order, each addition rounded to nearest even (d = 0: no term).  An
    // infinite or NaN term takes the fp64 addition, as a crossing; the sum is then an M 2^u as well, whose u (972
    // or more) no finite term reaches.
    __device__ __forceinline__ void add32(float d)
    {
        constexpr unsigned long long kTop = 1ull << 53;
        const uint32_t full = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        unsigned long long m;
        int k;
        square(d, m, k);
        uint32_t left = full;  // lanes not added yet (a suffix)
        while (true) {
            if (M == 0) {
                const uint32_t nz = __ballot_sync(full, m != 0) & left;
                if (nz == 0) return;
                const int j = __ffs(nz) - 1;
                const double dj = (double)__shfl_sync(full, d, j);
                set(__dmul_rn(dj, dj));
                left &= ~((2u << j) - 1u);
            }
            // the term in units of 2^u: n, its floor where it is a tie (capped: a sum of 2^53 is a crossing)
            const int sh = isfinite(d) ? k - u : 11;
            unsigned long long n = 0;
            bool tie = false;
            if ((left >> lane) & 1u) {
                if (sh >= 0) {
                    n = sh > 10 ? (m ? kTop : 0ull) : min(m << sh, kTop);
                } else if (sh > -50) {
                    const int r = -sh;
                    n = m >> r;
                    const unsigned long long rem = m & ((1ull << r) - 1), half = 1ull << (r - 1);
                    tie = rem == half;
                    n += rem > half;
                }
            }
            const uint32_t ties = __ballot_sync(full, tie);
            if (ties) {  // the sum before a tie: even after the last tie, else M's parity, plus the terms since
                const uint32_t odd = __ballot_sync(full, !tie && (n & 1));
                const uint32_t below = (1u << lane) - 1u, prev = ties & below;
                const uint32_t since = prev ? below & ~((2u << (31 - __clz(prev))) - 1u) : below;
                const uint32_t par = __popc(odd & since) + (prev ? 0u : (uint32_t)M);
                if (tie) n += (par + (uint32_t)n) & 1u;
            }
            const unsigned long long lo = __reduce_add_sync(full, (uint32_t)(n & 0x7FFFFFFu));
            const unsigned long long hi = __reduce_add_sync(full, (uint32_t)(n >> 27));
            const unsigned long long tot = lo + (hi << 27);
            if (M + tot < kTop) {
                M += tot;
                return;
            }
            // the sum leaves its binade: add the lanes before the first that crosses, then that one in fp64
            unsigned long long pre = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long t = __shfl_up_sync(full, pre, o);
                if (lane >= o) pre += t;
            }
            const int j = __ffs(__ballot_sync(full, M + pre >= kTop)) - 1;
            M += __shfl_sync(full, pre - n, j);
            const double dj = (double)__shfl_sync(full, d, j);
            set(__dadd_rn(value(), __dmul_rn(dj, dj)));
            left &= ~((2u << j) - 1u);
            if (left == 0) return;
        }
    }
};

// Rows of a stage: warps meet once per stage; with 128 rows every stage waited for some warp's binade
// crossing (6304 x 192: 91 us, with 1024 rows 62).  Channels of a block: the sums are bound by their
// instructions, so few, spread over the chip (6304 x 768: 2 channels 114 us, 4 channels 149).
constexpr int kSseRows = 1024, CH = 2;
constexpr int kSseFactors = 4;   // factors per block

// The range (min, max) of the partials part[nparts], to every thread of the block
__device__ __forceinline__ void fold_range(const float *__restrict__ part, int nparts, float &mn, float &mx)
{
    __shared__ float2 red[32];
    const int tid = threadIdx.x, nthreads = blockDim.x;
    mn = FLT_MAX, mx = -FLT_MAX;
    for (int i = tid; i < nparts; i += nthreads) {
        mn = fminf(mn, part[2 * i]);  // (a caller's range need not be 8-byte aligned)
        mx = fmaxf(mx, part[2 * i + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((tid & 31) == 0) red[tid >> 5] = make_float2(mn, mx);
    __syncthreads();
    for (int w = 0; w < nthreads / 32; ++w) {
        mn = fminf(mn, red[w].x);
        mx = fmaxf(mx, red[w].y);
    }
}

// The smallest factor with the least of a channel's errors err[0], err[step] .. err[K step]
__device__ __forceinline__ uint8_t least(const double *err, int step, int K)
{
    int ba = 0;
    for (int k = 1; k <= K; ++k)
        if (err[k * step] < err[ba * step]) ba = k;
    return (uint8_t)ba;
}

// Eq. 10 for few rows: a thread per (channel, factor), 32 channels a block, a warp per factor.  Bound by the chain
// of fp64 additions, 0.16 us a row, up to about 20 thousand sums; above by the fp64 pipe.
__global__ void __launch_bounds__(32 * kSseFactors)
    calib_sse_few_kernel(const float *__restrict__ x, int64_t rows, int C, int64_t ld, int K,
                         const float *__restrict__ part, int nparts, float *__restrict__ s_out,
                         int32_t *__restrict__ zp_out, double *__restrict__ sse, uint8_t *__restrict__ alpha)
{
    __shared__ double err[kSseFactors][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float mn, mx, s0, s;
    int32_t zp;
    fold_range(part, nparts, mn, mx);
    calib_scale(mn, mx, K, s0, s, zp);
    if (s_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        *s_out = s;
        *zp_out = zp;
    }
    const int c = blockIdx.x * 32 + lane, a = blockIdx.y * kSseFactors + warp;
    if (c < C && a <= K) {
        const float up = pow2f(K - a);                 // 1 / (2^(a-K))
        const float sa = __fmul_rn(s0, pow2f(a - K));  // 2^a s, exact
        const float lo = (float)(-zp), hi = (float)(255 - zp);
        double acc = 0.0;
        for (int64_t r0 = 0; r0 < rows; r0 += 4) {  // four rows' loads and errors side by side
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = __ldg(x + min(r0 + i, rows - 1) * ld + c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float q = fminf(fmaxf(rintf(__fmul_rn(__fdiv_rn(v[i], s0), up)), lo), hi);
                const double d = (double)__fsub_rn(v[i], __fmul_rn(q, sa));
                if (r0 + i < rows) acc = __dadd_rn(acc, __dmul_rn(d, d));
            }
        }
        sse[(int64_t)c * (K + 1) + a] = acc;
        err[warp][lane] = acc;
    }
    if (alpha) {
        __syncthreads();
        if (warp == 0 && c < C) alpha[c] = least(&err[0][lane], 32, K);
    }
}

// Eq. 10 for two channels and up to four factors per block, a warp per (channel, factor): sum over rows of
// (x - clip(rint(x / (2^a s)), -zp, 255-zp) * 2^a s)^2 in fp64, ascending rows.
// x / (2^a s) is computed as (x / s0) * 2^(K-a): scaling a correctly rounded
// quotient by a power of two is the correctly rounded quotient by the scaled
// divisor (values small enough to lose bits round to 0 either way).
// The range is the fold of the partials part[nparts]; s and zp (when not null) are written by the first
// block, alpha (when not null; all factors in one block) by the block of its channels.
__global__ void __launch_bounds__(32 * CH * kSseFactors)
    calib_sse_kernel(const float *__restrict__ x, int64_t rows, int C, int64_t ld, int K,
                     const float *__restrict__ part, int nparts, float *__restrict__ s_out,
                     int32_t *__restrict__ zp_out, double *__restrict__ sse, uint8_t *__restrict__ alpha)
{
    // x and x / s0 (one division for the factors)
    __shared__ float tile[2][CH][kSseRows + 4], tdiv[2][CH][kSseRows + 4];
    __shared__ double err[CH][kSseFactors];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthreads = blockDim.x;
    float mn, mx;
    fold_range(part, nparts, mn, mx);
    float s0, s;
    int32_t zp;
    calib_scale(mn, mx, K, s0, s, zp);
    if (s_out && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
        *s_out = s;
        *zp_out = zp;
    }
    const int c0 = blockIdx.x * CH, cw = warp % CH, a = blockIdx.y * kSseFactors + warp / CH;
    const bool active = c0 + cw < C && a <= K;
    const float up = pow2f(K - a);                 // 1 / (2^(a-K))
    const float sa = __fmul_rn(s0, pow2f(a - K));  // 2^a s, exact
    const float lo = (float)(-zp), hi = (float)(255 - zp);
    // stage loads: thread -> (row, channel), CH consecutive channels of a row together, 8 values in flight
    auto load_stage = [&](int64_t r0, int buf) {
        for (int e0 = tid; e0 < kSseRows * CH; e0 += 8 * nthreads) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = e0 + i * nthreads, row = e / CH, c = c0 + e % CH;
                v[i] = e < kSseRows * CH && r0 + row < rows && c < C ? __ldg(x + (r0 + row) * ld + c) : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = e0 + i * nthreads;
                if (e < kSseRows * CH) {
                    tile[buf][e % CH][e / CH] = v[i];
                    tdiv[buf][e % CH][e / CH] = __fdiv_rn(v[i], s0);
                }
            }
        }
    };
    SeqSum sum;
    load_stage(0, 0);
    __syncthreads();
    int buf = 0;
    for (int64_t r0 = 0; r0 < rows; r0 += kSseRows, buf ^= 1) {
        if (r0 + kSseRows < rows) load_stage(r0 + kSseRows, buf ^ 1);
        if (active) {
            const int nr = (int)min((int64_t)kSseRows, rows - r0);
#pragma unroll 1
            for (int r = 0; r < nr; r += 128) {
                float d[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float xv = tile[buf][cw][r + 32 * g + lane];
                    float q = rintf(__fmul_rn(tdiv[buf][cw][r + 32 * g + lane], up));
                    q = fminf(fmaxf(q, lo), hi);
                    d[g] = __fsub_rn(xv, __fmul_rn(q, sa));
                    if (r + 32 * g + lane >= nr) d[g] = 0.0f;
                }
                if (!sum.add128(d)) {
#pragma unroll 1
                    for (int g = 0; g < 4; ++g) sum.add32(g == 0 ? d[0] : g == 1 ? d[1] : g == 2 ? d[2] : d[3]);
                }
            }
        }
        __syncthreads();
    }
    if (lane == 0 && active) {
        const double e = sum.value();
        sse[(int64_t)(c0 + cw) * (K + 1) + a] = e;
        err[cw][warp / CH] = e;
    }
    if (alpha) {
        __syncthreads();
        if (tid < CH && c0 + tid < C) alpha[c0 + tid] = least(err[tid], 1, K);
    }
}

__global__ void calib_argmin_kernel(const double *__restrict__ sse, int C, int K,
                                    uint8_t *__restrict__ alpha)
{
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    alpha[c] = least(sse + (int64_t)c * (K + 1), 1, K);
}

// Eq. 7.  x / (2^alpha s) = (x / s) * 2^-alpha by the same scaling argument.
__device__ __forceinline__ uint32_t quant_code(float x, float s, float sc, float lo, float hi, int zp)
{
    const float q = fminf(fmaxf(rintf(__fmul_rn(__fdiv_rn(x, s), sc)), lo), hi);
    return (uint32_t)((int)q + zp);
}

// V: channels per thread and step (4: 16-byte loads and 4-byte stores; the rows and C are multiples of 4)
template <int V>
__global__ void __launch_bounds__(256) quantize_kernel(const float *__restrict__ x, int64_t rows, int C, int64_t ld_x,
                                                       float s, int zp, const uint8_t *__restrict__ alpha,
                                                       uint8_t *__restrict__ xq, int64_t ld_q)
{
    extern __shared__ __align__(16) float qsh[];  // 2^-alpha_c per channel
    pdl_release();
    pdl_wait();
    for (int c = threadIdx.x; c < C; c += blockDim.x) qsh[c] = pow2f(-(int)alpha[c]);
    __syncthreads();
    const float lo = (float)(-zp), hi = (float)(255 - zp);
    // threads along the row first, the rest of the block over rows (C = 384: 96 threads a row at V = 4)
    const int cv = C / V, tr = cv < (int)blockDim.x ? cv : (int)blockDim.x, rpb = blockDim.x / tr;
    const int rl = threadIdx.x / tr, cl = threadIdx.x - rl * tr;
    if (rl >= rpb) return;
    for (int64_t r = (int64_t)blockIdx.x * rpb + rl; r < rows; r += (int64_t)gridDim.x * rpb) {
        const float *xr = x + r * ld_x;
        uint8_t *qr = xq + r * ld_q;
        for (int i = cl; i < cv; i += tr) {
            if (V == 4) {
                const float4 v = __ldg(reinterpret_cast<const float4 *>(xr) + i);
                const float4 k = reinterpret_cast<const float4 *>(qsh)[i];
                reinterpret_cast<uint32_t *>(qr)[i] =
                    quant_code(v.x, s, k.x, lo, hi, zp) | quant_code(v.y, s, k.y, lo, hi, zp) << 8 |
                    quant_code(v.z, s, k.z, lo, hi, zp) << 16 | quant_code(v.w, s, k.w, lo, hi, zp) << 24;
            } else {
                qr[i] = (uint8_t)quant_code(__ldg(xr + i), s, qsh[i], lo, hi, zp);
            }
        }
    }
}

// blocks of the min / max pass
int minmax_blocks(int64_t rows)
{
    int nparts = (int)(rows < kMaxPartials ? rows : kMaxPartials);
    int nsm = sm_count();
    if (nparts > 4 * nsm) nparts = 4 * nsm;
    return nparts < 1 ? 1 : nparts;
}

}  // namespace

size_t calibrate_workspace_bytes(int64_t rows, int C, int K, bool sums)
{
    (void)rows;
    return (size_t)kWsHeader + sizeof(float2) * kMaxPartials + (sums ? sizeof(double) * (size_t)C * (K + 1) : 0);
}

namespace {

// The error sums (and s, zp, alpha where not null) from the range partials.  A plain launch: with
// programmatic serialization the blocks start while the range kernel's still hold most SMs and stack up on
// the others (6304 x 192: 141 us against 62).
//
// The rule: a warp's sum costs about 7 us and 2 ns per sum whatever the rows (its start crosses a binade every few
// rows, and a stage holds 1024), a thread's 0.16 us a row.  us of the sums alone, warps / threads: 8 channels,
// K = 3: 32 rows 8.5 / 7.4, 48 rows 9.1 / 9.7; 1024, K = 3: 64 rows 15.2 / 12.6, 128 rows 16.2 / 22.8; 4096,
// K = 3: 32 rows 40.2 / 7.5, 256 rows 61.8 / 44.0, 512 rows 83.7 / 85.6; 8192, K = 7: 512 rows 298 / 224.
cudaError_t launch_sse(const float *x, int64_t rows, int C, int64_t ld_x, int K, const float *part, int nparts,
                       float *s, int32_t *zp, double *sse, uint8_t *alpha, cudaStream_t st)
{
    const int nf = K + 1 < kSseFactors ? K + 1 : kSseFactors, ny = (K + kSseFactors) / kSseFactors;
    uint8_t *al = ny > 1 ? nullptr : alpha;
    if (rows < 36 + (int64_t)C * (K + 1) / 64) {
        const dim3 g((unsigned)((C + 31) / 32), (unsigned)ny);
        calib_sse_few_kernel<<<g, 32 * nf, 0, st>>>(x, rows, C, ld_x, K, part, nparts, s, zp, sse, al);
    } else {
        const dim3 g((unsigned)((C + CH - 1) / CH), (unsigned)ny);
        calib_sse_kernel<<<g, 32 * CH * nf, 0, st>>>(x, rows, C, ld_x, K, part, nparts, s, zp, sse, al);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_calibrate(const float *x, int64_t rows, int C, int64_t ld_x, int K, float *s,
                             int32_t *zp, uint8_t *alpha, double *sse, void *ws, cudaStream_t st)
{
    char *w = static_cast<char *>(ws);
    float2 *part = reinterpret_cast<float2 *>(w + kWsHeader);
    double *sse_buf = sse ? sse : reinterpret_cast<double *>(w + kWsHeader + sizeof(float2) * kMaxPartials);

    const int nparts = minmax_blocks(rows);
    cudaError_t e = launch_pdl(minmax_partial_kernel, dim3(nparts), dim3(256), 0, st, x, rows, C, ld_x, part);
    if (e != cudaSuccess) return e;
    e = launch_sse(x, rows, C, ld_x, K, reinterpret_cast<const float *>(part), nparts, s, zp, sse_buf, alpha, st);
    if (e != cudaSuccess || K < kSseFactors) return e;
    calib_argmin_kernel<<<(C + 127) / 128, 128, 0, st>>>(sse_buf, C, K, alpha);
    return cudaGetLastError();
}

cudaError_t launch_calibrate_minmax(const float *x, int64_t rows, int C, int64_t ld_x, float *mnmx, void *ws,
                                    cudaStream_t st)
{
    float2 *part = reinterpret_cast<float2 *>(static_cast<char *>(ws) + kWsHeader);
    const int nparts = minmax_blocks(rows);
    cudaError_t e = launch_pdl(minmax_partial_kernel, dim3(nparts), dim3(256), 0, st, x, rows, C, ld_x, part);
    if (e != cudaSuccess) return e;
    minmax_final_kernel<<<1, 32, 0, st>>>(part, nparts, mnmx);
    return cudaGetLastError();
}

cudaError_t launch_calibrate_sse_partial(const float *x, int64_t rows, int C, int64_t ld_x, int K,
                                         const float *mnmx, double *sse, void *ws, cudaStream_t st)
{
    (void)ws;  // the given range is the one partial
    return launch_sse(x, rows, C, ld_x, K, mnmx, 1, nullptr, nullptr, sse, nullptr,
                      st);
}

cudaError_t launch_quantize(const float *x, int64_t rows, int C, int64_t ld_x, float s, int32_t zp,
                            const uint8_t *alpha, uint8_t *xq, int64_t ld_q, cudaStream_t st)
{
    const bool vec = C % 4 == 0 && ld_x % 4 == 0 && ld_q % 4 == 0 && ((uintptr_t)x % 16) == 0 && ((uintptr_t)xq % 4) == 0;
    const int cv = vec ? C / 4 : C, rpb = cv < 256 ? 256 / cv : 1;
    const int64_t want = (rows + rpb - 1) / rpb, cap = (int64_t)sm_count() * 8;
    const dim3 g((unsigned)(want < cap ? want : cap));
    const size_t smem = sizeof(float) * C;
    return vec ? launch_pdl(quantize_kernel<4>, g, dim3(256), smem, st, x, rows, C, ld_x, s, zp, alpha, xq, ld_q)
               : launch_pdl(quantize_kernel<1>, g, dim3(256), smem, st, x, rows, C, ld_x, s, zp, alpha, xq, ld_q);
}

}  // namespace fqvit
