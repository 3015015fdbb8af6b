// lis_common.cuh -- device helpers shared by the Log-Int-Softmax kernels:
// the i-exp table (supplement Algorithm 1) and the division-free log2 code
// (Algorithm 2).  See lis.cu for the derivation of the code test.
#pragma once

#include <stdint.h>

#include <cmath>

namespace fqvit {
namespace lis {

// q~ in [-1335, 0]: int8 logits plus an int8 bias minus the maximum reach -510; with a window mask
// further, but e(q~) is constant below the clamp 15 q_ln2 >= -1335 (scales >= 2^-7), so indices past
// kLutSize - 1 read the last entry
constexpr int kLutSize = 1336;

struct IexpC {
    int q_ln2, q_b, q_c;
};

// e(-t) for t in [0, 287], n = 15
__device__ __forceinline__ uint32_t iexp_neg(int t, IexpC c)
{
    int q = -t;
    int lo = 15 * c.q_ln2;
    if (q < lo) q = lo;
    int z = q / c.q_ln2;
    int qp = q - z * c.q_ln2;
    int b = qp + c.q_b;
    uint32_t qL = (uint32_t)(b * b + c.q_c);
    return qL << (15 - z);
}

// Algorithm 1 constants of a scale, fp64 with one IEEE rounding per operation as in the
// oracle's definition; computed on the host once per launch (fp64 is slow on the device).
__host__ inline IexpC iexp_consts_host(float s)
{
    const double ln2 = 0.693147180559945309417232121458176568;
    const double sd = (double)s;
    IexpC c;
    c.q_ln2 = (int)floor(-ln2 / sd);
    c.q_b = (int)floor(1.353 / sd);
    c.q_c = (int)floor(0.344 / (0.3585 * (sd * sd)));
    return c;
}

__device__ __forceinline__ void build_lut(uint32_t *lut, IexpC c)
{
    for (int t = threadIdx.x; t < kLutSize; t += blockDim.x) lut[t] = iexp_neg(t, c);
}

struct RowSum {
    float hi, lo;  // 2S = hi + lo, hi = fp32(2S)
    int hibits;
};

__device__ __forceinline__ RowSum make_rowsum(unsigned long long S)
{
    unsigned long long s2 = 2ull * S;
    RowSum r;
    r.hi = __ull2float_rn(s2);
    r.lo = (float)(long long)(s2 - __float2ull_rn(r.hi));
    r.hibits = __float_as_int(r.hi);
    return r;
}

__device__ __forceinline__ uint32_t lis_code(uint32_t e, const RowSum &rs)
{
    float ef = __uint2float_rn(e);  // exact: e = q_L 2^(15-z), q_L < 2^16
    int k = (rs.hibits - __float_as_int(ef)) >> 23;
    if (k >= 16) return 15u;
    float Dk = (k == 1) ? 3.0f : __fsub_rn(__int_as_float(((k + 127) << 23) | 0x400000), 1.0f);
    float t = __fmaf_rn(ef, Dk, -rs.hi);
    return (uint32_t)(k - 1 + (t <= rs.lo ? 1 : 0));
}

// 8-bit requantization of an attention accumulator by the dyadic multiplier n2 / 2^n1 (n1 in
// [-10, 31]; the division rounds half up), plus the zero point, clipped to 0 .. 255
__device__ __forceinline__ uint32_t requant8(int acc, int n1, int n2, int zp)
{
    const long long num = (long long)n2 * acc;
    long long R = n1 > 0 ? (num + (1LL << (n1 - 1))) >> n1 : num * (1LL << -n1);
    R += zp;
    return (uint32_t)(R < 0 ? 0 : (R > 255 ? 255 : R));
}

// The same in one fused multiply-add: c = n2 2^-n1 and zp + 1/2 are exact, the exact value rounded down to
// fp32 has the same floor, and the conversion clips.  Needs acc exact as a float, which it is up to 2^24
// in magnitude; above, c 2^24 >= 256 saturates it either way.  (An accumulator's 64-bit form takes about
// 13 instructions: with it DeiT-S attention with 8-bit output took 25.4 us a call, now 21.4; 12 x 12
// windows 69.1 and 62.4.)
struct Requant8 {
    float c, zh;
    int n1, n2, zp, fast;
};

// For the Log-Int-Softmax codes of a row of L keys: a code below 15 says e D_(code+1) > 2S, so that 2^-code <
// 1.5 e / S (D_1 = 3, D_(k+1) = 3 2^k - 1), and a code of 15 adds 1: the row's operands 2^(15 - code) sum to
// less than 1.5 2^15 + L, and |acc| <= (128 + |zp_v|) (3 2^14 + L).  That is at most 2^24 for every zp_v of an int8
// code.  (Where it was taken for zp_v = 0 only, 400 heads of 320 keys with zp_v = -5 and s_v / s_out < 1/2 took
// 53.8 us, now 37.7.)
__host__ inline Requant8 requant8_of(int n1, int n2, int zp, int zp_v, int L)
{
    Requant8 r;
    r.c = (float)ldexp((double)n2, -n1);
    r.zh = (float)zp + 0.5f;
    r.n1 = n1;
    r.n2 = n2;
    r.zp = zp;
    r.fast = (128.0 + abs(zp_v)) * (49152.0 + L) <= 16777216.0 || ldexp((double)n2, 24 - n1) >= 256.0;
    return r;
}

__device__ __forceinline__ uint32_t requant8_fast(int acc, const Requant8 &r)
{
    uint32_t y;
    asm("cvt.rmi.sat.u8.f32 %0, %1;" : "=r"(y) : "f"(__fmaf_rd(__int2float_rn(acc), r.c, r.zh)));
    return y;
}

// four accumulators to a word of four bytes (r.fast is uniform over the launch)
__device__ __forceinline__ uint32_t requant8x4(int a0, int a1, int a2, int a3, const Requant8 &r)
{
    if (r.fast)
        return __byte_perm(__byte_perm(requant8_fast(a0, r), requant8_fast(a1, r), 0x0040),
                           __byte_perm(requant8_fast(a2, r), requant8_fast(a3, r), 0x0040), 0x5410);
    return requant8(a0, r.n1, r.n2, r.zp) | requant8(a1, r.n1, r.n2, r.zp) << 8 |
           requant8(a2, r.n1, r.n2, r.zp) << 16 | requant8(a3, r.n1, r.n2, r.zp) << 24;
}

__device__ __forceinline__ int relpos_idx(int i, int j, int w)
{
    int yi = i / w, xi = i - yi * w, yj = j / w, xj = j - yj * w;
    return (yi - yj + w - 1) * (2 * w - 1) + (xi - xj + w - 1);
}

}  // namespace lis
}  // namespace fqvit
