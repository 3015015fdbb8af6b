// linear_tc.cu -- the MinMax Linear layers of the fully quantized block on the
// 5th-generation tensor cores (tcgen05) of sm_103a.  Sec. 3 quantizes Linear
// layers with uniform MinMax; Sec. 4.1 makes the weights symmetric and
// channel-wise and the activations asymmetric and layer-wise:
//   acc[m][n] = sum_k (x[m][k] - zp_x) w[n][k] + b[n]
//   y[m][n]   = clip(floor((N2_n acc + 2^(N1_n - 1)) / 2^N1_n) + zp_y, 0, 255)
// with N1_n, N2_n the dyadic form of M_n = s_x s_w[n] / s_y (the output stage of
// the supplement's LayerNorm; N1_n <= 0 is a product by N2_n 2^min(-N1_n, 10)).
//
// Exactness.  x - zp_x (in -255 .. 255) and w (in -128 .. 127) are exact in
// fp16, every product is exact in fp32, and a sum of such integers is exact in
// fp32 while its partial sums stay within 2^24.  The reduction runs in equal
// chunks of at most kc steps of 64 with 64 kc max(zp_x, 255 - zp_x) 128 <= 2^24
// (kc = 16, 1024 products, at zp_x = 128; 8 at the ends of the range), so no
// partial sum in any order leaves that bound; the tests run sums at it, unit
// products among them.  Each chunk is accumulated afresh in tensor
// memory and, when a row has several, added as an integer by the epilogue.
//
// One launch per call.  The weights are fp16 [N][K] (fqvit_linear_pack_weight,
// once per layer) and reach shared memory by TMA tensor loads (128-byte
// swizzle); so do the activations, as bytes.  Two teams of four converter
// warps subtract the zero point in fp16 and store the A operand into tensor
// memory (4 stages of 64 reduction steps), from where the MMAs read it: an
// operand written to and read from shared memory took 80 KB of its bandwidth
// per 256-wide step against 48 KB (640 and 384 cycles, a step's MMAs 512).
// Before, one launch made an fp16 copy of X in memory and one the weight sums
// of its shift by 128.
//
// Tiles (TileCfg): pairs of CTAs on 256 x 192 outputs (cta_group::2, M = 256: each
// CTA holds its 128 rows of X and half of the weight rows), two accumulators
// of 192 columns and the operand stages filling tensor memory; or single CTAs
// on 128 x 128 or 128 x 64 where the larger tiles would leave SMs idle
// (launch_linear).  Row tiles come fastest, so a CTA's tiles lie in few columns.
//
// Roles (27 warps): warps 0-15 are the epilogue (warp w reads tensor-memory
// lanes 32 (w % 4) .. and columns BN/4 (w / 4) .. of a tile), warps 16-23 the
// converters; one lane each of warps 24 and 26 issues the loads of W and of X,
// and one of warp 25 (of the pair's first CTA) the MMAs.  The MMAs of the next
// chunk run while the epilogue reads the last.  The output bytes leave through
// 32-row staging areas by tensor stores (16-byte stores at the rows' stride
// cost fc1 of ViT-L/384 20 us of 129).
//
// Measured (us per call, back to back in a graph; the earlier form -> this one), M =
// 18464: QKV (3072 x 1024) 118.2 -> 74.7, projection (1024 x 1024) 46.8 -> 31.5, fc1
// (4096 x 1024) 148.0 -> 98.4 (1574 TFLOP/s), fc2 (1024 x 4096) 174.7 -> 97.7 (1585);
// M = 1576: 2304 x 768 17.1 -> 9.9, 768 x 3072 29.1 -> 16.2; M = 197: 192 x 192
// 8.8 -> 4.2.  (Up to 7 % more on some GPUs.)  A step of the large ones takes 518
// cycles, its MMAs 384.  Timed without the conversion 492, so that accounts for 26 of
// the difference; what takes the other 108 is not known.
//
// Requantization.  Where every channel of the CTA allows it (see channel_entry)
// y is one fused multiply-add rounded down and a saturating conversion:
// floor(RD(acc c + zp_y + 1/2)) with c = N2 2^-N1 exact; rounding down cannot
// cross an integer, so the floor is that of the exact value.  Else 64-bit
// integers, element by element.
//
// Every wait is bounded: after two seconds the kernel records a timeout
// status, drains the copies and MMAs it issued and returns.
#include "fqvit_internal.cuh"
#include "tc_common.cuh"

#include <cstring>
#include <type_traits>
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

namespace fqvit {

namespace {

using namespace tc;

constexpr int LM = 128;                   // output rows per CTA and tile (tensor-memory lanes)
constexpr int LK = 64;                    // reduction per step: one 128-byte swizzle row of fp16
constexpr int LEPI_WARPS = 16;            // epilogue: 4 warps per lane quarter
constexpr int LTEAMS = 2;                 // converter teams, each on every second step
constexpr int LCONV_WARPS = 4 * LTEAMS;   // a team: one warp per lane quarter
constexpr int LTMA_WARP = LEPI_WARPS + LCONV_WARPS;
constexpr int LMMA_WARP = LTMA_WARP + 1;
constexpr int LXTMA_WARP = LMMA_WARP + 1;
constexpr int LTHREADS = 32 * (LXTMA_WARP + 1);  // 27 warps, seven on a scheduler: 72 registers each
constexpr int LRAW_BYTES = LM * LK;       // X of a step as bytes, 8 KB
constexpr int LAS = 4;                    // operand stages in tensor memory
constexpr int LACOLS = LK / 2;            // tensor-memory columns of one: 64 fp16 per lane
constexpr int LTAB_TILES = 3;             // column tiles of the channel table
constexpr int LMAXN = 4096;               // channels of a layer

// CG CTAs on a tile of 128 CG x BN outputs.  Two rings of K-steps in shared memory, filled by TMA as far
// ahead as the space allows: PF stages of X as bytes (8 KB) and of weights (BN / CG rows).  (Pairs on
// 256 x 128 took 121 us for fc2 of ViT-L/384, on 256 x 192 94.)
template <int CG_, int BN_, int PF_>
struct TileCfg {
    static constexpr int CG = CG_, BN = BN_, PF = PF_;
    static constexpr int B_ROWS = BN / CG;
    static constexpr int B_BYTES = B_ROWS * LK * 2;       // (multiples of 1024: the swizzle's alignment)
    static constexpr int OFF_RAW = PF * B_BYTES;
    static constexpr int OFF_TAB = OFF_RAW + PF * LRAW_BYTES;
    static constexpr int COLS = BN / 4;                   // columns per epilogue warp
    static constexpr int OFF_OUT = (OFF_TAB + LTAB_TILES * BN * 8 + 1023) / 1024 * 1024;
    static constexpr int SMEM = 1024 + OFF_OUT + LM * BN;  // the output bytes on their way out
    static constexpr int TM_A = 2 * BN;                   // two accumulators, then the operand stages
    static constexpr int TMEM = TM_A + LAS * LACOLS <= 256 ? 256 : 512;
    static_assert(TM_A + LAS * LACOLS <= 512 && SMEM + 1024 <= 232448 && B_BYTES % 1024 == 0, "tile does not fit");
};
using PairTile = TileCfg<2, 192, 8>;
using MidTile = TileCfg<1, 128, 7>;
using SmallTile = TileCfg<1, 64, 10>;

struct LinParams {
    const uint8_t *x;
    int64_t M, ld_x;
    int N, K;
    int ksteps;    // ceil(K / 64)
    int kc;        // steps per exact chunk
    int zp_x, zp_y;
    int vec16;     // rows of x are 16-byte aligned
    float s_x, s_y;
    const float *s_w;
    const int32_t *bias;
    uint8_t *y;
    int64_t ld_y;
    int32_t *acc;
    int64_t ld_acc;
    int mtiles, ntiles;
};

template <class T>
struct LinShared {
    uint64_t wfull[T::PF], wempty[T::PF], rfull[T::PF], rempty[T::PF], afull[LAS], aempty[LAS];
    uint64_t cfull[2], cempty[2], fin;
    uint32_t tmem;
    int abort_flag;
    int wide;  // some channel needs the 64-bit requantization
};

// ---- cluster-scope barrier operations of a CTA pair (plain ones for a single CTA)
__device__ __forceinline__ uint32_t cta_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// arrives on the barrier at this shared-memory offset in the pair's first CTA
template <int CG>
__device__ __forceinline__ void arrive_leader(uint64_t *b)
{
    if (CG == 1) {
        mbar_arrive(b);
    } else {
        asm volatile(
            "{ .reg .b32 ra; mapa.shared::cluster.u32 ra, %0, 0;\n\t"
            "mbarrier.arrive.shared::cluster.b64 _, [ra]; }" ::"r"(sa(b))
            : "memory");
    }
}

template <int CG>
__device__ __forceinline__ void tma_load(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    if (CG == 1)
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
            "[%4];" ::"r"(sa(dst)),
            "l"(map), "r"(x), "r"(y), "r"(sa(bar))
            : "memory");
    else  // completes on the first CTA's barrier (bit 24 of a cluster address is the rank within the pair)
        asm volatile(
            "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
            "[%1, {%2, %3}], [%4];" ::"r"(sa(dst)),
            "l"(map), "r"(x), "r"(y), "r"(sa(bar) & 0xFEFFFFFFu)
            : "memory");
}

// 32 lanes of a warp x 32 columns into tensor memory
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    __syncwarp();
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
        "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// D (+)= A B, A in tensor memory (of both CTAs of a pair), B in shared memory
template <int CG>
__device__ __forceinline__ void mma_ts(uint32_t dt, uint32_t at, uint64_t bd, uint32_t idesc, bool accumulate)
{
    if (CG == 1)
        mma_f16_ta(dt, at, bd, accumulate, idesc);
    else
        asm volatile(
            "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p; }" ::"r"(
                dt),
            "r"(at), "l"(bd), "r"(idesc), "r"((uint32_t)accumulate)
            : "memory");
}

// arrives on the barrier (in both CTAs of a pair) when the MMAs issued so far have completed
template <int CG>
__device__ __forceinline__ void commit(uint64_t *b)
{
    if (CG == 1)
        mma_commit(b);
    else
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                sa(b)),
            "h"((uint16_t)3)
            : "memory");
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Per output channel: the multiplier and the shift of the requantization (mult < 2^18 in
// bits 0..17, shift 0..31 in bits 24..28) and the bias.  N1 <= 0 folds 2^min(-N1, 10) into
// the multiplier with shift 0.  The fp32 operations are single IEEE round-to-nearest ones,
// as on the host.  wide: the channel needs the 64-bit form.  The fp32 form takes acc as a
// float, exact below 2^24 in magnitude; a larger one must saturate: c 2^24 >= 2^9 (c = mult
// 2^-shift, zp_y + 1/2 < 2^8), and the bias itself must be exact.
__device__ __forceinline__ int2 channel_constants(const LinParams &p, int n, bool &bad, bool &wide)
{
    const float sw = p.s_w[n];
    const float Mn = __fdiv_rn(__fmul_rn(p.s_x, sw), p.s_y);
    int mult = 0, shift = 0;
    if (sw > 0.0f && Mn > 0.0f && Mn < 1.0e30f) {
        int n1 = 7 - ilogbf(Mn);
        if (n1 > 31) n1 = 31;
        const int n2 = (int)floorf(ldexpf(Mn, n1));
        if (n1 >= 0) {
            mult = n2;
            shift = n1;
        } else {
            mult = n2 << min(-n1, 10);
        }
    } else {
        bad = true;
    }
    const int b = p.bias ? p.bias[n] : 0;
    wide |= ((unsigned long long)(uint32_t)mult << 24) < (512ull << shift) || b < -(1 << 24) || b > (1 << 24);
    return make_int2(mult | (shift << 24), b);
}

// y code of one accumulator (the bias added): (mult acc + 2^(shift-1)) >> shift, + zp_y, clipped
// (out of line: the rare wide channels; it keeps the registers of the fp32 loop)
__device__ __noinline__ uint32_t y_code(int acc, int2 ch, int zp_y)
{
    const int mult = ch.x & 0xFFFFFF, shift = ch.x >> 24;
    const long long num = (long long)mult * acc + (long long)((1u << shift) >> 1);
    const long long R = (num >> shift) + zp_y;
    return (uint32_t)(R < 0 ? 0 : R > 255 ? 255 : R);
}

// two fp32 sums; two fused multiply-adds rounded down
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma2_rm(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long pack2(uint32_t lo, uint32_t hi)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}
// floor of both halves saturated to 0 .. 255, as bytes 0 and 1
__device__ __forceinline__ uint32_t floor_u8x2(unsigned long long y)
{
    uint32_t a, b;
    asm("{ .reg .f32 lo, hi; mov.b64 {lo, hi}, %2; cvt.rmi.sat.u8.f32 %0, lo; cvt.rmi.sat.u8.f32 %1, hi; }"
        : "=r"(a), "=r"(b)
        : "l"(y));
    return __byte_perm(a, b, 0x0040);
}

// Sixteen bytes to sixteen fp16 values minus a zero point (exact): byte b becomes the fp16
// 1024 + b (exponent of 1024, b in the mantissa), then z = 1024 + zp is subtracted.
__device__ __forceinline__ void bytes_to_h16(const uint4 &w, __half2 z, uint32_t *h)
{
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[2 * i] = __byte_perm(ww[i], 0x64u, 0x4140);
        h[2 * i + 1] = __byte_perm(ww[i], 0x64u, 0x4342);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        __half2 t = __hsub2(*reinterpret_cast<const __half2 *>(&h[i]), z);
        h[i] = *reinterpret_cast<const uint32_t *>(&t);
    }
}

// 16 bytes of a row of x from column k on; columns at or past K read as 0 (the weights are 0 there).
// Rows that are not multiples of 16 bytes (every contiguous x with K = 8 mod 16) come this way: 18464 x 4096
// x 1016 124 us (98 at K = 1024; the earlier form with its copy of x 196), 8200 x 1536 x 1000 28.0 (45.2).
__device__ __forceinline__ uint4 load_x16(const uint8_t *row, int k, int K)
{
    uint2 a = make_uint2(0, 0), b = make_uint2(0, 0);  // K and the stride are multiples of 8
    if (k + 8 <= K) a = __ldg(reinterpret_cast<const uint2 *>(row + k));
    if (k + 16 <= K) b = __ldg(reinterpret_cast<const uint2 *>(row + k + 8));
    return make_uint4(a.x, a.y, b.x, b.y);
}

template <class T, bool ACC>
__global__ void __launch_bounds__(LTHREADS, 1)
    linear_tc_kernel(const __grid_constant__ LinParams p, const __grid_constant__ CUtensorMap tmw,
                     const __grid_constant__ CUtensorMap tmx, const __grid_constant__ CUtensorMap tmy)
{
    constexpr int CG = T::CG, BN = T::BN, COLS = T::COLS, PF = T::PF;
    extern __shared__ unsigned char dsm_raw[];
    __shared__ LinShared<T> sh;
    unsigned char *base = dsm_raw + ((1024u - (sa(dsm_raw) & 1023u)) & 1023u);
    unsigned char *RAW = base + T::OFF_RAW;
    // channel table of this CTA's column tiles (from its first, nt0, on), two channels per 16 bytes:
    // {c0, c1, b0, b1} (fp32 form; b as an integer when a row has several chunks) or {m0, b0, m1, b1}
    // (wide form: packed multiplier and shift, integer bias)
    uint4 *CH = reinterpret_cast<uint4 *>(base + T::OFF_TAB);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t rank = CG == 2 ? cta_rank() : 0u;
    volatile int *abort_flag = &sh.abort_flag;
    pdl_release();
    if (tid == 0) {
        for (int s = 0; s < PF; ++s) {
            mbar_init(&sh.wfull[s], 1);
            mbar_init(&sh.wempty[s], 1);
            mbar_init(&sh.rfull[s], 1);
            mbar_init(&sh.rempty[s], 4);
        }
        for (int s = 0; s < LAS; ++s) {
            mbar_init(&sh.afull[s], CG * 4);
            mbar_init(&sh.aempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sh.cfull[b], 1);
            mbar_init(&sh.cempty[b], CG * LEPI_WARPS);
        }
        mbar_init(&sh.fin, 1);
        sh.abort_flag = 0;
        sh.wide = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        if (CG == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&sh.tmem)),
                         "r"(T::TMEM));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&sh.tmem)),
                         "r"(T::TMEM));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
        }
    }
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync();  // the other CTA's barriers are initialized
    tc_fence_after();
    const uint32_t tmem = sh.tmem;

    const int grp = (int)blockIdx.x / CG, ngrp = (int)gridDim.x / CG;
    const int64_t ntiles = (int64_t)p.mtiles * p.ntiles;
    const int t_begin = (int)((int64_t)grp * ntiles / ngrp);
    const int t_end = (int)((int64_t)(grp + 1) * ntiles / ngrp);
    const int nt0 = t_begin / p.mtiles, mt0 = t_begin - nt0 * p.mtiles;  // row tiles fastest
    pdl_wait();  // the set-up above touched no global memory

    if (warp >= LEPI_WARPS) {
        if (warp < LTMA_WARP) {
            // ---- converters: thread r turns the 64 bytes of row r of a step into 64 fp16 in lane r of an
            //      operand stage.  (The bytes' 16-byte unit u of row r is at u ^ (r / 2 % 4): no bank
            //      conflicts.)
            const int r = (tid - 32 * LEPI_WARPS) & 127, team = (warp - LEPI_WARPS) >> 2;
            const __half2 z = __half2half2(__int2half_rn(1024 + p.zp_x));
            const bool vec16 = p.vec16 != 0;
            const uint32_t ta = tmem + T::TM_A + ((uint32_t)(32 * (warp & 3)) << 16);
            const unsigned char *raw = RAW + r * LK;
            const uint32_t sw = (r >> 1) & 3;
            const int steps = (t_end - t_begin) * p.ksteps;
            int lmt = mt0, ks = team;  // rows without 16-byte alignment come straight from global memory
            uint32_t st = team, ph = 1, rs = team, rph = 0;  // the first pass over the stages waits for nothing
            for (int s = team; s < steps; s += LTEAMS) {
                uint4 v[4];
                bool ok = true;
                if (vec16) {
                    ok = mbar_wait_warp(&sh.rfull[rs], rph, abort_flag);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        v[j] = *reinterpret_cast<const uint4 *>(raw + rs * LRAW_BYTES + ((j ^ sw) << 4));
                } else {  // rows past the end: any bytes (their outputs are not stored)
                    while (ks >= p.ksteps) {
                        ks -= p.ksteps;
                        if (++lmt == p.mtiles) lmt = 0;
                    }
                    const int64_t row = ((int64_t)lmt * CG + rank) * LM + r;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        v[j] = load_x16(p.x + (row < p.M ? row : p.M - 1) * p.ld_x, ks * LK + 16 * j, p.K);
                    ks += LTEAMS;
                }
                if (!ok || !mbar_wait_warp(&sh.aempty[st], ph, abort_flag)) break;
                tc_fence_after();
                uint32_t o[32];
#pragma unroll
                for (int j = 0; j < 4; ++j) bytes_to_h16(v[j], z, o + 8 * j);
                tmem_st32(ta + st * LACOLS, o);
                if (lane == 0) mbar_arrive(&sh.rempty[rs]);  // (every lane's bytes are in registers)
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) arrive_leader<CG>(&sh.afull[st]);
                if ((st += LTEAMS) >= LAS) st -= LAS, ph ^= 1;
                if ((rs += LTEAMS) >= PF) rs -= PF, rph ^= 1;
            }
        } else if (warp == LXTMA_WARP) {
            // ---- TMA producer of the bytes of X
            if (p.vec16 && elect_one()) {
                uint32_t rs = 0, rph = 1;
                int mt = mt0, issued = 0;
                bool ok = true;
                for (int t = t_begin; t < t_end && ok; ++t) {
                    for (int ks = 0; ks < p.ksteps; ++ks) {
                        ok = mbar_wait(&sh.rempty[rs], rph, abort_flag);
                        if (!ok) break;
                        mbar_expect_tx(&sh.rfull[rs], LRAW_BYTES);
                        tma_load<1>(RAW + rs * LRAW_BYTES, &tmx, ks * LK, (mt * CG + (int)rank) * LM, &sh.rfull[rs]);
                        ++issued;
                        if (++rs == PF) rs = 0, rph ^= 1;
                    }
                    if (++mt == p.mtiles) mt = 0;
                }
                // the last loads may still be in flight if the consumers stopped early
                for (int j = issued > PF ? issued - PF : 0; j < issued; ++j)
                    mbar_wait(&sh.rfull[j % PF], (uint32_t)(j / PF) & 1, abort_flag, false);
            }
            __syncwarp();
        } else if (warp == LTMA_WARP) {
            // ---- TMA producer of the weights
            if (elect_one()) {
                uint32_t st = 0, ph = 1, issued = 0;
                int mt = mt0, nt = nt0;
                bool ok = true;
                for (int t = t_begin; t < t_end && ok; ++t) {
                    for (int ks = 0; ks < p.ksteps; ++ks) {
                        ok = mbar_wait(&sh.wempty[st], ph, abort_flag);
                        if (!ok) break;
                        if (rank == 0) mbar_expect_tx(&sh.wfull[st], CG * T::B_BYTES);
                        tma_load<CG>(base + st * T::B_BYTES, &tmw, ks * LK, nt * BN + (int)rank * T::B_ROWS,
                                     &sh.wfull[st]);
                        ++issued;
                        if (++st == PF) st = 0, ph ^= 1;
                    }
                    if (++mt == p.mtiles) mt = 0, ++nt;
                }
                if (rank == 0)  // the same; the first CTA's barriers count the bytes of both
                    for (uint32_t j = issued > PF ? issued - PF : 0; j < issued; ++j)
                        mbar_wait(&sh.wfull[j % PF], (j / PF) & 1, abort_flag, false);
                // The first CTA's commits arrive on the barriers of both.  The cluster barrier at the end orders
                // threads, not these arrivals: each CTA sees its own last ones here, so that none can land in
                // shared memory that already belongs to the next CTA of this SM.  (The epilogue waits for every
                // cfull.  Not while the loop runs: a wait has two seconds.)
                if (CG == 2) {
                    for (uint32_t j = issued > PF ? issued - PF : 0; j < issued && ok; ++j)
                        ok = mbar_wait(&sh.wempty[j % PF], (j / PF) & 1, abort_flag);
                    for (uint32_t j = issued > LAS ? issued - LAS : 0; j < issued && ok; ++j)
                        ok = mbar_wait(&sh.aempty[j % LAS], (j / LAS) & 1, abort_flag);
                    mbar_wait(&sh.fin, 0, abort_flag, false);
                }
            }
            __syncwarp();
        } else if (warp == LMMA_WARP && rank == 0) {
            // ---- MMA issuer: chunk gc accumulates in tensor-memory buffer gc % 2
            if (elect_one()) {
                constexpr uint32_t idesc =
                    (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)((LM * CG) >> 4) << 24);
                uint32_t st = 0, ph = 0, ws = 0, wph = 0, gc = 0, commits = 0;
                bool ok = true;
                for (int t = t_begin; t < t_end && ok; ++t) {
                    for (int c0 = 0; c0 < p.ksteps && ok; c0 += p.kc, ++gc) {
                        const uint32_t b = gc & 1;
                        if (gc >= 2 && !mbar_wait(&sh.cempty[b], ((gc >> 1) - 1) & 1, abort_flag)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const int c1 = min(p.ksteps, c0 + p.kc);
                        for (int ks = c0; ks < c1; ++ks) {
                            if (!mbar_wait(&sh.wfull[ws], wph, abort_flag) ||
                                !mbar_wait(&sh.afull[st], ph, abort_flag)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const uint32_t a0 = tmem + T::TM_A + st * LACOLS, b0 = sa(base) + ws * T::B_BYTES;
#pragma unroll
                            for (int s = 0; s < LK / 16; ++s)
                                mma_ts<CG>(tmem + b * BN, a0 + 8 * s, smem_desc(b0 + 32 * s, 16, 1024), idesc,
                                           ks > c0 || s > 0);
                            commit<CG>(&sh.aempty[st]);  // the stages are free once these MMAs completed
                            commit<CG>(&sh.wempty[ws]);
                            ++commits;
                            if (++st == LAS) st = 0, ph ^= 1;
                            if (++ws == PF) ws = 0, wph ^= 1;
                        }
                        if (!ok) break;
                        commit<CG>(&sh.cfull[b]);
                        ++commits;
                    }
                }
                if (commits > 0) {  // every MMA issued has completed before tensor memory is released
                    commit<CG>(&sh.fin);
                    mbar_wait(&sh.fin, 0, abort_flag, false);
                }
            }
            __syncwarp();
        }
    } else {
        const int nch = (p.ksteps + p.kc - 1) / p.kc;
        // ---- the constants of the channels this CTA's tiles cover (each thread a pair of channels)
        {
            bool bad = false, wide = false;
            const int pairs = ((t_end - 1) / p.mtiles - nt0 + 1) * (BN / 2);  // at most LTAB_TILES column tiles
            for (int pass = 0; pass < 2; ++pass) {
                for (int i = tid; i < pairs; i += 32 * LEPI_WARPS) {
                    const int n = nt0 * BN + 2 * i;
                    if (n >= p.N) continue;
                    if (pass == 0) {
                        const int2 a = channel_constants(p, n, bad, wide), b = channel_constants(p, n + 1, bad, wide);
                        CH[i] = make_uint4((uint32_t)a.x, (uint32_t)a.y, (uint32_t)b.x, (uint32_t)b.y);
                    } else if (!sh.wide) {  // to the fp32 form (the thread's own entries)
                        const uint4 e = CH[i];
                        auto scale = [](uint32_t m) {  // mult 2^-shift, exact
                            return __float_as_uint(__uint2float_rn(m & 0xFFFFFFu) *
                                                   __int_as_float((127 - (int)(m >> 24)) << 23));
                        };
                        const bool fb = nch == 1;
                        CH[i] = make_uint4(scale(e.x), scale(e.z),
                                                fb ? __float_as_uint(__int2float_rn((int)e.y)) : e.y,
                                                fb ? __float_as_uint(__int2float_rn((int)e.w)) : e.w);
                    }
                }
                if (pass == 0) {
                    if (bad) atomicExch(&g_status, 1);
                    if (wide) atomicExch(&sh.wide, 1);
                }
                __syncwarp();
                asm volatile("bar.sync 1, %0;" ::"n"(32 * LEPI_WARPS) : "memory");
            }
        }
        const bool wide = sh.wide != 0;
        // ---- epilogue: warp w, lanes 32 (w % 4) .. (tile rows), columns COLS (w / 4) ..
        const int q = warp & 3, h = warp >> 2;
        const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(COLS * h);
        const unsigned long long zh = pack2(__float_as_uint((float)p.zp_y + 0.5f), __float_as_uint((float)p.zp_y + 0.5f));
        unsigned char *out_st = base + T::OFF_OUT + warp * 32 * COLS;
        unsigned char *out_row = out_st + lane * COLS;
        const uint32_t out_sw = COLS == 32 ? (lane >> 2) & 1 : 0;
        uint32_t gc = 0;
        bool ok = true;
        int mt = mt0, nt = nt0;
        for (int t = t_begin; t < t_end && ok; ++t) {
            const int64_t row = ((int64_t)mt * CG + rank) * LM + 32 * q + lane;
            const int col0 = nt * BN + COLS * h;
            const int tcol = (nt - nt0) * BN + COLS * h;  // the first column's place in the table
            if (++mt == p.mtiles) mt = 0, ++nt;
            const bool row_ok = row < p.M;
            // the tile's bytes leave through this warp's 32 x COLS staging bytes (16-byte unit u of a row at
            // u ^ the swizzle of the tensor store: no bank conflicts); the previous tile's store has read them
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
            int32_t *arow = ACC ? p.acc + (row_ok ? row : 0) * p.ld_acc + col0 : nullptr;
            // 16 columns from g on (v: their sums as fp32 (one chunk) or integers): y and acc
            auto emit = [&](const uint32_t *v, int g, auto ints_tag) {
                constexpr bool INTS = decltype(ints_tag)::value;
                const uint4 *ch = CH + ((tcol + g) >> 1);
                uint32_t w[4];
                int a[16];
                if (!wide) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t hw[2];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int i = 4 * k + 2 * u;
                            const uint4 c = ch[i >> 1];
                            unsigned long long av;
                            if (INTS) {
                                const int i0 = (int)v[i] + (int)c.z, i1 = (int)v[i + 1] + (int)c.w;
                                if (ACC) a[i] = i0, a[i + 1] = i1;
                                av = pack2(__float_as_uint(__int2float_rn(i0)), __float_as_uint(__int2float_rn(i1)));
                            } else {
                                av = add2(pack2(v[i], v[i + 1]), pack2(c.z, c.w));
                                if (ACC) {
                                    a[i] = __float2int_rn(__uint_as_float(v[i])) + __float2int_rn(__uint_as_float(c.z));
                                    a[i + 1] =
                                        __float2int_rn(__uint_as_float(v[i + 1])) + __float2int_rn(__uint_as_float(c.w));
                                }
                            }
                            hw[u] = floor_u8x2(fma2_rm(av, pack2(c.x, c.y), zh));
                        }
                        w[k] = __byte_perm(hw[0], hw[1], 0x5410);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        w[k] = 0;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int i = 4 * k + u;
                            const uint4 c = ch[i >> 1];
                            const int2 e = (u & 1) ? make_int2((int)c.z, (int)c.w) : make_int2((int)c.x, (int)c.y);
                            a[i] = (INTS ? (int)v[i] : __float2int_rn(__uint_as_float(v[i]))) + e.y;
                            w[k] |= y_code(a[i], e, p.zp_y) << (8 * u);
                        }
                    }
                }
                *reinterpret_cast<uint4 *>(out_row + (((g >> 4) ^ out_sw) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                if (ACC && row_ok) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        reinterpret_cast<int4 *>(arow + g)[i] =
                            make_int4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
                }
            };
            if (nch == 1) {
                const uint32_t b = gc & 1;
                ok = mbar_wait_warp(&sh.cfull[b], (gc >> 1) & 1, abort_flag);
                ++gc;
                if (!ok) break;
                tc_fence_after();
                constexpr int LD = COLS % 32 == 0 ? 32 : 16;  // columns per load
#pragma unroll
                for (int j = 0; j < COLS / LD; ++j) {
                    uint32_t v[LD];
                    if constexpr (LD == 32)
                        tmem_ld32(tl + b * BN + LD * j, v);
                    else
                        tmem_ld16(tl + b * BN + LD * j, v);
                    tmem_wait_ld();
                    if (j == COLS / LD - 1) {  // read: the buffer may be rewritten
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) arrive_leader<CG>(&sh.cempty[b]);
                    }
#pragma unroll
                    for (int g = 0; g < LD; g += 16)
                        if (col0 + LD * j + g < p.N) emit(v + g, LD * j + g, std::false_type{});  // N % 16 == 0
                }
            } else {
                uint32_t sum[COLS];
#pragma unroll
                for (int i = 0; i < COLS; ++i) sum[i] = 0u;
                for (int c = 0; c < nch; ++c, ++gc) {
                    const uint32_t b = gc & 1;
                    ok = mbar_wait_warp(&sh.cfull[b], (gc >> 1) & 1, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int j = 0; j < COLS / 8; ++j) {
                        uint32_t v[8];
                        tmem_ld8(tl + b * BN + 8 * j, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) sum[8 * j + i] += (uint32_t)__float2int_rn(__uint_as_float(v[i]));
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_leader<CG>(&sh.cempty[b]);
                }
                if (!ok) break;
#pragma unroll
                for (int g = 0; g < COLS; g += 16)
                    if (col0 + g < p.N) emit(sum + g, g, std::true_type{});
            }
            fence_async_smem();  // the staging bytes are read by the tensor store
            __syncwarp();
            if (lane == 0) {
                const int row0 = (int)(row - lane);
                if (row0 < p.M && col0 < p.N)  // rows past M and columns past N are clipped
                    asm volatile(
                        "cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(&tmy),
                        "r"(col0), "r"(row0), "r"(sa(out_st))
                        : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
    }
    if (warp < LEPI_WARPS && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");  // stores completed
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync();  // both CTAs have seen the pair's last MMAs and arrivals
    tc_fence_after();
    if (warp == 0) {
        if (CG == 1)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T::TMEM));
        else
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T::TMEM));
    }
}

// Eight bytes to eight fp16 values minus a zero point z (exact): byte b becomes the fp16
// 1024 + b (exponent of 1024, b in the mantissa), then 1024 + zp is subtracted.  Signed codes
// arrive with their sign bit flipped (b = w + 128) and zp = 128.
__device__ __forceinline__ uint4 bytes_to_h8(uint2 w, __half2 z)
{
    uint32_t h[4] = {__byte_perm(w.x, 0x64u, 0x4140), __byte_perm(w.x, 0x64u, 0x4342),
                     __byte_perm(w.y, 0x64u, 0x4140), __byte_perm(w.y, 0x64u, 0x4342)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __half2 t = __hsub2(*reinterpret_cast<const __half2 *>(&h[i]), z);
        h[i] = *reinterpret_cast<const uint32_t *>(&t);
    }
    return make_uint4(h[0], h[1], h[2], h[3]);
}

// src [rows][ld] bytes (K a multiple of 8) -> dst [rows][K] fp16 of (byte ^ flip) - zp
__global__ void __launch_bounds__(256) bytes_to_half_kernel(const uint8_t *src, int64_t rows, int K, int64_t ld,
                                                            uint32_t flip, int zp, uint16_t *dst)
{
    pdl_release();
    pdl_wait();
    const int kv = K >> 3;
    const int64_t items = rows * kv;
    const __half2 z = __half2half2(__int2half_rn(1024 + zp));
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < items; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = x / kv;
        const int c = (int)(x - r * kv);
        uint2 w = __ldg(reinterpret_cast<const uint2 *>(src + r * ld + 8 * c));
        w.x ^= flip;
        w.y ^= flip;
        *reinterpret_cast<uint4 *>(dst + r * K + 8 * c) = bytes_to_h8(w, z);
    }
}

// A row-major [rows][cols] array of fp16 or bytes with row stride ld elements as a 2-d tensor for the TMA
// loads and stores: boxes of box_cols x box_rows, zeros outside.  False when the driver's encoder is
// unavailable or rejects the shape.
bool tensor_map(CUtensorMap *tm, const void *ptr, bool half, int64_t rows, int cols, int64_t ld, int box_cols,
                int box_rows, CUtensorMapSwizzle swizzle)
{
    const auto encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(tensor_map_encoder());
    if (!encode) return false;
    memset(tm, 0, sizeof(*tm));
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * (half ? 2 : 1)};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(tm, half ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                  const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <class T, bool ACC>
cudaError_t linear_launch_as(const LinParams &p, const CUtensorMap &tw, const CUtensorMap &tx,
                             const CUtensorMap &ty, int grid, cudaStream_t st)
{
    const size_t smem = T::SMEM;
    static SmemReady ready;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(LTHREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = T::CG;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = T::CG > 1 ? 2 : 1;
    return launch_prepared((const void *)linear_tc_kernel<T, ACC>, smem, ready,
                           [&] { return cudaLaunchKernelEx(&cfg, linear_tc_kernel<T, ACC>, p, tw, tx, ty); });
}

template <class T>
cudaError_t linear_launch(LinParams &p, const uint16_t *w_h, cudaStream_t st)
{
    CUtensorMap tw, tx, ty;
    memset(&tx, 0, sizeof(tx));
    constexpr CUtensorMapSwizzle out_sw = T::COLS == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE;
    if (!tensor_map(&tw, w_h, true, p.N, p.K, p.K, LK, T::B_ROWS, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !tensor_map(&ty, p.y, false, p.M, p.N, p.ld_y, T::COLS, 32, out_sw) ||
        (p.vec16 && !tensor_map(&tx, p.x, false, p.M, p.K, p.ld_x, LK, LM, CU_TENSOR_MAP_SWIZZLE_64B)))
        return cudaErrorInvalidValue;
    p.mtiles = (int)((p.M + LM * T::CG - 1) / (LM * T::CG));
    p.ntiles = (p.N + T::BN - 1) / T::BN;
    const int64_t tiles = (int64_t)p.mtiles * p.ntiles;
    const int64_t groups = sm_count() / T::CG;
    const int grid = (int)(tiles < groups ? tiles : groups) * T::CG;
    return p.acc ? linear_launch_as<T, true>(p, tw, tx, ty, grid, st)
                 : linear_launch_as<T, false>(p, tw, tx, ty, grid, st);
}

// Modelled cycles of a tile shape: the waves of its tiles over the SMs, each K-steps x cycles per step,
// plus a fixed part (pipeline fill, epilogue of the last tile).  The choice by these figures was the
// fastest, or within 2 % of it, on 24 shapes (M 41 .. 18464, N 80 .. 4096, K 192 .. 4096), e.g. us of
// pair / mid / small: 18464 x 1024 x 1024 30.8 / 37.4 / 63.8, 1576 x 768 x 768 7.3 / 6.2 / 8.7,
// 197 x 192 x 768 6.9 / 5.7 / 5.3.
template <class T>
double tile_cost(int64_t M, int N, int ksteps, double step, double fixed)
{
    const int64_t tiles = ((M + LM * T::CG - 1) / (LM * T::CG)) * ((N + T::BN - 1) / T::BN);
    const int64_t groups = sm_count() / T::CG;
    return (double)((tiles + groups - 1) / groups) * ksteps * step + fixed;
}

cudaError_t launch_bytes_to_half(const uint8_t *src, int64_t rows, int K, int64_t ld, uint32_t flip, int zp,
                                 uint16_t *dst, cudaStream_t st)
{
    const int64_t items = rows * (K / 8);
    int64_t blocks = (items + 255) / 256;
    const int64_t cap = (int64_t)sm_count() * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return launch_pdl(bytes_to_half_kernel, dim3((unsigned)blocks), dim3(256), 0, st, src, rows, K, ld, flip, zp,
                      dst);
}

// The bounded wait on a barrier that nothing completes: one thread of one CTA waits on phase 0
// of a fresh mbarrier of count 1, with the same two-second wait the kernels use; it gives up,
// records the timeout status and returns (the failure path, without a fault).
__global__ void bounded_wait_probe_kernel()
{
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) (void)mbar_wait(&bar, 0, &abort_flag);
}

}  // namespace

cudaError_t launch_bounded_wait_probe(cudaStream_t st)
{
    bounded_wait_probe_kernel<<<1, 32, 0, st>>>();
    return cudaGetLastError();
}

bool linear_supported(const LinearArgs &a) { return a.N <= LMAXN; }

cudaError_t launch_linear_pack_weight(const int8_t *w, int N, int K, int64_t ld_w, uint16_t *w_h, cudaStream_t st)
{
    return launch_bytes_to_half(reinterpret_cast<const uint8_t *>(w), N, K, ld_w, 0x80808080u, 128, w_h, st);
}

size_t linear_workspace_bytes(int64_t M, int K)
{
    return ((size_t)M * (size_t)K * 2 + 255) / 256 * 256 + (size_t)LMAXN * sizeof(int32_t);
}

cudaError_t launch_linear(const LinearArgs &a, cudaStream_t st)
{
    LinParams p{};
    p.x = a.x;
    p.ld_x = a.ld_x;
    // An output that overlaps the activations (a layer run in place): the tiles read x while others
    // write, so they read a copy in the workspace.
    auto overlaps = [&](const void *o, size_t bytes) {
        const uintptr_t x0 = (uintptr_t)a.x, x1 = x0 + (size_t)(a.M - 1) * a.ld_x + a.K, o0 = (uintptr_t)o;
        return o && o0 < x1 && x0 < o0 + bytes;
    };
    if (overlaps(a.y, (size_t)(a.M - 1) * a.ld_y + a.N) ||
        overlaps(a.acc, ((size_t)(a.M - 1) * a.ld_acc + a.N) * sizeof(int32_t))) {
        cudaError_t e = cudaMemcpy2DAsync(a.xh, a.K, a.x, a.ld_x, a.K, a.M, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return e;
        p.x = reinterpret_cast<const uint8_t *>(a.xh);
        p.ld_x = a.K;
    }
    p.M = a.M;
    p.N = a.N;
    p.K = a.K;
    p.ksteps = (a.K + LK - 1) / LK;
    const int xmax = a.zp_x > 255 - a.zp_x ? a.zp_x : 255 - a.zp_x;
    p.kc = (1 << 24) / (LK * 128 * xmax);
    p.kc = (p.ksteps + (p.ksteps + p.kc - 1) / p.kc - 1) / ((p.ksteps + p.kc - 1) / p.kc);  // equal chunks
    p.zp_x = a.zp_x;
    p.zp_y = a.zp_y;
    p.vec16 = p.ld_x % 16 == 0 && ((uintptr_t)p.x % 16) == 0;
    p.s_x = a.s_x;
    p.s_y = a.s_y;
    p.s_w = a.s_w;
    p.bias = a.bias;
    p.y = a.y;
    p.ld_y = a.ld_y;
    p.acc = a.acc;
    p.ld_acc = a.ld_acc;
    const double pair = tile_cost<PairTile>(a.M, a.N, p.ksteps, 400.0, 3000.0);
    const double mid = tile_cost<MidTile>(a.M, a.N, p.ksteps, 400.0, 2500.0);
    const double small = tile_cost<SmallTile>(a.M, a.N, p.ksteps, 260.0, 2000.0);
    if (small <= mid && small <= pair) return linear_launch<SmallTile>(p, a.w_h, st);
    if (mid <= pair) return linear_launch<MidTile>(p, a.w_h, st);
    return linear_launch<PairTile>(p, a.w_h, st);
}

cudaError_t read_clear_linear_status(int *status)
{
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(status, g_status, sizeof(int));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_status, &zero, sizeof(int));
}

}  // namespace fqvit
