// lis_gen.cu -- fused Log-Int-Softmax + BitShift attention times values on the
// tcgen05 tensor cores for the rows that the other two tensor-core kernels do
// not take: rows of 25 to 1024 keys with head dimension 32 or 64 (lis_tc.cu
// holds at most 592 keys and d = 64), and windows of up to 256 keys with a
// relative-position bias and a shifted-window mask (lis_win.cu: 64 keys).
// These ran on CUDA cores before (lis.cu), a multiply-add per key and value; shorter
// rows still do (GMIN_L).
//
// The product is the one of lis_tc.cu: acc = P V - zp_V (P 1) with
// P[i][j] = 2^(15 - code_ij), exact in fp16 with fp32 accumulation.  Nothing of
// a row's length has to be resident but its logits: the operands P pass
// through a ring of four 64-key blocks in tensor memory and V through a ring of
// three in shared memory, so a tile of 128 rows needs 128 ld bytes of logits, the
// i-exp table and 24 KB.
//
// Tiles: 128 rows.  From 128 keys on they are consecutive rows of all BH L, so a
// tile may end one head and begin the next: each block then multiplies two
// heads' V into two accumulators.  Shorter rows: one head per tile.
//
// Roles (22 warps):
//   warps 0-15, four threads per row (warp 4 q + r / 32, lane r % 32; part q takes keys
//     64 kb + 16 q .. of every 64-key block, or 4 keys of a last block of at most
//     16): row maximum, i-exp row sum, then each key's code (code_ops,
//     tc_common.cuh), the operands straight into tensor memory.  Only the
//     four warps of 32 rows meet (two named barriers per tile), so the four
//     groups drift apart and one's lookups overlap another's reductions.
//     Without a bias the logits are read again from shared memory in each of
//     the three passes (one 16-byte load per 16 keys) and a distance is one
//     byte; with a bias the sums q + bias - mask stay in registers as pairs of
//     16-bit lanes (as in lis_win.cu, up to 256 keys).
//   warps 16-19: V of a block as the fp16 B operand, and the accumulators out.
//   warp 20, one elected lane: the MMAs.  Warp 21, one elected lane: the copies
//     of the logits tiles.
//
// i-exp table: as in lis_win.cu (one 256-byte line per distance: 32 copies of
// e, then 32 of fp32 e).  Distances past 15 |q_ln2| all give the clamp's value.
//
// Measured (us per call): 8 x 12 heads of 785 keys, d = 64, 1129 on CUDA cores -> 62.5
// (59 M logits; 12 us of bytes); 12 x 12 windows, bias and mask, d = 32, 8-bit output,
// 1536 heads of 144 keys, 440 -> 56.4 (32 M logits; 7 us of bytes).  Issue-bound:
// about 22 warp instructions per 32 keys in all (V, read-out and waits among them) at 58 % of
// the issue slots.  Tried without a gain: distances held in registers (62.4 and 58.3 us), seven
// operand blocks and up to twelve V blocks in flight, V requested a block ahead.
//
// Every wait is bounded (two seconds); a role whose wait gave up records it and
// runs its loop to the end without waiting further, so every barrier is met.
#include "fqvit_internal.cuh"
#include "lis_common.cuh"
#include "tc_common.cuh"

namespace fqvit {

namespace {

using namespace lis;
using namespace tc;

constexpr int GM = 128;                 // rows per tile
constexpr int GSOFT_WARPS = 16;
constexpr int GV_WARP = GSOFT_WARPS;    // warps 16-19
constexpr int GMMA_WARP = GV_WARP + 4;
constexpr int GCOPY_WARP = GMMA_WARP + 1;
constexpr int GTHREADS = 32 * (GCOPY_WARP + 1);
constexpr int GPS = 4;                  // operand blocks in tensor memory (32 columns each)
constexpr int GVS = 3;                  // V blocks in shared memory (64 keys x 128 bytes)
constexpr uint32_t GV_BYTES = 64 * 128;
// Rows below this many keys stay on CUDA cores: a head is a tile, whose fixed cost (its barriers, the read-out of 128
// accumulator rows) does not shrink with the row.  us per call, CUDA cores / this kernel, d = 64, 3000 heads: 4 keys 15.0
// / 40.6, 16 keys 32.8 / 41.0, 24 keys 50.3 / 44.1, 32 keys 75.7 / 43.3; 3072 windows with a bias: 16 keys 45.7 / 53.8, 25
// keys 77.9 / 56.9; d = 32, 700 heads: 24 keys 11.9 / 12.7, 26 keys 14.0 / 12.8.
constexpr int GMIN_L = 25;
constexpr uint32_t kSmemOptin = 232448;
// tensor memory: accumulators [tile parity][head of the tile] of 64 columns, operands, row sums [parity]
constexpr uint32_t G_TA = 256, G_TR = G_TA + 32 * GPS, G_TMEM = 512;
// control area
constexpr uint32_t GC_ONES = 512, GC_RMAX = 1024, GC_RSUM = GC_RMAX + 4 * GM * 4, GC_END = GC_RSUM + 4 * GM * 8;

struct GenParams {
    const int8_t *logits;
    int64_t ld;
    const int8_t *v;
    int64_t ld_v;
    int32_t *acc;
    int64_t ld_acc;
    int64_t BH;
    int L;
    int zp;
    IexpC ic;
    int ne;       // table entries
    int small_e;  // every i-exp value below 2^28
    int pack;     // tiles packed across heads
    int nlg;      // logits buffers (1 or 2)
    const int8_t *bias;
    int heads, window;
    const uint8_t *region;
    int n_windows;
    int mask_c;  // |mask value| clamped to 1024 (exact: lis_win.cu)
    uint8_t *out8;
    int64_t ld_out8;
    Requant8 rq;
    uint32_t off_c, off_v, off_lg, off_b, off_r;  // shared-memory offsets: control, V ring, logits, bias, regions
};

struct GenShared {
    uint64_t lload[2], lfree[2], pfull[GPS], pfree[GPS], vfull[GVS], vfree[GVS], dfull[2], dfree[2], fin;
    uint32_t tmem;
    int abort_flag;
};
static_assert(sizeof(GenShared) <= GC_ONES, "control area");

struct GTile {
    int64_t g0;              // first row of all BH * L
    int rows, h0, nsplit;    // the first nsplit rows belong to head h0, the rest to h0 + 1
};

__device__ __forceinline__ GTile gen_tile(const GenParams &p, int64_t t, int tpb)
{
    GTile ti;
    if (p.pack) {
        ti.g0 = t * GM;
        ti.rows = (int)min((int64_t)GM, p.BH * p.L - ti.g0);
        ti.h0 = (int)(ti.g0 / p.L);
        ti.nsplit = (int)min((int64_t)ti.rows, (int64_t)(ti.h0 + 1) * p.L - ti.g0);
    } else {
        ti.h0 = (int)(t / tpb);
        const int r0 = (int)(t - (int64_t)ti.h0 * tpb) * GM;
        ti.g0 = (int64_t)ti.h0 * p.L + r0;
        ti.rows = min(GM, p.L - r0);
        ti.nsplit = ti.rows;
    }
    return ti;
}

// the tile after ti (a step of GM <= L rows crosses at most one head boundary)
__device__ __forceinline__ GTile gen_next(const GenParams &p, GTile ti)
{
    if (p.pack) {
        ti.g0 += GM;
        if (ti.g0 >= (int64_t)(ti.h0 + 1) * p.L) ++ti.h0;
        ti.rows = (int)min((int64_t)GM, p.BH * p.L - ti.g0);
        ti.nsplit = (int)min((int64_t)ti.rows, (int64_t)(ti.h0 + 1) * p.L - ti.g0);
    } else {
        int r0 = (int)(ti.g0 - (int64_t)ti.h0 * p.L) + GM;
        if (r0 >= p.L) {
            ++ti.h0;
            r0 = 0;
        }
        ti.g0 = (int64_t)ti.h0 * p.L + r0;
        ti.rows = min(GM, p.L - r0);
        ti.nsplit = ti.rows;
    }
    return ti;
}

__device__ __forceinline__ uint32_t ldu32(const unsigned char *p) { return *reinterpret_cast<const uint32_t *>(p); }
__device__ __forceinline__ float ldf32(const unsigned char *p) { return *reinterpret_cast<const float *>(p); }

// table line offset 256 d | off of distance byte J of a word, or of 16-bit half J of a pair word
template <int J>
__device__ __forceinline__ uint32_t line_b(uint32_t w, uint32_t off)
{
    return prmt(w, off, 0x7704u | (J << 4));  // bytes: off[0], w[J], 0, 0 (off < 256)
}
template <int J>
__device__ __forceinline__ uint32_t line_h(uint32_t w, uint32_t off)
{
    return prmt(w, off, J == 0 ? 0x7104u : 0x7324u);  // off[0], half's low byte, its high byte, 0
}

// NKB: 64-key blocks of a biased row (1 .. 4), 0 without a bias (any length, logits re-read)
template <int NKB, bool MASK, int D>
__global__ void __launch_bounds__(GTHREADS, 1) lis_attn_gen_kernel(const __grid_constant__ GenParams p)
{
    constexpr bool BIAS = NKB > 0;
    extern __shared__ __align__(1024) unsigned char dsm[];  // the i-exp table first: lookups add no base
    GenShared &sh = *reinterpret_cast<GenShared *>(dsm + p.off_c);
    unsigned char *ONES = dsm + p.off_c + GC_ONES;
    int *red_max = reinterpret_cast<int *>(dsm + p.off_c + GC_RMAX);
    unsigned long long *red_sum = reinterpret_cast<unsigned long long *>(dsm + p.off_c + GC_RSUM);
    unsigned char *VS = dsm + p.off_v;
    unsigned char *LG = dsm + p.off_lg;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    volatile int *abort_flag = &sh.abort_flag;
    const int L = p.L, Lp = (L + 15) & ~15;
    const int nkb = (L + 63) >> 6, nsteps = (L + 15) >> 4;
    const int nb = 2 * p.window - 1, nb2 = nb * nb;
    int *koff = reinterpret_cast<int *>(dsm + p.off_b);        // [64 NKB]
    int *qbase = koff + 64 * NKB;                              // [64 NKB]
    unsigned char *BT = reinterpret_cast<unsigned char *>(qbase + 64 * NKB);  // [heads][nb2], bias + 128
    unsigned char *RG = dsm + p.off_r;                         // [n_windows][Lp]
    unsigned char *RU = RG + p.n_windows * Lp;                 // [n_windows]: more than one region
    pdl_release();
    if ((sa(dsm) & 1023u) != 0) {  // the swizzled V blocks: reported (FQVIT_ERR_UNSUPPORTED) instead of run
        if (tid == 0) atomicCAS(&g_status, 0, 2);
        return;
    }
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sh.lload[b], 1);
            mbar_init(&sh.lfree[b], GSOFT_WARPS);
            mbar_init(&sh.dfull[b], 1);
            mbar_init(&sh.dfree[b], 4);
        }
        for (int s = 0; s < GPS; ++s) {
            mbar_init(&sh.pfull[s], GSOFT_WARPS);
            mbar_init(&sh.pfree[s], 1);
        }
        for (int s = 0; s < GVS; ++s) {
            mbar_init(&sh.vfull[s], 4);
            mbar_init(&sh.vfree[s], 1);
        }
        mbar_init(&sh.fin, 1);
        sh.abort_flag = 0;
    }
    if (warp == GMMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(&sh.tmem)),
                     "r"(G_TMEM));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // the i-exp table: 16-byte pieces, 8 of e then 8 of fp32 e per line
    for (int d = tid >> 2; d < p.ne; d += GTHREADS / 4) {
        const uint32_t e = iexp_neg(d, p.ic);
        const uint32_t w = (tid & 2) ? __float_as_uint(__uint2float_rn(e)) : e;
        uint4 *line = reinterpret_cast<uint4 *>(dsm + d * 256) + 4 * (tid & 3);
#pragma unroll
        for (int k = 0; k < 4; ++k) line[k] = make_uint4(w, w, w, w);
    }
    for (int i = tid; i < 128; i += GTHREADS) reinterpret_cast<uint32_t *>(ONES)[i] = 0x3C003C00u;
    if (D == 32)  // columns 32 .. 63 of the V blocks: fp16 1 in column 32 (its accumulator is P 1), zeros
        for (int x = tid; x < GVS * 64 * 4; x += GTHREADS) {
            const int key = x >> 2, u = 4 + (x & 3);
            *reinterpret_cast<uint4 *>(VS + key * 128 + ((u ^ (key & 7)) << 4)) =
                make_uint4(u == 4 ? 0x3C00u : 0u, 0, 0, 0);
        }
    if (BIAS) {
        for (int j = tid; j < 64 * NKB; j += GTHREADS) {
            const int jj = j < L ? j : 0, y = jj / p.window, x = jj - y * p.window;
            koff[j] = y * nb + x;
            qbase[j] = (y + p.window - 1) * nb + x + p.window - 1;
        }
    }
    pdl_wait();  // the set-up above touched no global memory
    if (BIAS)
        for (int x = tid; x < p.heads * nb2; x += GTHREADS) BT[x] = (unsigned char)((int)p.bias[x] + 128);
    if (MASK)
        for (int x = tid; x < p.n_windows * Lp; x += GTHREADS) {
            const int w = x / Lp, j = x - w * Lp;
            RG[x] = j < L ? p.region[(size_t)w * L + j] : 0;
        }
    if (MASK)
        for (int w = tid; w < p.n_windows; w += GTHREADS) {
            const uint8_t *rp = p.region + (size_t)w * L;
            int many = 0;
            for (int j = 1; j < L; ++j) many |= rp[j] ^ rp[0];
            RU[w] = many ? 1 : 0;
        }
    fence_async_smem();  // ONES and the V blocks are read by the MMAs
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem;

    const int tpb = (L + GM - 1) / GM;
    const int64_t ntiles = p.pack ? (p.BH * L + GM - 1) / GM : p.BH * tpb;
    const int64_t t_begin = (int64_t)blockIdx.x * ntiles / gridDim.x;
    const int n = (int)((int64_t)(blockIdx.x + 1) * ntiles / gridDim.x - t_begin);
    GTile ti = gen_tile(p, t_begin, tpb);

    if (warp < GSOFT_WARPS) {
        const int k4 = warp & 3, q = warp >> 2, r = 32 * k4 + lane;
        const uint32_t off = 4u * (uint32_t)lane;
        const uint32_t tA = tmem + G_TA + ((uint32_t)(32 * k4) << 16);
        const uint32_t cap2 = (uint32_t)(p.ne - 1) * 0x10001u;
        const float e0 = ldf32(dsm + 128);
        // the last block holds R = 1 .. 64 keys; with R <= 16 each part takes 4 of them (see above)
        const int R = L - (nkb - 1) * 64;
        const bool quarter = R <= 16;
        const int last_keys = quarter ? min(4, max(0, R - 4 * q)) : min(16, max(0, R - 16 * q));
        const int last_words = quarter ? 1 : 4;
        const int npad = last_keys > 0 ? 4 * last_words - last_keys : 0;
        const int last_off = (nkb - 1) * 64 + (quarter ? 4 * q : 16 * q);
        // byte masks of the last slice's words: keys below L
        auto keep = [&](int b) -> uint32_t {
            const int k = last_keys - 4 * b;
            return k >= 4 ? 0xFFFFFFFFu : k <= 0 ? 0u : (0xFFFFFFFFu >> (32 - 8 * k));
        };
        // four operand words of 16 keys; keys of the last slice at or past L are zero
        auto mask_ops = [&](uint32_t (&o)[8]) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (2 * c >= last_keys)
                    o[c] = 0;
                else if (2 * c + 1 == last_keys)
                    o[c] &= 0xFFFFu;
            }
        };
        auto group_bar = [&]() {  // the 128 threads of these 32 rows
            __syncwarp();
            asm volatile("bar.sync %0, 128;" ::"r"(1 + k4) : "memory");
        };
        uint32_t ps = 0, pph = 1;  // operand ring (the first pass over it waits for nothing)
        for (int it = 0; it < n; ++it, ti = gen_next(p, ti)) {
            const int lb = p.nlg == 2 ? it & 1 : 0;
            const uint32_t lph = (uint32_t)(p.nlg == 2 ? it >> 1 : it) & 1u;
            const unsigned char *lr = LG + (size_t)lb * GM * p.ld + (size_t)r * p.ld;
            mbar_wait_warp(&sh.lload[lb], lph, abort_flag);
            uint32_t vp[BIAS ? 8 * NKB : 1];  // pairs (4j, 4j + 2), (4j + 1, 4j + 3) of words j, four words per block
            int m;
            uint32_t mrep = 0;
            // 16 bytes of keys from key k0 on, the last slice's padding replaced by the byte pad
            auto last_word = [&](int b, uint32_t pad) -> uint32_t {
                if (b >= last_words || 4 * b >= last_keys) return pad;
                return (ldu32(lr + last_off + 4 * b) & keep(b)) | (pad & ~keep(b));
            };
            if constexpr (BIAS) {
                const int64_t g = min(ti.g0 + r, p.BH * L - 1);
                const int bh = r < ti.nsplit || ti.nsplit == ti.rows ? ti.h0 : ti.h0 + 1;
                const int i = min((int)(g - (int64_t)bh * L), L - 1);
                const unsigned char *bt = BT + (bh % p.heads) * nb2 + qbase[i];
                const int wdx = MASK ? (bh / p.heads) % p.n_windows : 0;
                const unsigned char *rg = RG + wdx * Lp;
                const bool masked = MASK && __any_sync(0xffffffffu, RU[wdx] != 0);  // some row's window has regions
                const uint32_t rib = MASK ? (uint32_t)rg[i] * 0x01010101u : 0u;
                uint32_t mx = 0;
                auto word = [&](uint32_t w, int key, uint32_t rw, uint32_t &pe, uint32_t &po) {
                    const uint32_t u = w ^ 0x80808080u;
                    const int4 ko = *reinterpret_cast<const int4 *>(koff + key);
                    const uint32_t b0 = bt[-ko.x], b1 = bt[-ko.y], b2 = bt[-ko.z], b3 = bt[-ko.w];
                    pe = prmt(u, 0u, 0x4240u) + (b0 | (b2 << 16));
                    po = prmt(u, 0u, 0x4341u) + (b1 | (b3 << 16));
                    if (MASK) {
                        pe += 0x04000400u;
                        po += 0x04000400u;
                        if (masked) {
                            const uint32_t x = rw ^ rib;  // byte nonzero: the key's region differs
                            const uint32_t me = ((prmt(x, 0u, 0x4240u) + 0x7FFF7FFFu) >> 15) & 0x00010001u;
                            const uint32_t mo = ((prmt(x, 0u, 0x4341u) + 0x7FFF7FFFu) >> 15) & 0x00010001u;
                            pe -= me * (uint32_t)p.mask_c;
                            po -= mo * (uint32_t)p.mask_c;
                        }
                    }
                };
#pragma unroll
                for (int kb = 0; kb < NKB - 1; ++kb) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(lr + 64 * kb + 16 * q);
                    const uint4 rr =
                        MASK ? *reinterpret_cast<const uint4 *>(rg + 64 * kb + 16 * q) : make_uint4(0, 0, 0, 0);
                    const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, rw[4] = {rr.x, rr.y, rr.z, rr.w};
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        word(xw[b], 64 * kb + 16 * q + 4 * b, rw[b], vp[8 * kb + 2 * b], vp[8 * kb + 2 * b + 1]);
                        mx = vmax16x2u(mx, vmax16x2u(vp[8 * kb + 2 * b], vp[8 * kb + 2 * b + 1]));
                    }
                }
#pragma unroll
                for (int b = 0; b < 4; ++b) {  // the last slice: lanes of keys at or past L are 0
                    uint32_t pe = 0, po = 0;
                    if (b < last_words && 4 * b < last_keys) {
                        word(ldu32(lr + last_off + 4 * b), last_off + 4 * b,
                             MASK ? ldu32(rg + last_off + 4 * b) : 0u, pe, po);
                        const uint32_t kp = keep(b);  // byte masks to 16-bit lane masks (sign replication)
                        pe &= prmt(kp, 0u, 0xA280u);
                        po &= prmt(kp, 0u, 0xB391u);
                    }
                    vp[8 * (NKB - 1) + 2 * b] = pe;
                    vp[8 * (NKB - 1) + 2 * b + 1] = po;
                    mx = vmax16x2u(mx, vmax16x2u(pe, po));
                }
                m = (int)max(mx & 0xFFFFu, mx >> 16);
            } else {
                // odd bytes as the high bytes of signed 16-bit lanes, even bytes biased in unsigned lanes
                uint32_t mo = 0x80008000u, me = 0u;
                auto upd = [&](uint32_t w) {
                    mo = vmax16x2(mo, w);
                    me = vmax16x2u(me, (w ^ 0x00800080u) & 0x00FF00FFu);
                };
                for (int kb = 0; kb < nkb - 1; ++kb) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(lr + 64 * kb + 16 * q);
                    upd(x.x), upd(x.y), upd(x.z), upd(x.w);
                }
#pragma unroll
                for (int b = 0; b < 4; ++b) upd(last_word(b, 0x80808080u));
                m = max(max(sbyte<1>(mo), sbyte<3>(mo)), max((int)(me & 0xFFFFu), (int)(me >> 16)) - 128);
            }
            red_max[q * GM + r] = m;
            group_bar();
            m = max(max(red_max[r], red_max[GM + r]), max(red_max[2 * GM + r], red_max[3 * GM + r]));
            // ---- i-exp row sum
            unsigned long long S = 0;
            auto add4 = [&](uint32_t e0, uint32_t e1, uint32_t e2, uint32_t e3) {
                if (p.small_e)
                    S += (e0 + e1) + (e2 + e3);
                else
                    S += (unsigned long long)(e0 + e1) + (unsigned long long)(e2 + e3);  // e < 2^31
            };
            if constexpr (BIAS) {
                const uint32_t m2 = (uint32_t)m * 0x10001u;
#pragma unroll
                for (int k = 0; k < 8 * NKB; ++k) vp[k] = vmin16x2u(m2 - vp[k], cap2);  // distances
#pragma unroll
                for (int j = 0; j < 4 * NKB; ++j) {
                    if (j < 4 * (NKB - 1) || ((j & 3) < last_words && 4 * (j & 3) < last_keys))
                        add4(ldu32(dsm + line_h<0>(vp[2 * j], off)), ldu32(dsm + line_h<1>(vp[2 * j], off)),
                             ldu32(dsm + line_h<0>(vp[2 * j + 1], off)), ldu32(dsm + line_h<1>(vp[2 * j + 1], off)));
                }
                // the padding lanes of words that hold keys (v = 0: distance m, clamped)
                const int pads = last_keys > 0 ? ((last_keys + 3) & ~3) - last_keys : 0;
                S -= (unsigned long long)pads * ldu32(dsm + ((uint32_t)min(m, p.ne - 1) << 8) + off);
            } else {
                mrep = (uint32_t)(m + 128) * 0x01010101u;
                auto sum4 = [&](uint32_t w) {
                    const uint32_t d = mrep - (w ^ 0x80808080u);
                    add4(ldu32(dsm + line_b<0>(d, off)), ldu32(dsm + line_b<1>(d, off)), ldu32(dsm + line_b<2>(d, off)),
                         ldu32(dsm + line_b<3>(d, off)));
                };
                for (int kb = 0; kb < nkb - 1; ++kb) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(lr + 64 * kb + 16 * q);
                    sum4(x.x), sum4(x.y), sum4(x.z), sum4(x.w);
                }
                if (last_keys > 0) {
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if (b < last_words) sum4(last_word(b, 0x80808080u));
                    S -= (unsigned long long)npad * ldu32(dsm + ((uint32_t)(m + 128) << 8) + off);
                }
            }
            red_sum[q * GM + r] = S;
            group_bar();
            S = red_sum[r] + red_sum[GM + r] + red_sum[2 * GM + r] + red_sum[3 * GM + r];
            const CodeRow rs = code_row(S, e0);
            const bool any_fix = __any_sync(0xffffffffu, rs.fix != 0);
            // ---- operands, block after block, into the ring
            auto ops4 = [&](uint32_t w, uint32_t &o0, uint32_t &o1) {  // a word of four distance bytes
                o0 = code_ops(ldf32(dsm + 128 + line_b<0>(w, off)), ldf32(dsm + 128 + line_b<1>(w, off)), rs);
                o1 = code_ops(ldf32(dsm + 128 + line_b<2>(w, off)), ldf32(dsm + 128 + line_b<3>(w, off)), rs);
                if (any_fix) {  // the key at distance 0, where 3 e > 2S
                    const uint32_t z = (~(((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) >> 7) & 0x01010101u;
                    o0 += prmt(z, 0u, 0x4140u) * rs.fix;
                    o1 += prmt(z, 0u, 0x4342u) * rs.fix;
                }
            };
            auto ops4h = [&](uint32_t pe, uint32_t po, uint32_t &o0, uint32_t &o1) {  // two pairs of 16-bit distances
                o0 = code_ops(ldf32(dsm + 128 + line_h<0>(pe, off)), ldf32(dsm + 128 + line_h<0>(po, off)), rs);
                o1 = code_ops(ldf32(dsm + 128 + line_h<1>(pe, off)), ldf32(dsm + 128 + line_h<1>(po, off)), rs);
                if (any_fix) {
                    const uint32_t ze = 0x00010001u - vmin16x2u(pe, 0x00010001u);
                    const uint32_t zo = 0x00010001u - vmin16x2u(po, 0x00010001u);
                    o0 += prmt(ze, zo, 0x5410u) * rs.fix;
                    o1 += prmt(ze, zo, 0x7632u) * rs.fix;
                }
            };
            auto block_out = [&](bool last, uint32_t (&o)[8]) {
                mbar_wait_warp(&sh.pfree[ps], pph, abort_flag);  // the MMAs of the slot's previous block are done
                tc_fence_after();
                if (!last) {
                    tmem_st8(tA + 32 * ps + 8 * q, o);
                } else {
                    mask_ops(o);
                    if (quarter)
                        tmem_st2(tA + 32 * ps + 2 * q, o[0], o[1]);
                    else if (16 * q < ((R + 15) & ~15))  // a 16-key step that the MMAs read
                        tmem_st8(tA + 32 * ps + 8 * q, o);
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.pfull[ps]);
                if (++ps == GPS) ps = 0, pph ^= 1;
            };
            if constexpr (BIAS) {
                if (lane == 0) mbar_arrive(&sh.lfree[lb]);  // (after group_bar: every lane's logits are in registers)
#pragma unroll
                for (int kb = 0; kb < NKB; ++kb) {
                    uint32_t o[8];
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        if (kb < NKB - 1 || b < last_words)
                            ops4h(vp[8 * kb + 2 * b], vp[8 * kb + 2 * b + 1], o[2 * b], o[2 * b + 1]);
                        else
                            o[2 * b] = o[2 * b + 1] = 0;
                    }
                    block_out(kb == NKB - 1, o);
                }
            } else {
                for (int kb = 0; kb < nkb - 1; ++kb) {
                    const uint4 x = *reinterpret_cast<const uint4 *>(lr + 64 * kb + 16 * q);
                    uint32_t o[8];
                    ops4(mrep - (x.x ^ 0x80808080u), o[0], o[1]);
                    ops4(mrep - (x.y ^ 0x80808080u), o[2], o[3]);
                    ops4(mrep - (x.z ^ 0x80808080u), o[4], o[5]);
                    ops4(mrep - (x.w ^ 0x80808080u), o[6], o[7]);
                    block_out(false, o);
                }
                uint32_t o[8];
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    if (b < last_words)
                        ops4(mrep - (last_word(b, 0x80808080u) ^ 0x80808080u), o[2 * b], o[2 * b + 1]);
                    else
                        o[2 * b] = o[2 * b + 1] = 0;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.lfree[lb]);  // the logits tile may be refilled
                block_out(true, o);
            }
        }
    } else if (warp < GMMA_WARP) {
        // ---------------- V blocks and read-out
        const int eq = warp & 3, vt = tid - 32 * GV_WARP, key = vt >> 1, half = vt & 1;
        const uint32_t etl = tmem + ((uint32_t)(32 * eq) << 16);
        uint32_t vs = 0, vph = 1;
        auto read_out = [&](const GTile &t, int par, uint32_t ph) {
            mbar_wait_warp(&sh.dfull[par], ph, abort_flag);
            tc_fence_after();
            const int i = 32 * eq + lane;
            const bool split = t.nsplit < t.rows;
            const bool any2 = split && t.nsplit < 32 * eq + 32, use2 = split && i >= t.nsplit;
            const bool row_ok = i < t.rows;
            const uint32_t d0 = etl + 128 * par;
            int zsum = 0;
            if (p.zp != 0) {
                uint32_t x;
                if (D == 32) {
                    tmem_ld1(d0 + 32, x);
                    if (any2) {
                        uint32_t y;
                        tmem_ld1(d0 + 64 + 32, y);
                        tmem_wait_ld();
                        x = use2 ? y : x;
                    }
                } else {
                    tmem_ld1(etl + G_TR + 16 * par, x);
                }
                tmem_wait_ld();
                zsum = p.zp * __float2int_rn(__uint_as_float(x));
            }
            const int64_t row = t.g0 + i;
#pragma unroll
            for (int c = 0; c < D / 16; ++c) {
                uint32_t a[16];
                tmem_ld16(d0 + 16 * c, a);
                tmem_wait_ld();
                if (any2) {
                    uint32_t b[16];
                    tmem_ld16(d0 + 64 + 16 * c, b);
                    tmem_wait_ld();
                    if (use2) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) a[k] = b[k];
                    }
                }
                if (!row_ok) continue;
                if (p.out8) {
                    uint32_t w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        int q[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) q[u] = __float2int_rn(__uint_as_float(a[4 * k + u])) - zsum;
                        w[k] = requant8x4(q[0], q[1], q[2], q[3], p.rq);
                    }
                    *reinterpret_cast<uint4 *>(p.out8 + row * p.ld_out8 + 16 * c) = make_uint4(w[0], w[1], w[2], w[3]);
                } else {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        int v8[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) v8[u] = __float2int_rn(__uint_as_float(a[8 * k + u])) - zsum;
                        stg256(p.acc + row * p.ld_acc + 16 * c + 8 * k, v8);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.dfree[par]);
        };
        GTile prev{};
        for (int it = 0; it < n; ++it, ti = gen_next(p, ti)) {
            if (it > 0) read_out(prev, (it - 1) & 1, (uint32_t)((it - 1) >> 1) & 1u);
            const int nh = ti.nsplit < ti.rows ? 2 : 1;
            for (int kb = 0; kb < nkb; ++kb) {
                for (int hh = 0; hh < nh; ++hh) {
                    const int j = 64 * kb + key;
                    const int8_t *src = p.v + ((size_t)(ti.h0 + hh) * L + j) * p.ld_v + half * (D / 2);
                    uint4 x[D / 32];
#pragma unroll
                    for (int c = 0; c < D / 32; ++c)
                        x[c] = j < L ? __ldg(reinterpret_cast<const uint4 *>(src) + c) : make_uint4(0, 0, 0, 0);
                    mbar_wait_warp(&sh.vfree[vs], vph, abort_flag);
                    unsigned char *row = VS + vs * GV_BYTES + key * 128;
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint4 lo = make_uint4(0, 0, 0, 0), hi = lo;
                        if (j < L) {
                            const uint32_t x0 = x[c].x ^ 0x80808080u, x1 = x[c].y ^ 0x80808080u;
                            const uint32_t x2 = x[c].z ^ 0x80808080u, x3 = x[c].w ^ 0x80808080u;
                            lo = make_uint4(i8x2_to_h2(x0, 0x5140), i8x2_to_h2(x0, 0x7362), i8x2_to_h2(x1, 0x5140),
                                            i8x2_to_h2(x1, 0x7362));
                            hi = make_uint4(i8x2_to_h2(x2, 0x5140), i8x2_to_h2(x2, 0x7362), i8x2_to_h2(x3, 0x5140),
                                            i8x2_to_h2(x3, 0x7362));
                        }
                        const int u = (D / 16) * half + 2 * c;
                        *reinterpret_cast<uint4 *>(row + ((u ^ (key & 7)) << 4)) = lo;
                        *reinterpret_cast<uint4 *>(row + (((u + 1) ^ (key & 7)) << 4)) = hi;
                    }
                    fence_async_smem();  // read by the MMAs
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sh.vfull[vs]);
                    if (++vs == GVS) vs = 0, vph ^= 1;
                }
            }
            prev = ti;
        }
        if (n > 0) read_out(prev, (n - 1) & 1, (uint32_t)((n - 1) >> 1) & 1u);
    } else if (warp == GMMA_WARP) {
        // ---------------- MMAs
        if (elect_one()) {
            const uint64_t ones = smem_desc_plain(sa(ONES), 128, 256);
            uint32_t vs = 0, vph = 0, ps = 0, pph = 0;
            for (int it = 0; it < n; ++it, ti = gen_next(p, ti)) {
                const int nh = ti.nsplit < ti.rows ? 2 : 1, par = it & 1;
                if (it >= 2) mbar_wait(&sh.dfree[par], (uint32_t)((it - 2) >> 1) & 1u, abort_flag);
                for (int kb = 0; kb < nkb; ++kb) {
                    const int ns = min(4, nsteps - 4 * kb);
                    mbar_wait(&sh.pfull[ps], pph, abort_flag);
                    const uint32_t at = tmem + G_TA + 32 * ps;
                    for (int hh = 0; hh < nh; ++hh) {
                        mbar_wait(&sh.vfull[vs], vph, abort_flag);
                        tc_fence_after();
                        const uint64_t bd = smem_desc(sa(VS) + vs * GV_BYTES, 1024, 1024);
                        for (int s = 0; s < ns; ++s)
                            mma_f16_ta(tmem + 128 * par + 64 * hh, at + 8 * s, bd + (uint64_t)(2048 >> 4) * s,
                                       (kb | s) != 0);
                        mma_commit(&sh.vfree[vs]);
                        if (++vs == GVS) vs = 0, vph ^= 1;
                    }
                    if (D == 64 && p.zp != 0)
                        for (int s = 0; s < ns; ++s)
                            mma_f16_ta(tmem + G_TR + 16 * par, at + 8 * s, ones, (kb | s) != 0, kIdescOnes);
                    mma_commit(&sh.pfree[ps]);
                    if (++ps == GPS) ps = 0, pph ^= 1;
                }
                mma_commit(&sh.dfull[par]);
            }
            // every MMA issued has completed before tensor memory is freed
            mma_commit(&sh.fin);
            mbar_wait(&sh.fin, 0, abort_flag, false);
        }
        __syncwarp();
    } else {
        // ---------------- copies of the logits tiles
        if (elect_one()) {
            int issued = 0;
            for (int it = 0; it < n; ++it, ti = gen_next(p, ti)) {
                const int lb = p.nlg == 2 ? it & 1 : 0, use = p.nlg == 2 ? it >> 1 : it;
                // (to the end of the last row's keys: the bytes behind them may not be the caller's to read)
                const uint32_t bytes = (uint32_t)((ti.rows - 1) * p.ld) + 16u * nsteps;
                if (it >= p.nlg) {
                    prefetch_l2(p.logits + (size_t)ti.g0 * p.ld, bytes);
                    if (!mbar_wait(&sh.lfree[lb], (uint32_t)(use - 1) & 1u, abort_flag)) break;
                }
                mbar_expect_tx(&sh.lload[lb], bytes);
                bulk_g2s(LG + (size_t)lb * GM * p.ld, p.logits + (size_t)ti.g0 * p.ld, bytes, &sh.lload[lb]);
                ++issued;
            }
            for (int j = issued > p.nlg ? issued - p.nlg : 0; j < issued; ++j)  // no copy may land after the exit
                mbar_wait(&sh.lload[p.nlg == 2 ? j & 1 : 0], (uint32_t)(p.nlg == 2 ? j >> 1 : j) & 1u, abort_flag, false);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == GMMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G_TMEM));
}

// Shared-memory layout for the shape; false when it does not fit
bool gen_layout(const LisArgs &a, GenParams &p, uint32_t &smem)
{
    const bool bias = a.bias != nullptr;
    const int nkb = (a.L + 63) / 64, Lp = (a.L + 15) & ~15;
    auto up = [](uint64_t x, uint64_t al) { return (x + al - 1) / al * al; };
    const int dmax = bias ? 510 : 255, clamp = 15 * -p.ic.q_ln2;
    p.ne = (bias ? (clamp < dmax ? clamp : dmax) : dmax) + 1;
    uint64_t o = up((uint64_t)p.ne * 256, 1024);
    p.off_c = (uint32_t)o;
    p.off_v = (uint32_t)(o = up(o + GC_END, 1024));
    p.off_b = (uint32_t)(o += GVS * GV_BYTES);
    const int nb = 2 * a.window - 1;
    if (bias) o = up(o + (uint64_t)nkb * 64 * 8 + (uint64_t)a.heads * nb * nb, 16);
    p.off_r = (uint32_t)o;
    if (a.region) o = up(o + (uint64_t)a.n_windows * (Lp + 1), 16);
    p.off_lg = (uint32_t)o;
    const uint64_t tile = (uint64_t)GM * a.ld_logit;
    p.nlg = o + 2 * tile <= kSmemOptin ? 2 : 1;
    o += p.nlg * tile;
    smem = (uint32_t)o;
    return o <= kSmemOptin;
}

template <int NKB, bool MASK, int D>
cudaError_t gen_launch(const GenParams &p, uint32_t smem, int grid, cudaStream_t st)
{
    static SmemReady ready;
    return launch_prepared((const void *)lis_attn_gen_kernel<NKB, MASK, D>, smem, ready, [&] {
        return launch_pdl(lis_attn_gen_kernel<NKB, MASK, D>, dim3(grid), dim3(GTHREADS), smem, st, p);
    });
}

template <int D>
cudaError_t gen_launch_d(const LisArgs &a, const GenParams &p, uint32_t smem, int grid, cudaStream_t st)
{
    if (!a.bias) return gen_launch<0, false, D>(p, smem, grid, st);
    const bool mask = a.region != nullptr;
    switch ((a.L + 63) / 64) {
    case 1: return mask ? gen_launch<1, true, D>(p, smem, grid, st) : gen_launch<1, false, D>(p, smem, grid, st);
    case 2: return mask ? gen_launch<2, true, D>(p, smem, grid, st) : gen_launch<2, false, D>(p, smem, grid, st);
    case 3: return mask ? gen_launch<3, true, D>(p, smem, grid, st) : gen_launch<3, false, D>(p, smem, grid, st);
    default: return mask ? gen_launch<4, true, D>(p, smem, grid, st) : gen_launch<4, false, D>(p, smem, grid, st);
    }
}

}  // namespace

bool lis_attention_gen_eligible(const LisArgs &a, const AttnVArgs &b)
{
    if (a.codes != nullptr || a.rowsum != nullptr || a.L < GMIN_L || a.L > 1024 || !(b.d == 32 || b.d == 64))
        return false;
    if (a.bias ? a.L > 256 : a.region != nullptr) return false;
    if (a.ld_logit % 16 != 0 || ((uintptr_t)a.logits % 16) != 0) return false;
    if (b.ld_v % 16 != 0 || ((uintptr_t)b.v % 16) != 0) return false;
    if (b.out8 ? (b.ld_out8 % 16 != 0 || ((uintptr_t)b.out8 % 16) != 0)
               : (b.ld_acc % 8 != 0 || ((uintptr_t)b.acc % 32) != 0))
        return false;
    GenParams p{};
    p.ic = iexp_consts_host(a.s_logit);
    if (a.region && 15 * -p.ic.q_ln2 > 510) return false;
    uint32_t smem;
    return gen_layout(a, p, smem);
}

cudaError_t launch_lis_attention_gen(const LisArgs &a, const AttnVArgs &b, cudaStream_t st)
{
    GenParams p{};
    p.logits = a.logits;
    p.ld = a.ld_logit;
    p.v = b.v;
    p.ld_v = b.ld_v;
    p.acc = b.acc;
    p.ld_acc = b.ld_acc;
    p.BH = b.BH;
    p.L = a.L;
    p.zp = b.zp_v;
    p.ic = iexp_consts_host(a.s_logit);
    p.small_e = ((double)p.ic.q_b * p.ic.q_b + p.ic.q_c) * 32768.0 < 268435456.0;  // e(0) < 2^28
    p.pack = a.L >= GM;
    p.bias = a.bias;
    p.heads = a.bias ? a.heads : 1;
    p.window = a.bias ? a.window : 1;
    p.region = a.region;
    p.n_windows = a.region ? a.n_windows : 1;
    p.mask_c = a.mask_value < -1024 ? 1024 : -a.mask_value;
    p.out8 = b.out8;
    p.ld_out8 = b.ld_out8;
    p.rq = requant8_of(b.rq_n1, b.rq_n2, b.rq_zp, b.zp_v, a.L);
    uint32_t smem;
    if (!gen_layout(a, p, smem)) return cudaErrorInvalidConfiguration;
    const int64_t ntiles = p.pack ? (b.BH * a.L + GM - 1) / GM : b.BH * ((a.L + GM - 1) / GM);
    const int grid = (int)(ntiles < sm_count() ? ntiles : sm_count());
    return b.d == 32 ? gen_launch_d<32>(a, p, smem, grid, st) : gen_launch_d<64>(a, p, smem, grid, st);
}

cudaError_t read_clear_gen_status(int *status)
{
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(status, g_status, sizeof(int));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_status, &zero, sizeof(int));
}

}  // namespace fqvit
