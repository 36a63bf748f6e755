// Digit-sliced form of the FP64 block-Toeplitz product on the tensor cores
// (kernel K3, any number of columns, stored generators).
//
// The FP64 pipe of this GPU (1.2 TFLOP/s) bounds the product at 60 times the
// time its bytes take, while the bf16 tensor cores stand idle at 1900.  The
// sums are therefore formed from exact integer products (Ozaki, Ogita, Oishi,
// Rump, "Error-free transformations of matrix multiplication", Numerical
// Algorithms 59, 2012): every generator and every scaled source value is
// written as kND = 7 signed digits of 8 bits below a common power of two,
//     v = 2^{E+1} sum_{i=1..7} d_i 256^{-i},   |d_i| <= 128,
// each digit is exact in bf16, products of digits and their sums over up to
// 9 K-steps of 16 are integers below 2^24 and so exact in the FP32
// accumulators of tcgen05.mma, and the sums of equal weight i + j are put
// together in 64-bit integers before they meet FP64.  The 28 digit products
// with i + j <= 8 are kept.  Per real product, what the digits cut off is below
// 2^-53 and what is dropped below 2^-51.4 of (largest generator) x (largest
// source value) of the group: six digit products of 2^14 at 2^{2 - 72}, for
// values just above half their power of two with every lower digit -128; with
// digits of either sign about 2^-55.  Folding a sum of up to 72 sources into
// 64 bits adds 2^-52 of that product once (tests/test_digit_mirror.py).
//
// With d = n - m (see k_matvec_tcs.cu) the sum over the sources q at fixed d
// is a GEMM whose K index runs over (q, {Re g, Im g}):
//   * A (M = 128 rows): source values, row = (mode j, column r, {Re, Im}) of a
//     tile of J modes x Rt columns; row Re holds (Re x, -Im x), row Im holds
//     (Im x, Re x).  A does not depend on d, so a CTA loads the digits of its
//     K-steps once and keeps them.
//   * B: generator digits of 32 targets; the rows of the digits j = 1, 2, ...
//     follow one another, so ONE MMA of digit i of A with N = 32 (8 - i) rows
//     of B forms all products (i, j), i + j <= 8, and its columns land on the
//     accumulators of the weights i + j, which lie in the same order.
// The result of shift d and row j belongs to target mode m = j - d: sums over
// d are kept in FP64 in shared memory in a window of J modes that moves by one
// per shift, and leave it (to the partial sums the finalize kernel adds) when
// their last shift has passed.
//
// The common powers of two.  E is taken per (target, shift) and per (mode,
// column) over a group of sources.  A term's error is then relative to the
// product of the two maxima, which belong to different sources; l_m g r_n is
// bounded by powers of (a_p + a_q)/b <= 1, and stays so with the largest a_q
// of the group in place of the source's own while the radii in a group differ
// by less than 2^{7.5/N} (which can put a source's terms 2^7.5 below the
// group's).  Sources are sorted by radius and grouped so; where eight neighbours
// in that order already differ by more, the form is not offered (ds_grouping).
//
// So the error of a row is one of the group's largest terms, which are the
// row's own where the columns are of similar size on all disks: at most 25
// roundings (2^-53) of |x| + sum |l g r x| of its row, 0.4 on average (radii
// 0.5 to 1.5, gaps of 0.01, N = 20, columns that fall off with the mode number
// or not).  Where a column is much larger on some disks than on others, rows
// that only see the small ones are less exact than with the FP64 pipe: disks
// of sizes spread over six decades, up to 2e4 roundings of such a row, 15 of
// the largest result.  msd_set_tile (KB = 4..7) keeps the row-wise accuracy.
//
//
// What bounds it: the drain of the accumulators.  A K-step of MMAs takes about
// 650 clocks (448 at the tensor pipe's peak; small N and the issue of short
// instructions take the rest), a shift's drain about 5600 for 8 x 16 results a
// warp, of which FP64 additions hold their pipe for 2048; long folds (up to 9
// K-steps) and few mode tiles make few drains.  Counters: tensor pipe 56 %, FP64
// pipe 28 %, DRAM 28 %.  Measured (GB300, whole product): 400 disks, N = 20, one
// column 1793 -> 188 to 202 us (by their groups of radii); 200 disks, N = 22, 16
// columns 9375 -> 480 us.  Against 64-bit references the error is that of the
// generators with either kernel (radii 0.5 to 1.5, gaps of 0.01, N = 20:
// 8.683e-15 here, 8.686e-15 with the FP64 pipe).
//
// Persistent: one CTA per SM walks its own list of items (ds_items cuts the
// work at equal shares, between shifts where it has to), so no wave is left
// half empty.  Roles: warp 0 issues the bulk copies (one thread), warp 1
// allocates TMEM and issues the MMAs (one thread), warps 2-17 drain the
// accumulators (two buffers, so that the MMAs of the next shift run
// meanwhile): warp w covers TMEM lanes 32 (w mod 4) .. and 8 of the 32
// targets; four such warps per scheduler hide one another's latencies (two
// took 1.25 times as long).  The integer sums become FP64 by integer
// instructions (to_fp64): a conversion would hold the FP64 pipe as long as the
// one addition that is left does.  Operand layout: K-major without swizzle, 8-row x 16-byte core
// matrices.  Every wait has a clock limit, as in k_matvec_tcs.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "msd_internal.cuh"
#include "pipeline.cuh"

__device__ int g_ds_status;  // bit 0: a wait of the digit-sliced kernel expired

namespace {

constexpr int kND = MSD_DS_DIGITS;
constexpr int kTile = MSD_TILE_P;            // targets per CTA
constexpr int kStage = kND * 2 * kTile * 16; // bytes of one B stage (one K-step): [Re, Im][digit][target][8 sources]
constexpr int kBHalf = kND * kTile * 16;
constexpr int kStagesMax = 16;               // B ring: as many stages as fit next to A and the window
constexpr int kDrainWarps = 16;              // four sets of four warps (128 lanes), eight targets a set
constexpr int kSetTargets = kTile / (kDrainWarps / 4);
constexpr int kCh = 4;                       // targets in flight per lane
constexpr int kEbShifts = 32 / kSetTargets;  // shifts whose exponents a warp holds
constexpr int kThreads = 64 + kDrainWarps * 32;
constexpr int kNonFinite = 1 << 24;          // exponent of a group with an infinity or NaN

// kind::f16 instruction descriptor: D F32, A and B BF16, both K-major.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
// (descriptors as two words: the upper ones are the same for every MMA)
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                         uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}" ::"r"(tmem_d),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(id), "r"(acc));
}
// 4 consecutive TMEM columns of this thread's lane
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

// ---------------------------------------------------------------- digits

__device__ __forceinline__ int biased_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Exponent E of a group from the largest biased exponent: |v| < 2^E.
__device__ __forceinline__ int group_exp(int ev) { return ev == 0x7ff ? kNonFinite : ev - 1022; }

// Digits of v (|v| < 2^E) as bf16 bit patterns, d[0] the leading one: the
// integer nearest to v 2^{8 kND - 1 - E}, split into bytes with the carries
// of balanced digits added at once.  0 for subnormal v and in a non-finite
// group (whose scale makes every result non-finite).
__device__ __forceinline__ void digits_of(double v, int E, uint32_t (&d)[kND]) {
    const int ev = biased_exp(v);
    const int hi = __double2hiint(v);
    long long I = 0;
    if (ev != 0 && E < kNonFinite) {
        const long long mant = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
        const int s = ev - 1075 + (8 * kND - 1) - E;  // <= 2 as |v| < 2^E
        if (s >= 0) I = mant << s;
        else if (s > -60) I = (mant + (1ll << (-s - 1))) >> -s;
        if (hi < 0) I = -I;
    }
    I += 0x808080808080ll;  // bias of the kND - 1 = 6 lower digits
#pragma unroll
    for (int b = 0; b < kND; ++b) {
        const int x = b < kND - 1 ? (int)((I >> (8 * b)) & 0xff) - 128 : (int)(I >> (8 * b));
        d[kND - 1 - b] = __float_as_uint((float)x) >> 16;
    }
}
static_assert(kND == 7, "the digit bias and the integer combination below are written for seven digits");

// E of the generators, EB[tile][group][l][target]: one CTA per (target,
// group, configuration), threads over l.
__global__ void __launch_bounds__(128) k_ds_exps_g(const DsCfg* __restrict__ cfgs, const int* __restrict__ grp_start,
                                                   const int* __restrict__ perm, const double2* __restrict__ G,
                                                   int* __restrict__ EB) {
    const DsCfg c = cfgs[blockIdx.z];
    const int p = blockIdx.x, g = blockIdx.y;
    if (p >= c.Mp || g >= c.ngrp) return;
    const int s0 = grp_start[c.grp_off + g] * 8, s1 = grp_start[c.grp_off + g + 1] * 8;
    for (int l = threadIdx.x; l < c.L; l += blockDim.x) {
        int ev = 0;
#pragma unroll 8
        for (int s = s0; s < s1; ++s) {
            const int q = perm[c.perm_off + s];
            if (q < 0) continue;
            const double2 v = G[c.gen_off + ((long long)q * c.Mp + p) * c.L + l];
            ev = max(ev, max(biased_exp(v.x), biased_exp(v.y)));
        }
        EB[c.eb_off + (((long long)(p / kTile) * c.ngrp + g) * c.L + l) * kTile + p % kTile] = group_exp(ev);
    }
}

// Digits of the generators in the B-operand order,
//   DG[tile][l][K-step][{Re, Im}][digit][target][8 sources].
// One CTA per (tile x 8 values of l, K-step, configuration): the 8 x 32 rows
// are staged so that reads run along l and writes along the targets.
constexpr int kDgL = 8;
__global__ void __launch_bounds__(256) k_ds_digits_g(const DsCfg* __restrict__ cfgs, const int* __restrict__ qgrp,
                                                     const int* __restrict__ perm, const double2* __restrict__ G,
                                                     const int* __restrict__ EB, unsigned char* __restrict__ DG) {
    __shared__ double2 sm[8][kTile][kDgL + 1];
    const DsCfg c = cfgs[blockIdx.z];
    const int lch = (c.L + kDgL - 1) / kDgL;
    const int tile = blockIdx.x / lch, l0 = (blockIdx.x % lch) * kDgL, qs = blockIdx.y;
    if (tile * kTile >= c.Mp || qs >= c.nqs) return;
    for (int i = threadIdx.x; i < 8 * kTile * kDgL; i += 256) {
        const int dl = i % kDgL, p = (i / kDgL) % kTile, s = i / (kDgL * kTile);
        const int q = perm[c.perm_off + qs * 8 + s];
        double2 v = make_double2(0.0, 0.0);
        if (q >= 0 && l0 + dl < c.L) v = G[c.gen_off + ((long long)q * c.Mp + tile * kTile + p) * c.L + l0 + dl];
        sm[s][p][dl] = v;
    }
    __syncthreads();
    const int p = threadIdx.x & 31, dl = threadIdx.x >> 5, l = l0 + dl;
    if (l >= c.L) return;
    const int E = EB[c.eb_off + (((long long)tile * c.ngrp + qgrp[c.qs_off + qs]) * c.L + l) * kTile + p];
    unsigned char* out = DG + (c.dg_off + ((long long)tile * c.L + l) * c.nqs + qs) * kStage + p * 16;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t w[kND][4];
#pragma unroll
        for (int s = 0; s < 8; s += 2) {
            uint32_t a[kND], b[kND];
            digits_of(h ? sm[s][p][dl].y : sm[s][p][dl].x, E, a);
            digits_of(h ? sm[s + 1][p][dl].y : sm[s + 1][p][dl].x, E, b);
#pragma unroll
            for (int i = 0; i < kND; ++i) w[i][s / 2] = a[i] | (b[i] << 16);
        }
#pragma unroll
        for (int i = 0; i < kND; ++i)
            *(uint4*)(out + h * kBHalf + i * kTile * 16) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
    }
}

// E of the scaled source columns, EX[group][j][r] (j, r as in memory): one
// CTA per (32 values of j R + r, group, configuration), eight warps over the
// sources of the group.
__global__ void __launch_bounds__(256) k_ds_exps_x(const DsCfg* __restrict__ cfgs, const int* __restrict__ grp_start,
                                                   const int* __restrict__ perm, int R, const double2* __restrict__ xs,
                                                   int* __restrict__ EX) {
    __shared__ int red[8][32];
    const DsCfg c = cfgs[blockIdx.z];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = blockIdx.y;
    const int e = blockIdx.x * 32 + lane, ne = c.n * R;
    if (blockIdx.x * 32 >= ne || g >= c.ngrp) return;
    const int s0 = grp_start[c.grp_off + g] * 8, s1 = grp_start[c.grp_off + g + 1] * 8;
    int ev = 0;
    if (e < ne) {
#pragma unroll 4
        for (int s = s0 + warp; s < s1; s += 8) {
            const int q = perm[c.perm_off + s];
            if (q < 0) continue;
            const double2 v = xs[(c.row_off + (long long)q * c.n) * R + e];
            ev = max(ev, max(biased_exp(v.x), biased_exp(v.y)));
        }
    }
    red[warp][lane] = ev;
    __syncthreads();
    if (warp == 0 && e < ne) {
        for (int w = 1; w < 8; ++w) ev = max(ev, red[w][lane]);
        EX[c.ex_off + (long long)g * ne + e] = group_exp(ev);
    }
}

// Digits of the scaled source columns in the A-operand order,
//   XD[column group][mode tile][K-step][digit][half][row][8 sources],
// row = 2 (j' Rt + r') + {Re, Im}; one thread per (j, r, K-step).
__global__ void __launch_bounds__(128) k_ds_digits_x(const DsCfg* __restrict__ cfgs, const int* __restrict__ qgrp,
                                                     const int* __restrict__ perm, int R, int Rt,
                                                     const double2* __restrict__ xs, const int* __restrict__ EX,
                                                     unsigned char* __restrict__ XD) {
    const DsCfg c = cfgs[blockIdx.z];
    const int e = blockIdx.x * 128 + threadIdx.x, ne = c.n * R, qs = blockIdx.y;
    if (e >= ne || qs >= c.nqs) return;
    const int j = e / R, r = e % R, cg = r / Rt, rr = r % Rt, mt = j / c.J, jj = j % c.J;
    const int E = EX[c.ex_off + (long long)qgrp[c.qs_off + qs] * ne + e];
    uint32_t re[kND][4], im[kND][4];
#pragma unroll
    for (int s = 0; s < 8; s += 2) {
        uint32_t a[kND], b[kND];
        double2 v[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int q = perm[c.perm_off + qs * 8 + s + k];
            v[k] = q < 0 ? make_double2(0.0, 0.0) : xs[(c.row_off + (long long)q * c.n) * R + e];
        }
        digits_of(v[0].x, E, a);
        digits_of(v[1].x, E, b);
#pragma unroll
        for (int i = 0; i < kND; ++i) re[i][s / 2] = a[i] | (b[i] << 16);
        digits_of(v[0].y, E, a);
        digits_of(v[1].y, E, b);
#pragma unroll
        for (int i = 0; i < kND; ++i) im[i][s / 2] = a[i] | (b[i] << 16);
    }
    const int half = c.rp * 16;
    unsigned char* out = XD + c.xd_off + (((long long)cg * c.mt + mt) * c.nqs + qs) * (2 * kND * half) +
                         2 * (jj * Rt + rr) * 16;
    constexpr uint32_t kNeg = 0x80008000u;  // sign of both bf16 values (-0 where a digit is 0)
#pragma unroll
    for (int i = 0; i < kND; ++i) {
        const uint4 x = make_uint4(re[i][0], re[i][1], re[i][2], re[i][3]);
        const uint4 y = make_uint4(im[i][0], im[i][1], im[i][2], im[i][3]);
        unsigned char* o = out + 2 * i * half;
        *(uint4*)(o) = x;                                                             // row Re, Re g
        *(uint4*)(o + 16) = y;                                                        // row Im, Re g
        *(uint4*)(o + half) = make_uint4(y.x ^ kNeg, y.y ^ kNeg, y.z ^ kNeg, y.w ^ kNeg);  // row Re, Im g
        *(uint4*)(o + half + 16) = x;                                                 // row Im, Im g
    }
}

// ---------------------------------------------------------------- the product

// t 2^ex rounded to 53 bits, 0 below the normal range, infinite above it.
__device__ __noinline__ double to_double_any(long long t, int ex) {
    unsigned long long u = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
    const int lz = __clzll((long long)u);
    u <<= (lz & 63);
    const int e = 1023 + 63 - lz + ex;  // biased exponent of t 2^ex
    // 53 bits with the leading one, which adds 1 to the exponent field; a carry of the rounding does too
    unsigned long long b = (u >> 11) + ((u >> 10) & 1) + ((unsigned long long)(unsigned)(e - 1) << 52);
    if (e < 1 || u == 0) b = 0;
    if (e > 2046) b = 0x7ff0000000000000ull;
    return __longlong_as_double((long long)(b | ((unsigned long long)t & 0x8000000000000000ull)));
}

// One result from its accumulators a_s (s = 2..8, |a_s| <= 2^21.2 (s - 1)):
// t = sum_s a_s 2^{56 - 8 s} as a 64-bit integer (below 2^62; a_8 rounded into
// a_7), then t 2^ex in FP64.  About 35 integer instructions: the usual case,
// |t| >= 2^32 and a result in the normal range, without branches (a negative t
// loses one unit, 2^-56 of the largest product); the rest in to_double_any.
__device__ __forceinline__ double to_fp64(const uint32_t (&v)[kND][kCh], int u, int ex, bool wanted) {
    const int x = (int)__uint_as_float(v[0][u]) * 256 + (int)__uint_as_float(v[1][u]);
    const int y = (int)__uint_as_float(v[2][u]) * 256 + (int)__uint_as_float(v[3][u]);
    const int z = __float2int_rn(fmaf(__uint_as_float(v[6][u]), 0.00390625f, __uint_as_float(v[5][u])));
    long long t = (long long)(int)__uint_as_float(v[4][u]) * 256 + z;
    t = (long long)y * 65536 + t;
    const int hi = (int)(t >> 32) + x;
    const uint32_t lo = (uint32_t)t;
    const int s = hi >> 31;
    const uint32_t ah = (uint32_t)(hi ^ s), al = lo ^ (uint32_t)s;
    const int lz = __clz((int)ah);
    const uint32_t h = __funnelshift_l(al, ah, lz), l = al << (lz & 31);
    const int e1 = 1022 + 63 + ex - lz;  // biased exponent less the leading one of the mantissa
    const unsigned long long m = ((unsigned long long)((h >> 11) + ((uint32_t)e1 << 20)) << 32 |
                                  __funnelshift_r(l, h, 11)) + ((l >> 10) & 1);
    double r = __longlong_as_double((long long)(m | (unsigned long long)((uint32_t)s & 0x80000000u) << 32));
    if (wanted && (ah == 0 || (unsigned)e1 > 2044u))
        r = to_double_any((long long)(((unsigned long long)(uint32_t)hi << 32) | lo), ex);
    return r;
}

struct DsParams {
    const DsCfg* cfgs;
    const DsWork* works;
    const int* cta_off;  // items of CTA b: [cta_off[b], cta_off[b + 1])
    const unsigned char* DG;
    const int* EB;
    const unsigned char* XD;
    const int* EX;
    double* part;
    const int* live;
    long long Ntot;
    int R, Rt, stages;
    unsigned ring_off, acc_off;  // shared memory: A at 0, the B ring, the FP64 window
    int expire_test;
};

// Whether an item has nothing to multiply: a slot its targets have no work
// for, or no active column (converged Krylov systems).  A whole warp.
__device__ __forceinline__ bool item_idle(const DsParams& P, const DsWork& w, int r0, int cols) {
    if (w.ks == 0) return true;
    if (!P.live) return false;
    bool any = false;
    for (int r = threadIdx.x & 31; r < cols; r += 32) any |= P.live[w.cfg * P.R + r0 + r] != 0;
    return !__any_sync(0xffffffffu, any);
}

__global__ void __launch_bounds__(kThreads, 1) k_bt_ds(DsParams P) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ uint32_t tmem_sh;
    __shared__ __align__(8) uint64_t a_full, a_empty, b_full[kStagesMax], b_empty[kStagesMax], acc_full[2], acc_empty[2],
        mma_done;
    __shared__ int abort_sh, never_sh;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = P.R, Rt = P.Rt, kStages = P.stages;
    const int it0 = P.cta_off[blockIdx.x], it1 = P.cta_off[blockIdx.x + 1];
    unsigned char* ring = sm + P.ring_off;
    double* acc = (double*)(sm + P.acc_off);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        abort_sh = 0;
        never_sh = 0;
        mbar_init(&a_full, 1);
        mbar_init(&a_empty, 1);
        for (int s = 0; s < kStagesMax; ++s) {
            mbar_init(&b_full[s], 1);
            mbar_init(&b_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kDrainWarps);
        }
        mbar_init(&mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_sh;
    volatile int* abort_v = &abort_sh;
    int issued_mma = 0;

    if (warp == 0) {
        // ---------------- producer: A of an item, then one B stage per (shift, K-step)
        int s = 0, used = 0, na = 0;  // ring position, stages filled, items loaded
        uint32_t ph = 1;              // parity of the release to wait for (from the second lap)
        bool dead = false;            // a wait has expired: the copies go on, waiting only for themselves
        for (int it = it0; it < it1; ++it) {
            const DsWork w = P.works[it];
            const DsCfg c = P.cfgs[w.cfg];
            if (item_idle(P, w, w.cg * Rt, min(Rt, R - w.cg * Rt))) continue;
            if (elect_one()) {
                const int ablk = 2 * kND * c.rp * 16;
                const uint32_t aprev = (uint32_t)((na - 1) & 1);
                if (na > 0) {  // the MMAs of the item before have read its A
                    if (!dead) dead = !mbar_wait(smem_u32(&a_empty), aprev, abort_v);
                    if (dead) mbar_settle(smem_u32(&a_full), aprev);
                }
                const unsigned char* xa = P.XD + c.xd_off + (((long long)w.cg * c.mt + w.mt) * c.nqs + w.qs0) * ablk;
                mbar_expect_tx(smem_u32(&a_full), (uint32_t)(w.ks * ablk));
                for (int k = 0; k < w.ks; ++k)
                    bulk_g2s(smem_u32(sm + k * ablk), xa + (long long)k * ablk, (uint32_t)ablk, smem_u32(&a_full));
                const unsigned char* gd = P.DG + (c.dg_off + ((long long)w.tile * c.L + w.dlo + 2 * c.N) * c.nqs +
                                                  w.qs0) * (long long)kStage;
                for (int d = w.dlo; d <= w.dhi; ++d, gd += (long long)c.nqs * kStage)
                    for (int k = 0; k < w.ks; ++k) {
                        if (used >= kStages) {
                            if (!dead) dead = !mbar_wait(smem_u32(&b_empty[s]), ph, abort_v);
                            if (dead) mbar_settle(smem_u32(&b_full[s]), ph);
                        }
                        mbar_expect_tx(smem_u32(&b_full[s]), kStage);
                        bulk_g2s(smem_u32(ring + s * kStage), gd + (long long)k * kStage, kStage,
                                 smem_u32(&b_full[s]));
                        ++used;
                        if (++s == kStages) {
                            s = 0;
                            ph ^= 1;
                        }
                    }
                ++na;
            }
            __syncwarp();
        }
        // every copy of this CTA has landed before it exits
        if (na > 0) mbar_settle(smem_u32(&a_full), (uint32_t)((na - 1) & 1));
        for (int s2 = 0; s2 < kStages; ++s2)
            if (used > s2) mbar_settle(smem_u32(&b_full[s2]), (uint32_t)(((used - 1 - s2) / kStages) & 1));
    } else if (warp == 1) {
        // ---------------- MMA issue
        const uint64_t bdesc0 = sdesc(smem_u32(ring), kBHalf, 128);
        int s = 0, na = 0, gd = 0;  // ring position, items begun, shifts issued
        uint32_t ph = 0;
        bool dead = false;
        for (int it = it0; it < it1; ++it) {
            const DsWork w = P.works[it];
            const DsCfg c = P.cfgs[w.cfg];
            if (item_idle(P, w, w.cg * Rt, min(Rt, R - w.cg * Rt))) continue;
            if (elect_one()) {
                const int half = c.rp * 16;
                const uint32_t astep = 2 * half >> 4;  // one digit of A
                const uint64_t adesc0 = sdesc(smem_u32(sm), half, 128);
                const uint32_t a_hi = (uint32_t)(adesc0 >> 32), b_hi = (uint32_t)(bdesc0 >> 32);
                if (!dead) dead = !mbar_wait(smem_u32(&a_full), (uint32_t)(na & 1), abort_v);
                if (P.expire_test && na == 0 && !wait_unset_flag(&never_sh)) {
                    *abort_v = 1;
                    dead = true;
                }
                for (int d = w.dlo; d <= w.dhi; ++d, ++gd) {
                    const int b = gd & 1;
                    if (gd >= 2 && !dead)
                        dead = !mbar_wait(smem_u32(&acc_empty[b]), (uint32_t)(((gd >> 1) - 1) & 1), abort_v);
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const uint32_t tc = tmem + b * 256;
                    uint32_t a_lo = (uint32_t)adesc0;
                    for (int k = 0; k < w.ks; ++k) {
                        if (!dead) dead = !mbar_wait(smem_u32(&b_full[s]), ph, abort_v);
                        if (!dead) {
                            const uint32_t b_lo = (uint32_t)bdesc0 + s * (kStage >> 4);
#pragma unroll
                            for (int i = 0; i < kND; ++i, a_lo += astep)
                                mma_bf16(tc + i * kTile, a_lo, a_hi, b_lo, b_hi, idesc_bf16(128, kTile * (kND - i)),
                                         i == 0 ? (uint32_t)k : 1u);
                            issued_mma = 1;
                        }
                        mma_commit(smem_u32(&b_empty[s]));
                        if (++s == kStages) {
                            s = 0;
                            ph ^= 1;
                        }
                    }
                    mma_commit(smem_u32(&acc_full[b]));
                }
                mma_commit(smem_u32(&a_empty));
                ++na;
            }
            __syncwarp();
        }
        if (issued_mma) mma_commit(smem_u32(&mma_done));
    } else {
        // ---------------- drain: digit weights -> FP64, window over the target modes
        const int quarter = warp & 3, set = (warp - 2) >> 2;
        const int row = quarter * 32 + lane, e = row >> 1, ri = row & 1;
        const int jj = e / Rt, r = e % Rt;
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(set * kSetTargets);
        int gd = 0;
        bool dead = false;
        for (int it = it0; it < it1; ++it) {
            const DsWork w = P.works[it];
            const DsCfg c = P.cfgs[w.cfg];
            const int n = c.n, r0 = w.cg * Rt, cols = min(Rt, R - r0);
            const int jlo = w.mt * c.J, jhi = min(jlo + c.J, n) - 1, j = jlo + jj;
            const int t0 = w.tile * kTile + set * kSetTargets;  // first target of the set
            double* const out = P.part + (long long)w.slot * P.Ntot * R * 2;
            const bool idle = item_idle(P, w, r0, cols);
            // results (p, m, r) that no shift of the item reaches: m outside [mlo, mhi]
            const int mlo = idle ? n : jlo - w.dhi, mhi = idle ? -1 : jhi - w.dlo;
            if (mlo > 0 || mhi < n - 1) {
                const int tot = kSetTargets * n * 2 * cols;
                for (int i = quarter * 32 + lane; i < tot; i += 128) {
                    const int rc = i % (2 * cols), m = (i / (2 * cols)) % n, p = t0 + i / (2 * cols * n);
                    if (p < c.M && (m < mlo || m > mhi))
                        out[((c.row_off + (long long)p * n + m) * R + r0) * 2 + rc] = 0.0;
                }
            }
            if (idle) continue;
            const bool rowok = j <= jhi && r < cols;
            const int rows2 = 2 * c.J * Rt;  // doubles of the window per target
            const int EA = (rowok ? P.EX[c.ex_off + ((long long)w.grp * n + j) * R + r0 + r] : 0) - 54;
            const int* eb = P.EB + c.eb_off + (((long long)w.tile * c.ngrp + w.grp) * c.L + w.dlo + 2 * c.N) * kTile +
                            set * kSetTargets + (lane / kSetTargets) * kTile + lane % kSetTargets;
            double* const my = acc + (size_t)(set * kSetTargets) * rows2 + r * 2 + ri;
            double* const dst = out + ((c.row_off + (long long)t0 * n) * R + r0 + r) * 2 + ri;
            int m = j - w.dlo, slot = rowok ? ((m % c.J) + c.J) % c.J : 0;  // window position of mode m
            // exponents of a few shifts, one per lane; the next few are on their way
            // while these are used (L2 does not keep them beside the stream of digits)
            const int nd = w.dhi - w.dlo + 1;
            int EB = lane / kSetTargets < nd ? eb[0] : 0, EBn = 0;
            for (int d = w.dlo; d <= w.dhi; ++d, ++gd) {
                const int dd = d - w.dlo;
                if (dd % kEbShifts == 0) {
                    if (dd > 0) EB = EBn;
                    EBn = dd + kEbShifts + lane / kSetTargets < nd ? eb[(long long)(dd + kEbShifts) * kTile] : 0;
                }
                bool ok = !dead && mbar_wait(smem_u32(&acc_full[gd & 1]), (uint32_t)((gd >> 1) & 1), abort_v);
                ok = __all_sync(0xffffffffu, ok);
                dead = !ok;
                const bool valid = rowok && m >= 0 && m < n;
                const bool work = ok && t0 < c.M && __any_sync(0xffffffffu, valid);
                const bool last = j == jhi || d == w.dhi;
                const bool add = valid && !(jj == 0 || d == w.dlo);
                // the sum stays in the window, or leaves it for the partial sums
                const double* const cell = my + (size_t)slot * Rt * 2;
                double* const put = last ? dst + (long long)m * R * 2 : my + (size_t)slot * Rt * 2;
                const int putstep = last ? n * R * 2 : rows2;
                const int puts = !valid ? 0 : last ? c.M - t0 : kSetTargets;
                if (work) asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
                for (int h = 0; h < kSetTargets; h += kCh) {
                    uint32_t v[kND][kCh];
                    if (work) {
#pragma unroll
                        for (int s = 0; s < kND; ++s) tmem_ld4(lane_addr + (gd & 1) * 256 + s * kTile + h, v[s]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    }
                    if (h + kCh == kSetTargets) {  // the buffer is read: the MMAs of the shift after next may start
                        asm volatile("tcgen05.fence::before_thread_sync;");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&acc_empty[gd & 1]));
                    }
                    if (work) {
                        double x[kCh];
#pragma unroll
                        for (int u = 0; u < kCh; ++u) {
                            // 2^{EA + EB + 2 - 56}; a non-finite group's exponent makes its results infinite
                            const int ex = EA + __shfl_sync(0xffffffffu, EB, (dd % kEbShifts) * kSetTargets + h + u);
                            x[u] = to_fp64(v, u, ex, valid);
                        }
#pragma unroll
                        for (int u = 0; u < kCh; ++u) x[u] += add ? cell[(size_t)(h + u) * rows2] : 0.0;
#pragma unroll
                        for (int u = 0; u < kCh; ++u)
                            if (h + u < puts) put[(long long)(h + u) * putstep] = x[u];
                    }
                }
                --m;
                slot = slot == 0 ? c.J - 1 : slot - 1;
                // the window cells of this shift are written before the next shift reads them
                asm volatile("bar.sync %0, 128;" ::"r"(1 + set) : "memory");
            }
        }
    }
    // every MMA has completed before TMEM is freed
    __syncthreads();
    bool drained = true;
    if (issued_mma) drained = mbar_settle(smem_u32(&mma_done), 0);
    drained = __syncthreads_and(drained);
    if (tid == 0 && (abort_sh || !drained)) atomicOr(&g_ds_status, 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

}  // namespace

size_t ds_stage_bytes() { return kStage; }
size_t ds_xblk_bytes(int rp) { return (size_t)2 * kND * rp * 16; }

// Shared memory of one CTA with up to ks K-steps of A of rp rows and a window
// of rows2 doubles per target; the MMA of the last digit may read up to 128
// rows past its start, into the ring.
DsSmem ds_smem(int ks, int rp, int rows2) {
    DsSmem s;
    s.ring_off = (unsigned)((ks * ds_xblk_bytes(rp) + 127) / 128 * 128);
    const size_t window = (size_t)kTile * rows2 * sizeof(double);
    const long long room = (long long)kDsSmemCap - (long long)s.ring_off - (long long)window;
    s.stages = (int)std::max<long long>(3, std::min<long long>(kStagesMax, room / kStage));
    s.acc_off = s.ring_off + s.stages * kStage;
    s.total = s.acc_off + window;
    return s;
}

void launch_ds_build(const DsCfg* d_cfg, int C, int max_Mp, int max_grp, int max_L, int max_nqs, const int* d_grp_start,
                     const int* d_qgrp, const int* d_perm, const double2* G, int* EB, unsigned char* DG,
                     cudaStream_t s) {
    k_ds_exps_g<<<dim3(max_Mp, max_grp, C), 128, 0, s>>>(d_cfg, d_grp_start, d_perm, G, EB);
    k_ds_digits_g<<<dim3(max_Mp / kTile * ((max_L + kDgL - 1) / kDgL), max_nqs, C), 256, 0, s>>>(d_cfg, d_qgrp, d_perm,
                                                                                                G, EB, DG);
    g_msd_launches += 2;
}

void launch_ds_prep(const DsCfg* d_cfg, int C, int max_n, int max_grp, int max_nqs, const int* d_grp_start,
                    const int* d_qgrp, const int* d_perm, int R, int Rt, const double2* xs, int* EX, unsigned char* XD,
                    cudaStream_t s) {
    k_ds_exps_x<<<dim3((max_n * R + 31) / 32, max_grp, C), 256, 0, s>>>(d_cfg, d_grp_start, d_perm, R, xs, EX);
    k_ds_digits_x<<<dim3((max_n * R + 127) / 128, max_nqs, C), 128, 0, s>>>(d_cfg, d_qgrp, d_perm, R, Rt, xs, EX, XD);
    g_msd_launches += 2;
}

void launch_ds(const DsCfg* d_cfg, const DsWork* d_work, const int* d_cta_off, int nctas, const DsSmem& sm, const unsigned char* DG,
               const int* EB, const unsigned char* XD, const int* EX, double2* part, long long Ntot, int R, int Rt,
               cudaStream_t s, const int* live) {
    cudaFuncSetAttribute(k_bt_ds, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDsSmemCap);
    const DsParams P{d_cfg, d_work, d_cta_off, DG, EB, XD, EX, (double*)part, live, Ntot, R, Rt, sm.stages, sm.ring_off, sm.acc_off,
                     g_msd_expire_waits.load()};
    k_bt_ds<<<(unsigned)nctas, kThreads, sm.total, s>>>(P);
    g_msd_launches += 1;
}

int ds_status_and_clear() {
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_ds_status, sizeof(int)) != cudaSuccess) return -1;
    if (v) {
        const int z = 0;
        cudaMemcpyToSymbol(g_ds_status, &z, sizeof(int));
    }
    return v;
}
