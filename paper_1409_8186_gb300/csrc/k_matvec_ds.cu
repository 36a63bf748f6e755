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
// with i + j <= 8 are kept; what is dropped, and what the digits cut off, is
// below 2^-55 of (largest generator) x (largest source value), the size of an
// FP64 rounding error.
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
// by less than 2^{4/N}.  Sources are sorted by radius and grouped so; where
// eight neighbours in that order already differ by more, the form is not
// offered (ds_grouping).
//
// What bounds it: the tensor pipe for one column (28 products per
// multiply-add, 64 % of the rows in use), the FP64 pipe (a conversion and a
// multiply-add per shift and fold) from a few columns on.  Measured (GB300,
// whole product): 400 disks, N = 20, one column 1794 -> 436 us; 200 disks,
// N = 22, 16 columns 9371 -> 811 us; the error against 64-bit references is
// that of the generators on both sides (2.5e-14 before, 1.6e-14 now).
//
// Roles: warp 0 issues the bulk copies (one thread), warp 1 allocates TMEM
// and issues the MMAs (one thread), warps 2-9 drain the accumulators (two
// buffers, so that the MMAs of the next shift run meanwhile): warp w covers
// TMEM lanes 32 (w mod 4) .. and 16 of the 32 targets.  Operand layout:
// K-major without swizzle, 8-row x 16-byte core matrices.  Every wait has a
// clock limit, as in k_matvec_tcs.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "msd_internal.cuh"

__device__ int g_ds_status;  // bit 0: a wait of the digit-sliced kernel expired

namespace {

constexpr int kND = MSD_DS_DIGITS;
constexpr int kTile = MSD_TILE_P;            // targets per CTA
constexpr int kStage = kND * 2 * kTile * 16; // bytes of one B stage (one K-step): [Re, Im][digit][target][8 sources]
constexpr int kBHalf = kND * kTile * 16;
constexpr int kStages = 5;                   // B ring
constexpr int kThreads = 320;
constexpr int kNonFinite = 1 << 24;          // exponent of a group with an infinity or NaN
constexpr long long kWaitCycles = 2000000000LL;  // ~1 s at 2 GHz
constexpr long long kTestWaitCycles = 20000;     // msd_test_expire_waits

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: K-major, no swizzle, given strides
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}
// kind::f16 instruction descriptor: D F32, A and B BF16, both K-major.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, q;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > kWaitCycles) return false;
    }
}
__device__ __forceinline__ bool wait_unset_flag(const volatile int* flag) {
    const long long t0 = clock64();
    while (!*flag)
        if (clock64() - t0 > kTestWaitCycles) return false;
    return true;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// global -> shared bulk copy completing on an mbarrier (16-byte aligned, size % 16 == 0)
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar));
}
// 8 consecutive TMEM columns of this thread's lane, as integers
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
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

// Integer sum_s a_s 2^{56 - 8 s} (s = 2..8; a_8 rounded) of the accumulators
// of one result; |a_s| <= 2^21.2 (s - 1), so it stays below 2^62.
__device__ __forceinline__ double combine(const int (&a)[kND]) {
    long long t = (long long)(a[0] * 256 + a[1]) * (1ll << 32);
    t += (long long)a[2] * (1 << 24);
    t += (long long)a[3] * (1 << 16);
    t += (long long)a[4] * (1 << 8);
    t += (long long)(a[5] + ((a[6] + 128) >> 8));
    return (double)t;
}

struct DsParams {
    const DsCfg* cfgs;
    const DsWork* works;
    const unsigned char* DG;
    const int* EB;
    const unsigned char* XD;
    const int* EX;
    double* part;
    const int* live;
    long long Ntot;
    int R, Rt;
    unsigned ring_off, acc_off;  // shared memory: A at 0, the B ring, the FP64 window
    int expire_test;
};

__global__ void __launch_bounds__(kThreads, 1) k_bt_ds(DsParams P) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ uint32_t tmem_sh;
    __shared__ __align__(8) uint64_t a_full, b_full[kStages], b_empty[kStages], acc_full[2], acc_empty[2], mma_done;
    __shared__ int abort_sh, never_sh;

    const DsWork w = P.works[blockIdx.x];
    const DsCfg c = P.cfgs[w.cfg];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = P.R, Rt = P.Rt, n = c.n, N = c.N, L = c.L;
    const int r0 = w.cg * Rt, cols = min(Rt, R - r0);
    const int p0 = w.tile * kTile;
    double* const out = P.part + (long long)w.slot * P.Ntot * R * 2;

    // results (p, m, r) of this item that no shift reaches: m outside [mlo, mhi]
    auto zero_outside = [&](int mlo, int mhi, int first, int step) {
        if (mlo <= 0 && mhi >= n - 1) return;
        const int tot = kTile * n * 2 * cols;
        for (int i = first; i < tot; i += step) {
            const int rc = i % (2 * cols), m = (i / (2 * cols)) % n, p = p0 + i / (2 * cols * n);
            if (p < c.M && (m < mlo || m > mhi))
                out[((c.row_off + (long long)p * n + m) * R + r0) * 2 + rc] = 0.0;
        }
    };
    bool none = w.ks == 0;  // a slot this configuration has no work for
    if (!none && P.live) {  // no active column (converged Krylov systems)
        bool any = false;
        for (int r = 0; r < cols; ++r) any |= P.live[w.cfg * R + r0 + r] != 0;
        none = !any;
    }
    if (none) {
        zero_outside(n, -1, tid, kThreads);
        return;
    }

    const int half = c.rp * 16, ablk = 2 * kND * half;  // bytes of one K half and of one K-step of A
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
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&b_full[s], 1);
            mbar_init(&b_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 8);
        }
        mbar_init(&mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_sh;
    volatile int* abort_v = &abort_sh;
    const int nd = w.dhi - w.dlo + 1;
    int issued_mma = 0;

    if (warp == 0 && lane == 0) {
        // ---------------- producer: A once, then one B stage per (shift, K-step)
        const unsigned char* xa = P.XD + c.xd_off + (((long long)w.cg * c.mt + w.mt) * c.nqs + w.qs0) * ablk;
        mbar_expect_tx(smem_u32(&a_full), (uint32_t)(w.ks * ablk));
        for (int k = 0; k < w.ks; ++k)
            bulk_g2s(smem_u32(sm + k * ablk), xa + (long long)k * ablk, (uint32_t)ablk, smem_u32(&a_full));
        const unsigned char* gd =
            P.DG + (c.dg_off + ((long long)w.tile * L + w.dlo + 2 * N) * c.nqs + w.qs0) * (long long)kStage;
        int s = 0, used = 0;  // ring position, stages filled so far
        uint32_t ph = 1;      // parity of the release to wait for (from the second lap)
        for (int d = 0; d < nd; ++d, gd += (long long)c.nqs * kStage)
            for (int k = 0; k < w.ks; ++k) {
                if (used >= kStages) {
                    if (!*abort_v && !mbar_wait(smem_u32(&b_empty[s]), ph)) *abort_v = 1;
                    mbar_wait(smem_u32(&b_full[s]), ph);  // own previous copy landed before re-arming
                }
                mbar_expect_tx(smem_u32(&b_full[s]), kStage);
                bulk_g2s(smem_u32(ring + s * kStage), gd + (long long)k * kStage, kStage, smem_u32(&b_full[s]));
                ++used;
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1;
                }
            }
        // every copy of this CTA has landed before it exits
        mbar_wait(smem_u32(&a_full), 0);
        for (int s2 = 0; s2 < kStages; ++s2)
            if (used > s2) mbar_wait(smem_u32(&b_full[s2]), (uint32_t)(((used - 1 - s2) / kStages) & 1));
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issue
        const uint64_t adesc0 = sdesc(smem_u32(sm), half, 128), bdesc0 = sdesc(smem_u32(ring), kBHalf, 128);
        bool ok = mbar_wait(smem_u32(&a_full), 0);
        if (P.expire_test) ok = wait_unset_flag(&never_sh) && ok;
        if (!ok) *abort_v = 1;
        int s = 0;
        uint32_t ph = 0;
        for (int d = 0; d < nd; ++d) {
            const int b = d & 1;
            if (d >= 2 && !*abort_v && !mbar_wait(smem_u32(&acc_empty[b]), (uint32_t)(((d >> 1) - 1) & 1)))
                *abort_v = 1;
            for (int k = 0; k < w.ks; ++k) {
                if (!*abort_v && !mbar_wait(smem_u32(&b_full[s]), ph)) *abort_v = 1;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint64_t bd = bdesc0 + (uint64_t)(s * (kStage >> 4));
                const uint64_t ad = adesc0 + (uint64_t)(k * (ablk >> 4));
                if (!*abort_v) {
#pragma unroll
                    for (int i = 0; i < kND; ++i)
                        mma_bf16(tmem + b * 256 + i * kTile, ad + (uint64_t)(i * (2 * half >> 4)), bd,
                                 idesc_bf16(128, kTile * (kND - i)), (i == 0 && k == 0) ? 0u : 1u);
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
        mma_commit(smem_u32(&mma_done));
    } else if (warp >= 2) {
        // ---------------- drain: digit weights -> FP64, window over the target modes
        const int quarter = warp & 3, set = (warp - 2) >> 2;
        const int row = quarter * 32 + lane, e = row >> 1, ri = row & 1;
        const int jj = e / Rt, r = e % Rt;
        const int jlo = w.mt * c.J, jhi = min(jlo + c.J, n) - 1, j = jlo + jj;
        const bool rowok = j <= jhi && r < cols;
        const int rows2 = 2 * c.J * Rt;  // doubles of the window per target
        const int EA = rowok ? P.EX[c.ex_off + ((long long)w.grp * n + j) * R + r0 + r] : 0;
        const int* eb = P.EB + c.eb_off + (((long long)w.tile * c.ngrp + w.grp) * L + w.dlo + 2 * N) * kTile +
                        set * 16 + (lane & 15);
        const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(set * 16);
        double* const my = acc + (size_t)(set * 16) * rows2 + r * 2 + ri;
        double* const dst = out + ((c.row_off + (long long)(p0 + set * 16) * n) * R + r0 + r) * 2 + ri;
        int m = j - w.dlo, slot = rowok ? ((m % c.J) + c.J) % c.J : 0;  // window position of mode m
        int EB = *eb;
        for (int d = 0; d < nd; ++d) {
            const int EBn = d + 1 < nd ? eb[(long long)(d + 1) * kTile] : 0;
            bool ok = *abort_v ? false : mbar_wait(smem_u32(&acc_full[d & 1]), (uint32_t)((d >> 1) & 1));
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) *abort_v = 1;
            const bool valid = rowok && m >= 0 && m < n;
            if (ok && __any_sync(0xffffffffu, valid)) {
                asm volatile("tcgen05.fence::after_thread_sync;");
                const bool first = jj == 0 || d == 0, last = j == jhi || d == nd - 1;
                double* const cell = my + (size_t)slot * Rt * 2;
                double* const cellout = dst + (long long)m * R * 2;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t v[kND][8];
#pragma unroll
                    for (int s = 0; s < kND; ++s) tmem_ld8(lane_addr + (d & 1) * 256 + s * kTile + h * 8, v[s]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int t = h * 8 + u;
                        // 2^{EA + EB + 2 - 56}, 0 below the normal range, infinite above it
                        const int ex = EA + __shfl_sync(0xffffffffu, EB, t) + (1023 - 54);
                        const double scale = __hiloint2double(max(0, min(2047, ex)) << 20, 0);
                        int a[kND];
#pragma unroll
                        for (int s = 0; s < kND; ++s) a[s] = (int)__uint_as_float(v[s][u]);
                        if (valid) {
                            const double old = first ? 0.0 : cell[(size_t)t * rows2];
                            const double s = fma(combine(a), scale, old);
                            if (!last) cell[(size_t)t * rows2] = s;
                            else if (p0 + set * 16 + t < c.M) cellout[(long long)t * n * R * 2] = s;
                        }
                    }
                }
            }
            EB = EBn;
            --m;
            slot = slot == 0 ? c.J - 1 : slot - 1;
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[d & 1]));
            // the window cells of this shift are written before the next shift reads them
            asm volatile("bar.sync %0, 128;" ::"r"(1 + set) : "memory");
        }
        if (!*abort_v) zero_outside(jlo - w.dhi, jhi - w.dlo, tid - 64, kThreads - 64);
    }
    // every MMA has completed before TMEM is freed
    __syncthreads();
    bool drained = true;
    if (tid == 32 && issued_mma) drained = mbar_wait(smem_u32(&mma_done), 0);
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
    s.acc_off = s.ring_off + kStages * kStage;
    s.total = s.acc_off + (size_t)kTile * rows2 * sizeof(double);
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

void launch_ds(const DsCfg* d_cfg, const DsWork* d_work, int nwork, const DsSmem& sm, const unsigned char* DG,
               const int* EB, const unsigned char* XD, const int* EX, double2* part, long long Ntot, int R, int Rt,
               cudaStream_t s, const int* live) {
    if (nwork <= 0) return;
    cudaFuncSetAttribute(k_bt_ds, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDsSmemCap);
    const DsParams P{d_cfg, d_work, DG, EB, XD, EX, (double*)part, live, Ntot, R, Rt, sm.ring_off, sm.acc_off,
                     g_msd_expire_waits.load()};
    k_bt_ds<<<(unsigned)nwork, kThreads, sm.total, s>>>(P);
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
