// K6: far field of the single-layer representation (section 4.4):
//   a_L(theta) = sum_p sum_m c^p_m(theta) rho^p_m,
//   c^p_m(theta) = i e^{-i pi/4} sqrt(a_p) / (2 sqrt k) e^{-i k theta_hat . O_p}
//                  J_m(k a_p) e^{i m (theta - pi/2)},
// or, with J_m replaced by the row factor w_L J_m - k w_M J'_m, of the
// representation u = w_L L + w_M M (the double-layer vector a_M is
// -k J'_m / J_m times the single-layer one);
// (b_p cos(theta - alpha_p) = theta_hat . O_p).
//
// Bound by the FP64 pipe (2 multiply-adds per clock and SM).  With phi =
// theta - pi/2 the mode sum of a disk is taken in pairs +-m,
//   sum_m w_m e^{i m phi} = w_0 + sum_{m >= 1} A_m cos(m phi) + i B_m sin(m phi),
//   A_m = w_m + w_{-m}, B_m = w_m - w_{-m}, w_m = J_m rho_m,
// which is 4 real multiply-adds per pair and column instead of the 8 of two
// complex products; cos(m phi) and sin(m phi) do not depend on the disk, so
// a CTA makes them once for its 32 angles, and the disk's phase is applied
// once to the finished sum.  Lanes are angles; each warp takes its own disks
// (A_m, B_m staged in shared memory, read as broadcasts) and up to eight
// columns; the warps' sums meet in shared memory, and the disks are split
// over as many CTAs as fill the chip, whose sums a second kernel adds.
// Measured (GB300, the whole call): 400 disks, N = 20, 360 angles, one column
// 903 -> 86 us (one thread per angle and disk, complex recurrence in every
// thread, one CTA per angle before); the multiply-adds alone are 37 us.
#include <algorithm>

#include "msd_internal.cuh"

namespace {
constexpr int kAngles = 32;  // sample angles of a CTA, one per lane
constexpr int kWarps = 4;    // disks in flight per CTA

// Shared memory: cos, sin [Nmax + 1][32], then per warp A, B [Nmax + 1][RC];
// the A, B area is also the warps' reduction area.
size_t ff_smem(int Nmax, int RC) {
    return (size_t)(Nmax + 1) * kAngles * 16 +
           std::max((size_t)kWarps * (Nmax + 1) * RC * 32, (size_t)kWarps * kAngles * RC * 16);
}

template <int RC>
__global__ void __launch_bounds__(kWarps * 32)
    k_farfield(const MsdConfig* __restrict__ cfgs, int C, int Nmax, const double2* __restrict__ centre,
               const double* __restrict__ radius, const double2* __restrict__ J, int R, int T, int ttiles,
               const double* __restrict__ thetas, const double2* __restrict__ rho, double2* __restrict__ out) {
    extern __shared__ double2 ff_sh[];
    double2* cs = ff_sh;                                    // (cos m phi, sin m phi) at [m][lane]
    double2* ab = ff_sh + (size_t)(Nmax + 1) * kAngles;     // [warp][m][{A, B}][RC]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tile = blockIdx.x % ttiles, r0 = (blockIdx.x / ttiles) * RC;
    const int ci = blockIdx.y, z = blockIdx.z;
    const MsdConfig c = cfgs[ci];
    const int N = c.N;
    const int t = tile * kAngles + lane;
    const double th = thetas[min(t, T - 1)];
    double st, ct;
    sincos(th, &st, &ct);
    {  // warp w: orders w, w + kWarps, ... from e^{i w phi} and e^{i kWarps phi}
        const double phi = th - 0.5 * M_PI;
        double2 e, f;
        sincos(warp * phi, &e.y, &e.x);
        sincos(kWarps * phi, &f.y, &f.x);
        for (int m = warp; m <= N; m += kWarps) {
            cs[m * kAngles + lane] = e;
            e = cmul(e, f);
        }
    }
    __syncthreads();
    const double2 pre = cscale(cmul(make_double2(0.0, 1.0), make_double2(cos(-0.25 * M_PI), sin(-0.25 * M_PI))),
                               0.5 / sqrt(c.k));
    double2 acc[RC];
#pragma unroll
    for (int j = 0; j < RC; ++j) acc[j] = make_double2(0.0, 0.0);
    double2* my = ab + (size_t)warp * (Nmax + 1) * 2 * RC;
    for (int p = z * kWarps + warp; p < c.M; p += gridDim.z * kWarps) {
        const long long row0 = c.row_off + (long long)p * c.n + N;  // mode 0
        __syncwarp();
        for (int i = lane; i < (N + 1) * RC; i += 32) {
            const int m = i / RC, j = i % RC;
            double2 wp = make_double2(0.0, 0.0), wm = wp;
            if (r0 + j < R) {
                wp = cmul(J[row0 + m], rho[(row0 + m) * R + r0 + j]);
                if (m > 0) wm = cmul(J[row0 - m], rho[(row0 - m) * R + r0 + j]);
            }
            my[m * 2 * RC + j] = cadd(wp, wm);
            my[m * 2 * RC + RC + j] = csub(wp, wm);
        }
        __syncwarp();
        const int d = c.disk_off + p;
        const double2 O = centre[d];
        double sp, cp;
        sincos(-c.k * (ct * O.x + st * O.y), &sp, &cp);
        const double2 ph = cscale(cmul(pre, make_double2(cp, sp)), sqrt(radius[d]));
        double2 s[RC];
#pragma unroll
        for (int j = 0; j < RC; ++j) s[j] = my[j];
        for (int m = 1; m <= N; ++m) {
            const double2 e = cs[m * kAngles + lane];
#pragma unroll
            for (int j = 0; j < RC; ++j) {
                const double2 A = my[m * 2 * RC + j], B = my[m * 2 * RC + RC + j];
                s[j].x = fma(-B.y, e.y, fma(A.x, e.x, s[j].x));
                s[j].y = fma(B.x, e.y, fma(A.y, e.x, s[j].y));
            }
        }
#pragma unroll
        for (int j = 0; j < RC; ++j) cfma(acc[j], ph, s[j]);
    }
    __syncthreads();  // A, B are no longer read
#pragma unroll
    for (int j = 0; j < RC; ++j) ab[(warp * RC + j) * kAngles + lane] = acc[j];
    __syncthreads();
    for (int i = threadIdx.x; i < RC * kAngles; i += kWarps * 32) {
        const int tt = tile * kAngles + i / RC, j = i % RC;
        if (tt >= T || r0 + j >= R) continue;
        double2 s = make_double2(0.0, 0.0);
        for (int w = 0; w < kWarps; ++w) s = cadd(s, ab[(w * RC + j) * kAngles + i / RC]);
        out[(((long long)z * C + ci) * T + tt) * R + r0 + j] = s;
    }
}

// F = sum over the nz disk groups; eight lanes per element.
__global__ void k_farfield_sum(long long tot, int nz, const double2* __restrict__ part, double2* __restrict__ F) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long i = t / 8;
    double2 s = make_double2(0.0, 0.0);
    if (i < tot)
        for (int z = (int)(t % 8); z < nz; z += 8) s = cadd(s, part[z * tot + i]);
    for (int off = 4; off > 0; off >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    if (i < tot && t % 8 == 0) F[i] = s;
}

// Columns of a CTA: eight share the angle's phase and table reads, one for
// single columns; the disks are split so that about eight CTAs per SM run
// (four warps each keep the FP64 pipes busy), never below one disk per warp.
struct FfShape {
    int RC, ttiles, rgroups, nz;
};
FfShape ff_shape(int C, const MsdConfig* h_cfg, int R, int T) {
    FfShape f;
    f.RC = R >= 5 ? 8 : R >= 2 ? 4 : 1;
    f.ttiles = (T + kAngles - 1) / kAngles;
    f.rgroups = (R + f.RC - 1) / f.RC;
    int Mmax = 1;
    for (int c = 0; c < C; ++c) Mmax = std::max(Mmax, h_cfg[c].M);
    const long long base = (long long)f.ttiles * f.rgroups * C;
    const long long want = (152 * 8 + base - 1) / base;
    f.nz = (int)std::max<long long>(1, std::min<long long>({want, (Mmax + kWarps - 1) / kWarps, 1024}));
    return f;
}

template <int RC>
void ff_launch(const FfShape& f, const MsdConfig* d_cfg, int C, int Nmax, const double2* centre, const double* radius,
               const double2* J, int R, int T, const double* th, const double2* rho, double2* out, cudaStream_t s) {
    const size_t smem = ff_smem(Nmax, RC);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_farfield<RC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_farfield<RC><<<dim3(f.ttiles * f.rgroups, C, f.nz), kWarps * 32, smem, s>>>(d_cfg, C, Nmax, centre, radius, J, R,
                                                                                 T, f.ttiles, th, rho, out);
    g_msd_launches += 1;
}
}  // namespace

size_t farfield_part_bytes(int C, const MsdConfig* h_cfg, int R, int T) {
    const FfShape f = ff_shape(C, h_cfg, R, T);
    return f.nz > 1 ? (size_t)f.nz * C * T * R * sizeof(double2) : 0;
}

void launch_farfield(const MsdConfig* d_cfg, int C, const MsdConfig* h_cfg, const double2* d_centre,
                     const double* d_radius, const double2* J, int R, int T, const double* d_thetas,
                     const double2* rho, double2* part, double2* F, cudaStream_t s) {
    const FfShape f = ff_shape(C, h_cfg, R, T);
    int Nmax = 0;
    for (int c = 0; c < C; ++c) Nmax = std::max(Nmax, h_cfg[c].N);
    double2* out = f.nz > 1 ? part : F;
    if (f.RC == 8) ff_launch<8>(f, d_cfg, C, Nmax, d_centre, d_radius, J, R, T, d_thetas, rho, out, s);
    else if (f.RC == 4) ff_launch<4>(f, d_cfg, C, Nmax, d_centre, d_radius, J, R, T, d_thetas, rho, out, s);
    else ff_launch<1>(f, d_cfg, C, Nmax, d_centre, d_radius, J, R, T, d_thetas, rho, out, s);
    if (f.nz > 1) {
        const long long tot = (long long)C * T * R;
        k_farfield_sum<<<(unsigned)((tot * 8 + 255) / 256), 256, 0, s>>>(tot, f.nz, part, F);
        g_msd_launches += 1;
    }
}
