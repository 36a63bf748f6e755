// K4: batched restarted GMRES on the device (section 5: preconditioned
// Krylov solve; the restarted GMRES call of section 6.2).
//
// A "system" is one (configuration, column) pair s = cfg*R + r; all systems
// advance in lock step (one block product per Arnoldi step serves all of
// them) and each carries its own Hessenberg matrix, Givens rotations and
// convergence state.
//
// Orthogonalisation is classical Gram-Schmidt with one selective
// re-orthogonalisation pass (Daniel-Gragg-Kaufman-Stewart criterion: repeat
// the projection when it left less than a fraction eta2 of ||w||^2, by
// default one half; the solver option reorth sets eta2).  Per-thread
// sums of dot products and updates run in the storage precision of the
// basis (FP32 for the inner sweeps of a mixed solve, whose FP64 pipe would
// otherwise bound them), cross-chunk reductions and the batches of the solution
// update in FP64.  Vectors are
// [rows][R] with R innermost; reductions run over row chunks that never
// straddle two configurations, of a size that follows the number of elements
// (rows x R) and not of rows alone, so that a few thousand rows with many
// columns still fill the chip.  Measured (GB300, averages over a solve): the
// FP64 gradient of 40 disks with 16 columns (1800 rows) took 100 us a
// projection and 155 us an update with row chunks, one vector per warp and FP64
// atomics, 355 -> 149 ms as a whole; eight FP32 systems of 60 disks with 32
// columns 303 -> 247 ms.
//
// The Givens rotations of a new Hessenberg column form the first-order
// linear recurrence z_{i+1} = -conj(s_i) z_i + c_i h_{i+1} (z_0 = h_0,
// rotated entry i = c_i z_i + s_i h_{i+1}); it is evaluated with a
// parallel scan of affine maps over one CTA per system (warp shuffles, then
// across warps), so a step costs O(j / threads + log threads) instead of a
// j-long dependency chain.
#include <algorithm>
#include <type_traits>

#include "msd_internal.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

template <typename V> __device__ __forceinline__ double2 to_d2(V v) { return make_double2(v.x, v.y); }

template <typename V> __device__ __forceinline__ V from_d2(double2 v) {
    return V{(decltype(V{}.x))v.x, (decltype(V{}.x))v.y};
}

// Columns of a column group (blockIdx of the kernels below): lane l of a warp
// holds column l mod RC of row l / RC of the warp's RPW = 32 / RC rows, so a
// warp reads RPW rows of one group as one contiguous stretch when R <= 32.
__host__ __device__ inline int col_group(int R) { return R < 32 ? R : 32; }

// Partial sums over one chunk of rows (blockIdx.x) and the columns of group
// blockIdx.z of the vectors i in the list V_0..V_{nv-1} followed, when self
// != 0, by w itself:
//   part[chunk][i][r] = sum_rows conj(u_i[row][r]) * w[row][r].
// Systems with skip[s] == skipval contribute zeros.  A warp takes IV vectors
// (each value of w read serves them all) and UN row groups at a time: IV UN +
// UN loads in flight per lane.
template <typename V, int IV>
__global__ void __launch_bounds__(kThreads) k_dots(const RowChunk* __restrict__ chunks, int R,
                                                   const V* __restrict__ Vb, long long vstride, int nv, int self,
                                                   const V* __restrict__ w, const int* __restrict__ skip, int skipval,
                                                   double2* __restrict__ part) {
    typedef decltype(V{}.x) A;
    constexpr int UN = 4;
    const RowChunk ch = chunks[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int RC = col_group(R), RPW = 32 / RC, nvv = nv + self;
    const int i0 = (blockIdx.y * kWarps + warp) * IV;
    if (i0 >= nvv) return;  // a whole warp
    const int ro = lane / RC, r = blockIdx.z * 32 + lane % RC;
    const bool act = ro < RPW && r < R && !(skip && skip[ch.cfg * R + r] == skipval);
    A ax[IV], ay[IV];
#pragma unroll
    for (int k = 0; k < IV; ++k) ax[k] = ay[k] = A(0);
    if (__any_sync(0xffffffffu, act)) {
        const V* u[IV];
#pragma unroll
        for (int k = 0; k < IV; ++k) u[k] = i0 + k < nv ? Vb + (long long)(i0 + k) * vstride : w;
        const int rows = (int)(ch.row1 - ch.row0);
        long long e = (ch.row0 + ro) * R + r;
        const long long step = (long long)RPW * R;
        for (int q = ro; q < rows; q += RPW * UN, e += UN * step) {
            V wv[UN], uv[UN][IV];
#pragma unroll
            for (int n = 0; n < UN; ++n) {
                const bool ok = act && q + n * RPW < rows;
                wv[n] = ok ? w[e + n * step] : V{A(0), A(0)};
#pragma unroll
                for (int k = 0; k < IV; ++k) uv[n][k] = ok ? u[k][e + n * step] : V{A(0), A(0)};
            }
#pragma unroll
            for (int n = 0; n < UN; ++n)
#pragma unroll
                for (int k = 0; k < IV; ++k) {  // conj(u) * w
                    ax[k] = fma(uv[n][k].x, wv[n].x, fma(uv[n][k].y, wv[n].y, ax[k]));
                    ay[k] = fma(uv[n][k].x, wv[n].y, fma(-uv[n][k].y, wv[n].x, ay[k]));
                }
        }
    }
    // lanes of one column: l, l + RC, ... (in the storage precision: at most 32 terms)
#pragma unroll
    for (int k = 0; k < IV; ++k) {
        if ((RC & (RC - 1)) == 0) {
            for (int off = 16; off >= RC; off >>= 1) {
                ax[k] += __shfl_xor_sync(0xffffffffu, ax[k], off);
                ay[k] += __shfl_xor_sync(0xffffffffu, ay[k], off);
            }
        } else {
            const A x0 = ax[k], y0 = ay[k];
            for (int n = 1; n < RPW; ++n) {
                ax[k] += __shfl_down_sync(0xffffffffu, x0, n * RC);
                ay[k] += __shfl_down_sync(0xffffffffu, y0, n * RC);
            }
        }
        if (lane < RC && r < R && i0 + k < nvv)
            part[((long long)blockIdx.x * nvv + i0 + k) * R + r] = make_double2((double)ax[k], (double)ay[k]);
    }
}

// The same for an FP32 basis with 16-byte loads, two neighbouring elements per
// lane: two columns of a row (R even), or two rows of a single column (R =
// 1).  For vectors and chunks that start on an even element (GmresDims::pairs),
// so that a chunk of a single column has an even number of rows.
// Halves the load instructions and doubles the bytes in flight: eight systems
// of 60 disks with 32 columns, 74 -> 54 us a projection (k_update_pair: 88 ->
// 62 us an update).
template <int IV>
__global__ void __launch_bounds__(kThreads) k_dots_pair(const RowChunk* __restrict__ chunks, int R,
                                                        const float2* __restrict__ Vb, long long vstride, int nv,
                                                        int self, const float2* __restrict__ w,
                                                        const int* __restrict__ skip, int skipval,
                                                        double2* __restrict__ part) {
    constexpr int UN = 4;
    const RowChunk ch = chunks[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool one = R == 1;
    const int PC = one ? 1 : col_group(R) / 2, RPW = 32 / PC, nvv = nv + self;
    const int i0 = (blockIdx.y * kWarps + warp) * IV;
    if (i0 >= nvv) return;  // a whole warp
    const int ro = lane / PC, r = blockIdx.z * 32 + 2 * (lane % PC);
    const bool in = ro < RPW && r < R;
    const bool act0 = in && !(skip && skip[ch.cfg * R + r] == skipval);
    const bool act1 = in && (one ? act0 : !(skip && skip[ch.cfg * R + r + 1] == skipval));
    float ax[IV][2], ay[IV][2];
#pragma unroll
    for (int k = 0; k < IV; ++k) ax[k][0] = ax[k][1] = ay[k][0] = ay[k][1] = 0.f;
    if (__any_sync(0xffffffffu, act0 || act1)) {
        const float2* u[IV];
#pragma unroll
        for (int k = 0; k < IV; ++k) u[k] = i0 + k < nv ? Vb + (long long)(i0 + k) * vstride : w;
        const int rows = (int)(ch.row1 - ch.row0);
        const int units = one ? rows / 2 : rows;        // a unit: a row, or two rows of one column
        const int unit = one ? 2 : R;                   // elements from one unit to the next
        long long e = ch.row0 * R + (long long)ro * unit + r;
        const long long step = (long long)RPW * unit;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = ro; q < units; q += RPW * UN, e += UN * step) {
            float4 wv[UN], uv[UN][IV];
#pragma unroll
            for (int n = 0; n < UN; ++n) {
                const bool ok = in && q + n * RPW < units;
                // (a branch: as conditional loads they are compiled to 64 registers with spills, 74 us for 67)
                if (ok) {
                    wv[n] = *(const float4*)(w + e + n * step);
#pragma unroll
                    for (int k = 0; k < IV; ++k) uv[n][k] = *(const float4*)(u[k] + e + n * step);
                } else {
                    wv[n] = zero;
#pragma unroll
                    for (int k = 0; k < IV; ++k) uv[n][k] = zero;
                }
            }
#pragma unroll
            for (int n = 0; n < UN; ++n)
#pragma unroll
                for (int k = 0; k < IV; ++k) {  // conj(u) * w
                    const float4 a = uv[n][k], b = wv[n];
                    ax[k][0] = fmaf(a.x, b.x, fmaf(a.y, b.y, ax[k][0]));
                    ay[k][0] = fmaf(a.x, b.y, fmaf(-a.y, b.x, ay[k][0]));
                    ax[k][1] = fmaf(a.z, b.z, fmaf(a.w, b.w, ax[k][1]));
                    ay[k][1] = fmaf(a.z, b.w, fmaf(-a.w, b.z, ay[k][1]));
                }
        }
    }
#pragma unroll
    for (int k = 0; k < IV; ++k) {
        if (one) {
            ax[k][0] += ax[k][1];
            ay[k][0] += ay[k][1];
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (one && c) continue;
            if ((PC & (PC - 1)) == 0) {
                for (int off = 16; off >= PC; off >>= 1) {
                    ax[k][c] += __shfl_xor_sync(0xffffffffu, ax[k][c], off);
                    ay[k][c] += __shfl_xor_sync(0xffffffffu, ay[k][c], off);
                }
            } else {
                const float x0 = ax[k][c], y0 = ay[k][c];
                for (int n = 1; n < RPW; ++n) {
                    ax[k][c] += __shfl_down_sync(0xffffffffu, x0, n * PC);
                    ay[k][c] += __shfl_down_sync(0xffffffffu, y0, n * PC);
                }
            }
            const bool act = c ? act1 : act0;
            if (lane < PC && r + c < R && i0 + k < nvv)
                part[((long long)blockIdx.x * nvv + i0 + k) * R + r + c] =
                    act ? make_double2((double)ax[k][c], (double)ay[k][c]) : make_double2(0.0, 0.0);
        }
    }
}

// ||w'||^2 = ||w||^2 - sum_{i <= j} |h_i|^2 and (skip2 != nullptr) the
// re-orthogonalisation flag of one system, reduced over the CTA (every thread
// calls it).
__device__ void reorth_flag_cta(const double2* h, int j, double2* wn2, int act, int* skip2, double eta2) {
    double acc = 0.0;
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
        const double2 v = __ldcg(h + i);
        acc += cabs2(v);
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    __shared__ double red[32];  // one slot per warp (blocks of up to 1024 threads)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double ss = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) ss += red[k];
        const double before = __ldcg(h + j + 1).x;  // ||w||^2 before the projection
        const double after = before - ss;
        *wn2 = make_double2(after, 0.0);
        if (skip2) *skip2 = !(act && after < eta2 * before);
    }
}

// out[s * ostride + i] = sum over the chunks of cfg(s) of part[chunk][i][r],
// and the same in the basis type, transposed to hT[cfg][i][r] (rows of ldh
// vectors), as the update kernel reads it.  One CTA per configuration
// (blockIdx.y) and 32 consecutive values of i R + r, whose partials lie
// side by side; eight threads share an output's chunks.
// With tail.cnt set (few systems), the last block to finish also forms
// wn2[s] = out[s][j + 1] - sum_{i <= j} |out[s][i]|^2 and, with tail.skip2,
// the re-orthogonalisation flags (k_reorth_flags), and puts the counter back
// to zero.
struct FinTail {
    int* cnt = nullptr;
    int S = 0, j = 0;
    double2* wn2 = nullptr;
    const int* active = nullptr;
    int* skip2 = nullptr;
    double eta2 = 0.5;  // second pass when ||w'||^2 < eta2 ||w||^2
};
constexpr int kFinY = 8;
template <typename V>
__global__ void __launch_bounds__(32 * kFinY) k_dots_fin(int R, int nvv, const int* __restrict__ cfg_chunk_off,
                                                         const double2* __restrict__ part, double2* __restrict__ out,
                                                         int ostride, V* __restrict__ hT, long long ldh,
                                                         FinTail tail) {
    __shared__ double2 red[kFinY][32];
    const int c = blockIdx.y, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + tx, ne = nvv * R;
    double2 acc = make_double2(0.0, 0.0);
    if (e < ne) {
        const int k1 = cfg_chunk_off[c + 1];
#pragma unroll 4
        for (int k = cfg_chunk_off[c] + ty; k < k1; k += kFinY) acc = cadd(acc, part[(long long)k * ne + e]);
    }
    red[ty][tx] = acc;
    __syncthreads();
    if (ty == 0 && e < ne) {
#pragma unroll
        for (int y = 1; y < kFinY; ++y) acc = cadd(acc, red[y][tx]);
        const int i = e / R, r = e % R;
        out[(long long)(c * R + r) * ostride + i] = acc;
        if (hT) hT[((long long)c * ldh + i) * R + r] = from_d2<V>(acc);
        if (tail.cnt) __threadfence();
    }
    if (!tail.cnt) return;
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(tail.cnt, 1) == (int)(gridDim.x * gridDim.y) - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int sy = 0; sy < tail.S; ++sy)
        reorth_flag_cta(out + (long long)sy * ostride, tail.j, tail.wn2 + (long long)sy * ostride,
                        tail.active ? tail.active[sy] : 1, tail.skip2 ? tail.skip2 + sy : nullptr, tail.eta2);
    if (threadIdx.x == 0) *tail.cnt = 0;
}

// hT[cfg][i][r] = y[s][i] in the basis type (the coefficients of the solution
// update at the end of a cycle).
template <typename V>
__global__ void k_coeffs(int C, int R, int nv, const double2* __restrict__ y, int ystride, V* __restrict__ hT,
                         long long ldh) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)C * nv * R) return;
    const int r = (int)(t % R), i = (int)((t / R) % nv), c = (int)(t / ((long long)R * nv));
    hT[((long long)c * ldh + i) * R + r] = from_d2<V>(y[(long long)(c * R + r) * ystride + i]);
}

// w[row][r] += sign * sum_{i < nv} V_i[row][r] hT[cfg][i][r], lane = element.
// SPLIT warps share 32 elements, each taking every SPLIT-th batch of U
// vectors (all U loads in flight, their coefficients coming from L1); a batch is
// summed in the basis precision and the batches in that of w (FP64 for the
// solution of a mixed solve, whose basis of up to 4000 FP32 vectors would lose
// the small terms otherwise; FP32 for a vector of its sweep).  The warps' sums
// meet in shared memory and w is written once, without atomics.
template <typename V, typename W, int SPLIT>
__global__ void __launch_bounds__(kThreads, sizeof(V) == 8 ? 4 : 2)
    k_update(const RowChunk* __restrict__ chunks, int R, const V* __restrict__ Vb, long long vstride, int nv,
             const V* __restrict__ hT, long long ldh, const int* __restrict__ skip, int skipval, double sign,
             W* __restrict__ w) {
    typedef decltype(V{}.x) A;
    typedef decltype(W{}.x) B;
    constexpr int U = 8;
    constexpr int kCols = kWarps / SPLIT;  // groups of 32 elements of the CTA
    __shared__ W red[kCols][SPLIT][32];
    const RowChunk ch = chunks[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sp = warp % SPLIT, cg = warp / SPLIT;
    const int rel = (blockIdx.y * kCols + cg) * 32 + lane;  // element within the chunk
    const int tot = (int)(ch.row1 - ch.row0) * R;
    bool act = rel < tot;
    const int r = act ? rel % R : 0;
    if (skip && act) act = skip[ch.cfg * R + r] != skipval;
    const long long e = ch.row0 * R + rel;
    B ax[2] = {B(0), B(0)}, ay[2] = {B(0), B(0)};
    if (__any_sync(0xffffffffu, act)) {
        const V* vp = Vb + (act ? e : ch.row0 * R);
        const V* hp = hT + (long long)ch.cfg * ldh * R + r;
        for (int i0 = sp * U; i0 < nv; i0 += SPLIT * U) {
            V vv[U], hh[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = min(i0 + u, nv - 1);
                vv[u] = vp[(long long)i * vstride];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u;
                hh[u] = i < nv ? hp[(long long)i * R] : V{A(0), A(0)};
            }
            A bx[2] = {A(0), A(0)}, by[2] = {A(0), A(0)};
#pragma unroll
            for (int u = 0; u < U; ++u) {
                bx[u & 1] = fma(vv[u].x, hh[u].x, fma(-vv[u].y, hh[u].y, bx[u & 1]));
                by[u & 1] = fma(vv[u].x, hh[u].y, fma(vv[u].y, hh[u].x, by[u & 1]));
            }
            ax[0] += (B)bx[0];
            ax[1] += (B)bx[1];
            ay[0] += (B)by[0];
            ay[1] += (B)by[1];
        }
    }
    red[cg][sp][lane] = W{ax[0] + ax[1], ay[0] + ay[1]};
    if (SPLIT > 1) __syncthreads();
    if (sp != 0 || !act) return;
    W d = red[cg][0][lane];
#pragma unroll
    for (int k = 1; k < SPLIT; ++k) {
        d.x += red[cg][k][lane].x;
        d.y += red[cg][k][lane].y;
    }
    const W o = w[e];
    const B sg = (B)sign;
    w[e] = W{o.x + sg * d.x, o.y + sg * d.y};
}

// The same for an FP32 basis and 16-byte loads, two neighbouring elements per
// lane (two columns of a row, or two rows when R = 1), as in k_dots_pair.
template <typename W, int SPLIT>
__global__ void __launch_bounds__(kThreads, 2)
    k_update_pair(const RowChunk* __restrict__ chunks, int R, const float2* __restrict__ Vb, long long vstride, int nv,
                  const float2* __restrict__ hT, long long ldh, const int* __restrict__ skip, int skipval, double sign,
                  W* __restrict__ w) {
    typedef decltype(W{}.x) B;
    struct Pair {
        B x, y, z, w;
    };
    constexpr int U = 8;
    constexpr int kCols = kWarps / SPLIT;
    __shared__ Pair red[kCols][SPLIT][32];
    const RowChunk ch = chunks[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sp = warp % SPLIT, cg = warp / SPLIT;
    const int rel = ((blockIdx.y * kCols + cg) * 32 + lane) * 2;
    const int tot = (int)(ch.row1 - ch.row0) * R;
    const bool one = R == 1;
    const int r = rel < tot ? rel % R : 0;
    bool act0 = rel < tot, act1 = rel + 1 < tot;
    if (skip && act0) act0 = skip[ch.cfg * R + r] != skipval;
    if (skip && act1) act1 = one ? act0 : skip[ch.cfg * R + r + 1] != skipval;
    const long long e = ch.row0 * R + rel;
    Pair acc{B(0), B(0), B(0), B(0)};
    if (__any_sync(0xffffffffu, act0 || act1)) {
        const float2* vp = Vb + (rel < tot ? e : ch.row0 * R);
        const float2* hp = hT + (long long)ch.cfg * ldh * R + r;
        for (int i0 = sp * U; i0 < nv; i0 += SPLIT * U) {
            float4 vv[U], hh[U];
#pragma unroll
            for (int u = 0; u < U; ++u) vv[u] = *(const float4*)(vp + (long long)min(i0 + u, nv - 1) * vstride);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = min(i0 + u, nv - 1);
                if (one) {
                    const float2 h = hp[i];
                    hh[u] = make_float4(h.x, h.y, h.x, h.y);
                } else {
                    hh[u] = *(const float4*)(hp + (long long)i * R);
                }
                if (i0 + u >= nv) hh[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                b.x = fmaf(vv[u].x, hh[u].x, fmaf(-vv[u].y, hh[u].y, b.x));
                b.y = fmaf(vv[u].x, hh[u].y, fmaf(vv[u].y, hh[u].x, b.y));
                b.z = fmaf(vv[u].z, hh[u].z, fmaf(-vv[u].w, hh[u].w, b.z));
                b.w = fmaf(vv[u].z, hh[u].w, fmaf(vv[u].w, hh[u].z, b.w));
            }
            acc.x += (B)b.x;
            acc.y += (B)b.y;
            acc.z += (B)b.z;
            acc.w += (B)b.w;
        }
    }
    if (SPLIT > 1) {
        red[cg][sp][lane] = acc;
        __syncthreads();
        if (sp != 0) return;
#pragma unroll
        for (int k = 1; k < SPLIT; ++k) {
            const Pair o = red[cg][k][lane];
            acc.x += o.x;
            acc.y += o.y;
            acc.z += o.z;
            acc.w += o.w;
        }
    }
    const B sg = (B)sign;
    if (act0) {
        const W o = w[e];
        w[e] = W{o.x + sg * acc.x, o.y + sg * acc.y};
    }
    if (act1) {
        const W o = w[e + 1];
        w[e + 1] = W{o.x + sg * acc.z, o.y + sg * acc.w};
    }
}

// v = w * scale[s] for active systems, 0 otherwise; with xs (FP32 basis),
// also xs = rf .* v, the scaled columns the next product reads (the
// arithmetic of k_scale_cols on the stored v).
template <typename Vin, typename Vout>
__global__ void k_scale(const RowChunk* __restrict__ chunks, int R, const Vin* __restrict__ w,
                        const double* __restrict__ scale, const int* __restrict__ active,
                        Vout* __restrict__ v, const float* __restrict__ rf, float2* __restrict__ xs) {
    const RowChunk ch = chunks[blockIdx.x];
    // arithmetic in the wider of the two storage types (FP32 for an FP32 basis)
    typedef decltype(Vin{}.x + Vout{}.x) A;
    const int tot = (int)(ch.row1 - ch.row0) * R;
    const long long e0 = ch.row0 * R;
    for (int rel = blockIdx.y * blockDim.x + threadIdx.x; rel < tot; rel += gridDim.y * blockDim.x) {
        const int r = rel % R, s = ch.cfg * R + r;
        const A f = (A)(active[s] ? scale[s] : 0.0);
        const Vin a = w[e0 + rel];
        const Vout o = Vout{(decltype(Vout{}.x))((A)a.x * f), (decltype(Vout{}.x))((A)a.y * f)};
        v[e0 + rel] = o;
        if (xs) {
            const float c = rf[ch.row0 + rel / R];
            xs[e0 + rel] = make_float2(c * (float)o.x, c * (float)o.y);
        }
    }
}

// Selective re-orthogonalisation flags, one CTA per system: ||w'||^2 after
// the first projection is ||w||^2 - sum_i |h_i|^2 (Pythagoras, V orthonormal);
// need[s] = 1 for an active system where that is below ||w||^2 / 2.  The
// estimate is written to wn2 (the subdiagonal when no second pass runs);
// where cancellation makes it inaccurate the second pass runs and measures
// the norm itself.
__global__ void k_reorth_flags(int S, const double2* __restrict__ h1, int hstride, int j,
                               double2* __restrict__ wn2, const int* __restrict__ active,
                               int* __restrict__ skip2, double eta2) {
    const int s = blockIdx.x;
    const double2* h = h1 + (long long)s * hstride;
    double acc = 0.0;
    for (int i = threadIdx.x; i <= j; i += blockDim.x) acc += cabs2(h[i]);
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    __shared__ double part[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) part[warp] = acc;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double ss = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) ss += part[k];
    const double before = h[j + 1].x;  // ||w||^2 before the projection
    const double after = before - ss;
    wn2[(long long)s * hstride] = make_double2(after, 0.0);
    skip2[s] = !(active[s] && after < eta2 * before);
}

// ||w'||^2 after the second projection of every system with skip2 == 0, one CTA
// each: ||w1||^2 - |h2|^2 from the sums of that projection (h2[j + 1] holds
// ||w1||^2) while at least half is left, where the difference is as exact as the
// norm itself; else, as near a breakdown, measured on w.
template <typename V>
__global__ void __launch_bounds__(128) k_second_norm(const RowChunk* __restrict__ chunks,
                                                     const int* __restrict__ cfg_chunk_off, int R,
                                                     const double2* __restrict__ h2, int hstride, int j,
                                                     const int* __restrict__ skip2, const V* __restrict__ w,
                                                     double2* __restrict__ wn2) {
    __shared__ double red[4];
    const int s = blockIdx.x, c = s / R, r = s % R;
    if (skip2[s]) return;
    auto cta_sum = [&](double v) {
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
        __syncthreads();
        return red[0] + red[1] + red[2] + red[3];
    };
    const double2* h = h2 + (long long)s * hstride;
    double acc = 0.0;
    for (int i = threadIdx.x; i <= j; i += blockDim.x) acc += cabs2(h[i]);
    const double before = h[j + 1].x;
    double after = before - cta_sum(acc);
    if (!(after >= 0.5 * before)) {
        acc = 0.0;
        const long long r1 = chunks[cfg_chunk_off[c + 1] - 1].row1;
        for (long long row = chunks[cfg_chunk_off[c]].row0 + threadIdx.x; row < r1; row += blockDim.x)
            acc += cabs2(to_d2(w[row * R + r]));
        after = cta_sum(acc);
    }
    if (threadIdx.x == 0) wn2[(long long)s * hstride] = make_double2(after, 0.0);
}

// Start of a cycle: beta = ||r||; systems whose residual already meets
// tol_abs are done.  g = [beta, 0, ...], scale = 1/beta.
__global__ void k_start(int S, int m, const double2* __restrict__ rr, int hstride,
                        const double* __restrict__ tol_abs, double* __restrict__ beta_out,
                        double* __restrict__ vscale, double2* __restrict__ g, int* __restrict__ active,
                        int* __restrict__ kconv, int* __restrict__ any_active) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const double beta = sqrt(fmax(rr[(long long)s * hstride].x, 0.0));
    beta_out[s] = beta;
    kconv[s] = 0;
    const int act = (beta > tol_abs[s]) && isfinite(beta);
    active[s] = act;
    vscale[s] = act ? 1.0 / beta : 0.0;
    double2* gs = g + (long long)s * (m + 1);
    gs[0] = make_double2(act ? beta : 0.0, 0.0);
    for (int i = 1; i <= m; ++i) gs[i] = make_double2(0.0, 0.0);
    if (act) atomicOr(any_active, 1);
}

// affine map z -> A z + B (complex); compose(second, first) = second o first
struct Aff {
    double2 A, B;
};
__device__ __forceinline__ Aff compose(const Aff& second, const Aff& first) {
    return Aff{cmul(second.A, first.A), cadd(cmul(second.A, first.B), second.B)};
}
// the same maps in FP32 (z_j of the FP32 inner sweeps of a mixed solve)
struct AffF {
    float2 A, B;
};
__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ AffF compose(const AffF& second, const AffF& first) {
    const float2 ab = cmulf(second.A, first.B);
    return AffF{cmulf(second.A, first.A), make_float2(ab.x + second.B.x, ab.y + second.B.y)};
}
template <typename M> struct AffOps;
template <> struct AffOps<Aff> {
    __device__ static Aff id() { return Aff{make_double2(1.0, 0.0), make_double2(0.0, 0.0)}; }
    __device__ static Aff step(double2 c, double2 sv, double2 hn1) {
        return Aff{cscale(cconj(sv), -1.0), cscale(hn1, c.x)};
    }
    __device__ static double2 apply(const Aff& f, double2 z) { return cadd(cmul(f.A, z), f.B); }
};
template <> struct AffOps<AffF> {
    __device__ static AffF id() { return AffF{make_float2(1.f, 0.f), make_float2(0.f, 0.f)}; }
    __device__ static AffF step(double2 c, double2 sv, double2 hn1) {
        return AffF{make_float2((float)-sv.x, (float)sv.y), make_float2((float)(hn1.x * c.x), (float)(hn1.y * c.x))};
    }
    __device__ static double2 apply(const AffF& f, double2 z) {
        const float2 r = cmulf(f.A, make_float2((float)z.x, (float)z.y));
        return make_double2((double)r.x + f.B.x, (double)r.y + f.B.y);
    }
};

// Arnoldi step j for one system per CTA: column h = h1 + h2 (h2 only where
// the second projection ran), h[j+1] = ||w||.  The step needs only the last
// entry z_j of the rotated column (for the new rotation and the residual
// estimate): z_j = A_{j-1}(...A_0(h_0)) with A_i(z) = c_i h_{i+1} -
// conj(s_i) z, an ordered reduction of affine maps over the CTA, in FP64
// (Map = Aff) or, for the FP32 inner sweeps of a mixed solve, in FP32 (Map =
// AffF: a warp-wide FP64 instruction costs ~64 cycles of an SM sub-partition
// on this GPU, and the chain made the step ~20 us).  The rotation itself is
// formed in FP64.  The raw column is stored; k_apply_rotations rotates all
// columns at the end of the cycle in FP64, in parallel across columns.
// Warp-shuffle transfer of the maps (lane + off -> lane).
__device__ __forceinline__ Aff shfl_down(const Aff& f, int off) {
    return Aff{make_double2(__shfl_down_sync(0xffffffffu, f.A.x, off), __shfl_down_sync(0xffffffffu, f.A.y, off)),
               make_double2(__shfl_down_sync(0xffffffffu, f.B.x, off), __shfl_down_sync(0xffffffffu, f.B.y, off))};
}
__device__ __forceinline__ AffF shfl_down(const AffF& f, int off) {
    return AffF{make_float2(__shfl_down_sync(0xffffffffu, f.A.x, off), __shfl_down_sync(0xffffffffu, f.A.y, off)),
                make_float2(__shfl_down_sync(0xffffffffu, f.B.x, off), __shfl_down_sync(0xffffffffu, f.B.y, off))};
}
// Ordered reduction over the 32 lanes of a warp: lane 0 receives
// f_31 o ... o f_1 o f_0 (later lanes compose onto earlier ones).
template <typename Map>
__device__ __forceinline__ Map warp_compose(Map f) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off *= 2) {
        const Map later = shfl_down(f, off);
        if ((lane & (2 * off - 1)) == 0) f = compose(later, f);
    }
    return f;
}

constexpr int kGivensThreads = 1024;

template <typename Map>
__global__ void __launch_bounds__(kGivensThreads) k_givens(int m, int j, const double2* __restrict__ h1,
                                                     const double2* __restrict__ h2, int hstride,
                                                     const double2* __restrict__ wn2a,
                                                     const double2* __restrict__ wn2b,
                                                     const int* __restrict__ skip2,
                                                     const double* __restrict__ tol_cycle,
                                                     double2* __restrict__ H, double2* __restrict__ cs,
                                                     double2* __restrict__ sn, double2* __restrict__ g,
                                                     double* __restrict__ vscale, int* __restrict__ active,
                                                     int* __restrict__ kconv, int* __restrict__ iters,
                                                     int* __restrict__ any_active, int* __restrict__ nonfinite,
                                                     double2* __restrict__ rdiag) {
    const int s = blockIdx.x;
    if (!active[s]) return;
    __shared__ Map red[kGivensThreads / 32];
    const int tid = threadIdx.x, T = blockDim.x;
    const bool second = !skip2[s];
    const double2* a = h1 + (long long)s * hstride;
    const double2* b = h2 + (long long)s * hstride;
    const double2* csj = cs + (long long)s * m;
    const double2* snj = sn + (long long)s * m;
    double2* Hc = H + ((long long)s * m + j) * (m + 1);  // column j, rows 0..j+1
    auto hval = [&](int i) {
        double2 v = a[i];
        if (second) v = cadd(v, b[i]);
        return v;
    };
    // operands of the tail, loaded before the reduction so that their
    // latency overlaps it (thread 0 finishes the step)
    double wn = 0.0, tol = 0.0;
    double2 h0 = make_double2(0.0, 0.0), gj = make_double2(0.0, 0.0);
    if (tid == 0) {
        wn = second ? wn2b[(long long)s * hstride].x : wn2a[(long long)s * hstride].x;
        tol = tol_cycle[s];
        h0 = hval(0);
        gj = g[(long long)s * (m + 1) + j];
    }
    for (int i = tid; i <= j; i += T) Hc[i] = hval(i);  // raw column
    // segment of rotations [lo, hi) owned by this thread
    const int per = (j + T - 1) / T;
    const int lo = min(j, tid * per), hi = min(j, lo + per);
    Map seg = AffOps<Map>::id();
    for (int i = lo; i < hi; ++i) seg = compose(AffOps<Map>::step(csj[i], snj[i], hval(i + 1)), seg);
    // ordered reduction: within each warp by shuffles, then over the warps
    seg = warp_compose(seg);
    const int nw = T >> 5;
    if ((tid & 31) == 0) red[tid >> 5] = seg;
    __syncthreads();
    if (tid >= 32) return;
    seg = tid < nw ? red[tid] : AffOps<Map>::id();
    seg = warp_compose(seg);
    if (tid != 0) return;
    const double2 hjj = AffOps<Map>::apply(seg, h0);
    // rotation c = |hjj| / den, s = (hjj / |hjj|) hn / den, den^2 = |hjj|^2 + hn^2,
    // from reciprocal square roots (the FP64 pipe of this GPU is narrow, and
    // this chain runs on one thread): 1/|hjj|, 1/den, 1/hn
    wn = fmax(wn, 0.0);
    const double a2 = cabs2(hjj);
    const double rw = wn > 0.0 ? rsqrt(wn) : 0.0;
    const double hn = wn * rw;
    double2 c, sv;
    if (a2 + wn == 0.0) {
        c = make_double2(1.0, 0.0);
        sv = make_double2(0.0, 0.0);
    } else if (a2 == 0.0) {
        c = make_double2(0.0, 0.0);
        sv = make_double2(1.0, 0.0);  // hn real and positive
    } else {
        const double ra = rsqrt(a2), rd = rsqrt(a2 + wn);
        c = make_double2(a2 * ra * rd, 0.0);
        sv = cscale(hjj, hn * ra * rd);  // ph * conj(hn) / den, hn real
    }
    cs[(long long)s * m + j] = c;
    sn[(long long)s * m + j] = sv;
    const double2 rjj = cadd(cscale(hjj, c.x), cscale(sv, hn));
    rdiag[(long long)s * m + j] = make_double2(hn, 0.0);  // R_jj is formed in FP64 at the end of the cycle
    double2* gs = g + (long long)s * (m + 1);
    const double2 gn = cscale(cmul(cconj(sv), gj), -1.0);
    gs[j + 1] = gn;
    gs[j] = cscale(gj, c.x);
    iters[s] += 1;
    const double res2 = cabs2(gn);  // squared residual estimate
    const bool bad = !isfinite(res2) || !isfinite(rjj.x) || !isfinite(rjj.y);
    if (bad) *nonfinite = 1;  // every writer stores the same value (the flag may live in host memory)
    if (bad || res2 <= tol * tol || hn == 0.0 || j + 1 == m) {
        active[s] = 0;
        kconv[s] = j + 1;
        vscale[s] = 0.0;
    } else {
        vscale[s] = rw;
        *any_active = 1;
    }
}

// End of a cycle: rotate every stored column j < kconv (raw h_0..h_j) by the
// rotations 0..j-1 into the triangle R, in FP64, and form R_jj from the
// rotated z_j with rotation j and the stored subdiagonal ||w_j||; one thread
// per column, all columns and systems in parallel.
__global__ void k_apply_rotations(int m, double2* __restrict__ H, const double2* __restrict__ cs,
                                  const double2* __restrict__ sn, const double2* __restrict__ rdiag,
                                  const int* __restrict__ kconv) {
    const int s = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kconv[s]) return;
    double2* Hc = H + ((long long)s * m + j) * (m + 1);
    const double2* csj = cs + (long long)s * m;
    const double2* snj = sn + (long long)s * m;
    double2 z = Hc[0];
    for (int i = 0; i < j; ++i) {
        const double2 c = csj[i], sv = snj[i], hn1 = Hc[i + 1];
        Hc[i] = cadd(cscale(z, c.x), cmul(sv, hn1));
        z = csub(cscale(hn1, c.x), cmul(cconj(sv), z));
    }
    // R_jj = c_j z_j + s_j ||w_j|| (the subdiagonal entry, real)
    Hc[j] = cadd(cscale(z, csj[j].x), cscale(snj[j], rdiag[(long long)s * m + j].x));
    Hc[j + 1] = make_double2(0.0, 0.0);
}

// Back substitution H y = g on the leading kconv x kconv triangle, one CTA
// per system: column-oriented, the CTA updates the remaining right-hand
// side in parallel after each pivot.
__global__ void __launch_bounds__(kThreads) k_lsq(int m, const double2* __restrict__ H,
                                                  const double2* __restrict__ g, const int* __restrict__ kconv,
                                                  double2* __restrict__ y, double2* __restrict__ work) {
    const int s = blockIdx.x;
    const int k = kconv[s];
    double2* ys = y + (long long)s * m;
    // the x update sweeps every column of the cycle: zero what this system did not use
    for (int i = k + threadIdx.x; i < m; i += blockDim.x) ys[i] = make_double2(0.0, 0.0);
    if (k == 0) return;
    const double2* Hs = H + (long long)s * m * (m + 1);
    double2* rhs = work + (long long)s * (m + 1);
    for (int i = threadIdx.x; i < k; i += blockDim.x) rhs[i] = g[(long long)s * (m + 1) + i];
    __shared__ double2 yi_sh;
    __syncthreads();
    for (int i = k - 1; i >= 0; --i) {
        if (threadIdx.x == 0) {
            const double2 d = Hs[(long long)i * (m + 1) + i];
            const double2 v = (d.x == 0.0 && d.y == 0.0) ? make_double2(0.0, 0.0) : cdiv(rhs[i], d);
            ys[i] = v;
            yi_sh = v;
        }
        __syncthreads();
        const double2 v = yi_sh;
        const double2* col = Hs + (long long)i * (m + 1);
        for (int t = threadIdx.x; t < i; t += blockDim.x) rhs[t] = csub(rhs[t], cmul(col[t], v));
        __syncthreads();
    }
}

__global__ void k_residual(long long n, const double2* __restrict__ b, const double2* __restrict__ Ax,
                           double2* __restrict__ r) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = csub(b[i], Ax[i]);
}

__global__ void k_zero(long long n, double2* __restrict__ x) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = make_double2(0.0, 0.0);
}

inline unsigned blocks_for(long long n, int th) { return (unsigned)((n + th - 1) / th); }

}  // namespace

// ---------------------------------------------------------------- host wrappers

template <typename V>
bool gm_dots(const GmresDims& d, const RowChunk* chunks, const int* cfg_chunk_off, const V* Vb, long long vstride,
             int nv, int self, const V* w, const int* skip, double2* part, double2* out, int ostride, V* hT,
             cudaStream_t s, int skipval, const GmDotsFuse* fuse) {
    const int nvv = nv + self;
    const unsigned zg = (unsigned)((d.R + 31) / 32);
    const long long warps = (long long)d.nchunk * zg * nvv;  // with one vector each
    // several vectors per warp (more loads in flight and fewer reads of w: two
    // instead of four FP32 vectors took twice as long on 400 disks), one while
    // there are few
    const bool few = warps < 152 * 16;
    const int per = kWarps * (few ? 1 : sizeof(V) == 8 ? 4 : 2);
    const dim3 grid(d.nchunk, (nvv + per - 1) / per, zg);
    if (few) {
        k_dots<V, 1><<<grid, kThreads, 0, s>>>(chunks, d.R, Vb, vstride, nv, self, w, skip, skipval, part);
    } else if constexpr (sizeof(V) == 8) {
        if (d.pairs)
            k_dots_pair<4><<<grid, kThreads, 0, s>>>(chunks, d.R, Vb, vstride, nv, self, w, skip, skipval, part);
        else
            k_dots<V, 4><<<grid, kThreads, 0, s>>>(chunks, d.R, Vb, vstride, nv, self, w, skip, skipval, part);
    } else {
        k_dots<V, 2><<<grid, kThreads, 0, s>>>(chunks, d.R, Vb, vstride, nv, self, w, skip, skipval, part);
    }
    FinTail tail;
    const bool tail_done = fuse && fuse->wn2 && d.S <= kFuseMaxSystems;
    if (tail_done) {
        tail.cnt = fuse->cnt;
        tail.S = d.S;
        tail.j = fuse->j;
        tail.wn2 = fuse->wn2;
        tail.active = fuse->active;
        tail.skip2 = fuse->skip2;
        tail.eta2 = fuse->eta2;
    }
    k_dots_fin<V><<<dim3((unsigned)(((long long)nvv * d.R + 31) / 32), d.C), 32 * kFinY, 0, s>>>(
        d.R, nvv, cfg_chunk_off, part, out, ostride, hT, d.ldh, tail);
    g_msd_launches += 2;
    return tail_done;
}

template <typename V>
void gm_coeffs(const GmresDims& d, int nv, const double2* y, int ystride, V* hT, cudaStream_t s) {
    if (nv <= 0) return;
    k_coeffs<V><<<blocks_for((long long)d.C * nv * d.R, 256), 256, 0, s>>>(d.C, d.R, nv, y, ystride, hT, d.ldh);
    g_msd_launches += 1;
}

// SPLIT: enough warps for the chip (32 per SM) where the elements alone do
// not give them, but at least one batch of vectors per warp.  FP32 bases of
// more than 9 728 elements take pairs (400 disks, one column: the mixed solve
// 431 -> 404 ms with eight warps a pair group against single elements).  That
// first step of the pairs' ladder is measured; its later ones, and the ladder of
// single elements, follow the count of warps alone.
template <typename V, typename W>
void gm_update(const GmresDims& d, const RowChunk* chunks, const V* Vb, long long vstride, int nv, const V* hT,
               const int* skip, double sign, W* w, cudaStream_t s, int skipval) {
    if (nv <= 0) return;
    constexpr int U = 8;
    const long long cols = d.Ntot * d.R / 32 + 1;
    const int most = std::max(1, nv / U);
    if constexpr (sizeof(V) == 8) {
        if (d.pairs && cols >= 152 * 2) {
            auto go = [&](auto split) {
                constexpr int SP = decltype(split)::value;
                const int per = kWarps / SP * 64;
                k_update_pair<W, SP><<<dim3(d.nchunk, (d.chunk_elems + per - 1) / per), kThreads, 0, s>>>(
                    chunks, d.R, Vb, vstride, nv, hT, d.ldh, skip, skipval, sign, w);
            };
            if (cols <= 152 * 8 && nv >= 64) go(std::integral_constant<int, 8>());
            else if (cols <= 152 * 32 && nv >= 32) go(std::integral_constant<int, 4>());
            else if (cols / 2 <= 152 * 32 && nv >= 16) go(std::integral_constant<int, 2>());
            else go(std::integral_constant<int, 1>());
            g_msd_launches += 1;
            return;
        }
    }
    auto go = [&](auto split) {
        constexpr int SP = decltype(split)::value;
        const int per = kWarps / SP * 32;
        k_update<V, W, SP><<<dim3(d.nchunk, (d.chunk_elems + per - 1) / per), kThreads, 0, s>>>(
            chunks, d.R, Vb, vstride, nv, hT, d.ldh, skip, skipval, sign, w);
    };
    if (cols * 4 <= 152 * 32 && most >= 4) go(std::integral_constant<int, 8>());
    else if (cols * 2 <= 152 * 32 && most >= 2) go(std::integral_constant<int, 4>());
    else if (cols <= 152 * 32 && most >= 2) go(std::integral_constant<int, 2>());
    else go(std::integral_constant<int, 1>());
    g_msd_launches += 1;
}

template <typename Vin, typename Vout>
void gm_scale(const GmresDims& d, const RowChunk* chunks, const Vin* w, const double* scale, const int* active,
              Vout* v, cudaStream_t s, const float* rf, float2* xs) {
    k_scale<Vin, Vout><<<dim3(d.nchunk, (d.chunk_elems + kThreads - 1) / kThreads), kThreads, 0, s>>>(chunks, d.R, w, scale, active,
                                                                                         v, rf, xs);
    g_msd_launches += 1;
}

template <typename V>
void gm_second_norm(const GmresDims& d, const RowChunk* chunks, const int* cfg_chunk_off, const double2* h2,
                    int hstride, int j, const int* skip2, const V* w, double2* wn2, cudaStream_t s) {
    k_second_norm<V><<<d.S, 128, 0, s>>>(chunks, cfg_chunk_off, d.R, h2, hstride, j, skip2, w, wn2);
    g_msd_launches += 1;
}

void gm_reorth_flags(const GmresDims& d, const double2* h1, int hstride, int j, double2* wn2,
                     const int* active, int* skip2, cudaStream_t s, double eta2) {
    k_reorth_flags<<<d.S, 128, 0, s>>>(d.S, h1, hstride, j, wn2, active, skip2, eta2);
    g_msd_launches += 1;
}

void gm_start(const GmresDims& d, const double2* rr, int hstride, const double* tol_abs, double* beta,
              double* vscale, double2* g, int* active, int* kconv, int* any_active, cudaStream_t s) {
    k_start<<<blocks_for(d.S, 128), 128, 0, s>>>(d.S, d.m, rr, hstride, tol_abs, beta, vscale, g, active, kconv,
                                                 any_active);
    g_msd_launches += 1;
}

// Threads of the Givens step: about two rotations per thread, whole warps.
static int givens_threads(int j) {
    const int t = ((j + 1) / 2 + 31) / 32 * 32;
    return std::min(kGivensThreads, std::max(32, t));
}

void gm_givens(const GmresDims& d, int j, const double2* h1, const double2* h2, int hstride, const double2* wn2a,
               const double2* wn2b, const int* skip2, const double* tol_cycle, double2* H, double2* cs,
               double2* sn, double2* g, double* vscale, int* active, int* kconv, int* iters, int* any_active,
               int* nonfinite, double2* rdiag, bool fp32_maps, cudaStream_t s) {
    if (fp32_maps)
        k_givens<AffF><<<d.S, givens_threads(j), 0, s>>>(d.m, j, h1, h2, hstride, wn2a, wn2b, skip2, tol_cycle, H,
                                                         cs, sn, g, vscale, active, kconv, iters, any_active,
                                                         nonfinite, rdiag);
    else
        k_givens<Aff><<<d.S, givens_threads(j), 0, s>>>(d.m, j, h1, h2, hstride, wn2a, wn2b, skip2, tol_cycle, H,
                                                        cs, sn, g, vscale, active, kconv, iters, any_active,
                                                        nonfinite, rdiag);
    g_msd_launches += 1;
}

void gm_lsq(const GmresDims& d, double2* H, const double2* cs, const double2* sn, const double2* rdiag,
            const double2* g, const int* kconv, double2* y, double2* work, cudaStream_t s) {
    k_apply_rotations<<<dim3(blocks_for(d.m, 128), d.S), 128, 0, s>>>(d.m, H, cs, sn, rdiag, kconv);
    k_lsq<<<d.S, kThreads, 0, s>>>(d.m, H, g, kconv, y, work);
    g_msd_launches += 2;
}

void gm_residual(long long n, const double2* b, const double2* Ax, double2* r, cudaStream_t s) {
    k_residual<<<blocks_for(n, 256), 256, 0, s>>>(n, b, Ax, r);
    g_msd_launches += 1;
}

void gm_zero(long long n, double2* x, cudaStream_t s) {
    k_zero<<<blocks_for(n, 256), 256, 0, s>>>(n, x);
    g_msd_launches += 1;
}

template bool gm_dots<double2>(const GmresDims&, const RowChunk*, const int*, const double2*, long long, int, int,
                               const double2*, const int*, double2*, double2*, int, double2*, cudaStream_t, int,
                               const GmDotsFuse*);
template bool gm_dots<float2>(const GmresDims&, const RowChunk*, const int*, const float2*, long long, int, int,
                              const float2*, const int*, double2*, double2*, int, float2*, cudaStream_t, int,
                              const GmDotsFuse*);
template void gm_second_norm<double2>(const GmresDims&, const RowChunk*, const int*, const double2*, int, int,
                                      const int*, const double2*, double2*, cudaStream_t);
template void gm_second_norm<float2>(const GmresDims&, const RowChunk*, const int*, const double2*, int, int,
                                     const int*, const float2*, double2*, cudaStream_t);
template void gm_coeffs<double2>(const GmresDims&, int, const double2*, int, double2*, cudaStream_t);
template void gm_coeffs<float2>(const GmresDims&, int, const double2*, int, float2*, cudaStream_t);
template void gm_update<double2, double2>(const GmresDims&, const RowChunk*, const double2*, long long, int,
                                          const double2*, const int*, double, double2*, cudaStream_t, int);
template void gm_update<float2, float2>(const GmresDims&, const RowChunk*, const float2*, long long, int,
                                        const float2*, const int*, double, float2*, cudaStream_t, int);
template void gm_update<float2, double2>(const GmresDims&, const RowChunk*, const float2*, long long, int,
                                         const float2*, const int*, double, double2*, cudaStream_t, int);
template void gm_scale<double2, double2>(const GmresDims&, const RowChunk*, const double2*, const double*,
                                         const int*, double2*, cudaStream_t, const float*, float2*);
template void gm_scale<double2, float2>(const GmresDims&, const RowChunk*, const double2*, const double*,
                                        const int*, float2*, cudaStream_t, const float*, float2*);
template void gm_scale<float2, float2>(const GmresDims&, const RowChunk*, const float2*, const double*, const int*,
                                       float2*, cudaStream_t, const float*, float2*);
