// Householder QR of a tall panel (m x nb, column-major, real or complex), the
// step of full -> band (Sec. 2, two-stage reduction) that forms a chain: nb
// reflectors, each needing sums over all rows of the one before.
//
// The panel stays in registers from its load to its only store: its rows are
// dealt in runs of CH = LPC * RPT to the blocks, and in a block LPC threads
// hold one column, RPT rows each.  Per column i
//   1. the column's threads put its rows below i, x, into shared memory;
//   2. every column j >= i forms its partial sum of conj(x) a_j (j = i: the
//      squared norm) and the partials are exchanged once; row i goes along;
//   3. every block derives tau, the scale and beta from them, and updates
//      a_j -= x (scale w_j), w_j = conj(tau) (a_ij + conj(scale) sum_j), which is
//      H(i)^H applied with v = [1; scale x].
// One exchange per column, against two grid-wide barriers and four passes
// over the panel in L2 for a form with separate norm, dot and update phases.
//
// The exchange: blocks of one cluster (up to 16) write their partials into
// each other's shared memory and arrive on each other's mbarriers; taller
// panels use a cooperative grid, partials in global memory and one counter.
//
// What bounds it: FP64 issue (2 multiply-adds per clock and SM: about
// m nb^2 / (2 blocks) clocks a panel) and the exchange's latency.
// Measured on a GB300: a 992 x 32 panel takes 0.14 ms (4.4 us a column), a
// complex 960 x 64 one 1.0 ms; the forms before (two launches or grid barriers
// per column) took about 35 us a column.  full -> band of n = 1024, nbw = 32:
// 37.7 -> 22.8 ms, n = 8192, nbw = 64: 467 -> 312 ms.
//
// On exit the panel holds R on and above the diagonal and v below it (LAPACK
// layout, v_0 = 1 implicit), tau the nb scalars, and Y (if given) the explicit
// unit lower trapezoidal reflectors.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "elpa_gb300.h"
#include "reduction.cuh"

namespace gb {

namespace cg = cooperative_groups;

namespace {

constexpr long long kPanelWaitNs = 10LL * 1000 * 1000 * 1000;
constexpr int kClusterMax = 16;

template <class T, int NB, int CH>
struct PanelShared {
    T x[2][CH];
    T ms[2][kClusterMax][NB];   // cluster exchange: partial sums by rank
    T ma[2][NB];                // row i
    T tau[2], scal[2];
    double beta[2];
    unsigned long long bar[2];
    int gave_up;
};

// Exchange area of the grid form, in global memory.
template <class T, int NB>
struct PanelGrid {
    unsigned int arrivals;
    unsigned int pad[63];
    T ma[2][NB];
    T ms[1];                    // [2][blocks][NB]
};

// How a panel's waits end: their limit, the status word that receives
// GB_ERR_TIMEOUT (or null) and, for tests, the column at which block 0 does not
// arrive (-1: none).
struct PanelWait {
    long long ns = kPanelWaitNs;
    int *status = nullptr;
    int hold = -1;
};

template <class T, int NB, int LPC, int RPT, bool GRID>
__global__ void __launch_bounds__(NB *LPC, 1)
panel_qr_kernel(int m, int nb, T *__restrict__ P, long long lda, T *__restrict__ tau_out, T *__restrict__ Y,
                long long ldy, PanelGrid<T, NB> *gx, PanelWait pw)
{
    constexpr int CH = LPC * RPT;
    __shared__ PanelShared<T, NB, CH> sm;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int col = tid / LPC, part = tid % LPC;
    const int blocks = (int)gridDim.x, rank = (int)blockIdx.x;   // one cluster, or the whole grid
    const int r0 = rank * CH;
    cg::cluster_group cluster = cg::this_cluster();

    T a[RPT];
#pragma unroll
    for (int t = 0; t < RPT; t++) {
        const int r = r0 + part + LPC * t;
        zero_of(a[t]);
        if (col < nb && r < m) a[t] = P[(long long)col * lda + r];
    }
    if (tid == 0) {
        sm.gave_up = 0;
        if (!GRID) {
            tc5::mbar_init(tc5::smem_addr(&sm.bar[0]), blocks);
            tc5::mbar_init(tc5::smem_addr(&sm.bar[1]), blocks);
            tc5::mbar_init_fence();
        }
    }
    if (!GRID) cluster.sync();

    const int steps = min(nb, m);
    for (int i = 0; i < steps; i++) {
        const int par = i & 1;
        const bool live = (warp * 32) / LPC + 32 / LPC > i;   // a column of this warp is not done yet
        if (col == i) {
#pragma unroll
            for (int t = 0; t < RPT; t++) {
                T x = a[t];
                if (r0 + part + LPC * t <= i) zero_of(x);
                sm.x[par][part + LPC * t] = x;
            }
        }
        __syncthreads();
        const int il = i - r0;                                   // row i in this block, if it holds it
        const bool owner = il >= 0 && il < CH;
        if (live) {
            constexpr int NA = 8 / LPC;
            T acc[NA];
#pragma unroll
            for (int t = 0; t < NA; t++) zero_of(acc[t]);
#pragma unroll
            for (int t = 0; t < RPT; t++) acc[t % NA] = madc(sm.x[par][part + LPC * t], a[t], acc[t % NA]);
            const T sum = tree_sum<8, LPC>(acc);
            T ai;
            zero_of(ai);
            if (owner) {
                // the entry of row i, from the lane that holds it
#pragma unroll
                for (int t = 0; t < RPT; t++)
                    if (part + LPC * t == il) ai = a[t];
#pragma unroll
                for (int o = LPC / 2; o >= 1; o /= 2) ai = xor_add(ai, o);   // the other lanes hold zero
            }
            if (GRID) {
                if (part == 0) {
                    gx->ms[((size_t)par * blocks + rank) * NB + col] = sum;
                    if (owner) gx->ma[par][col] = ai;
                }
            } else {
                for (int d = part; d < blocks; d += LPC) {
                    cluster.map_shared_rank(&sm.ms[par][rank][col], d)[0] = sum;
                    if (owner) cluster.map_shared_rank(&sm.ma[par][col], d)[0] = ai;
                }
            }
        }
        __syncthreads();
        // a block that gave up neither waits nor arrives any more, so that no
        // other block takes a late arrival for the one it waits for
        const bool arrive = !sm.gave_up && (i != pw.hold || rank != 0);
        if (GRID) {
            if (tid == 0) {
                __threadfence();
                if (arrive)
                    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gx->arrivals) : "memory");
                const unsigned int need = (unsigned int)(i + 1) * (unsigned int)blocks;
                unsigned long long t0 = 0;
                for (long long it = 0; !sm.gave_up; it++) {
                    unsigned int got;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(&gx->arrivals) : "memory");
                    if (got >= need) break;
                    if (it == 0) t0 = now_ns();
                    if ((it & 63) == 63 && (long long)(now_ns() - t0) > pw.ns) sm.gave_up = 1;
                }
            }
            __syncthreads();
        } else {
            if (tid < blocks && arrive) {
                asm volatile("fence.acq_rel.cluster;" ::: "memory");
                mbar_arrive_remote(&sm.bar[par], tid);
            }
            const uint32_t bar = tc5::smem_addr(&sm.bar[par]);
            const uint32_t phase = (uint32_t)(i >> 1) & 1;
            if (!*(volatile int *)&sm.gave_up && !mbar_try_cluster(bar, phase)) {
                const unsigned long long t0 = now_ns();
                for (long long it = 1; !mbar_try_cluster(bar, phase); it++)
                    if ((it & 63) == 0 && (long long)(now_ns() - t0) > pw.ns) {
                        sm.gave_up = 1;
                        break;
                    }
            }
        }
        T sum, ai;
        zero_of(sum);
        zero_of(ai);
        if (live) {
            constexpr int NA = 8 / LPC;
            T acc[NA];
#pragma unroll
            for (int t = 0; t < NA; t++) zero_of(acc[t]);
            // partials of blocks part, part + LPC, ...: the same order for every form
            for (int d = part; d < blocks; d += 8) {
#pragma unroll
                for (int t = 0; t < NA; t++)
                    if (d + LPC * t < blocks)
                        acc[t] = add(acc[t], GRID ? ld_cg(&gx->ms[((size_t)par * blocks + d + LPC * t) * NB + col])
                                                  : sm.ms[par][d + LPC * t][col]);
            }
            sum = tree_sum<8, LPC>(acc);
            ai = GRID ? ld_cg(&gx->ma[par][col]) : sm.ma[par][col];
            if (warp == (i * LPC) / 32) {   // the warp that holds column i
                const int src = (i * LPC) & 31;
                const double ss = __shfl_sync(0xffffffffu, re_of(sum), src);
                const T alpha = lane_of(ai, src);
                const auto h = reflector(alpha, ss);
                if ((tid & 31) == 0) {
                    sm.tau[par] = h.tau;
                    sm.scal[par] = h.scal;
                    sm.beta[par] = h.beta;
                    if (rank == 0) tau_out[i] = h.tau;
                }
            }
        }
        __syncthreads();
        if (live) {
            const T tau = sm.tau[par], scal = sm.scal[par];
            if (col > i) {
                const T w = mul(conj_of(tau), mad(conj_of(scal), sum, ai));
                const T f = mul(scal, w);
#pragma unroll
                for (int t = 0; t < RPT; t++) a[t] = nmad(sm.x[par][part + LPC * t], f, a[t]);
                if (owner) {
#pragma unroll
                    for (int t = 0; t < RPT; t++)
                        if (part + LPC * t == il) a[t] = nmad(w, one_v<T>(), a[t]);
                }
            } else if (col == i) {
                T beta;
                zero_of(beta);
                *(double *)&beta = sm.beta[par];
#pragma unroll
                for (int t = 0; t < RPT; t++) {
                    const int r = r0 + part + LPC * t;
                    if (r > i) a[t] = mul(a[t], scal);
                    else if (r == i) a[t] = beta;
                }
            }
        }
    }
    T nan;
    zero_of(nan);
    *(double *)&nan = __longlong_as_double(0x7ff8000000000000ll);
    // a wait gave up: the result is void and says so, in this block's rows
    // (which no other block writes), in tau and in the status word
    if (sm.gave_up) {
        if (tid < nb) tau_out[tid] = nan;
        if (tid == 0 && pw.status) atomicExch(pw.status, GB_ERR_TIMEOUT);
#pragma unroll
        for (int t = 0; t < RPT; t++) a[t] = nan;
    }
    if (rank == 0 && tid >= steps && tid < nb) zero_of(tau_out[tid]);
#pragma unroll
    for (int t = 0; t < RPT; t++) {
        const int r = r0 + part + LPC * t;
        if (col < nb && r < m) {
            P[(long long)col * lda + r] = a[t];
            if (Y) {
                T y = a[t];
                if (r < col) zero_of(y);
                else if (r == col) one_of(y);
                if (sm.gave_up) y = nan;
                Y[(long long)col * ldy + r] = y;
            }
        }
    }
    if (!GRID) {
        __syncwarp();
        cluster.sync();   // no block leaves while a peer may still reach its shared memory
    }
}

template <class T, int NB, int LPC, int RPT>
cudaError_t launch_cluster(int m, int nb, T *P, long long lda, T *tau, T *Y, long long ldy, const PanelWait &pw,
                           cudaStream_t st)
{
    constexpr int CH = LPC * RPT;
    auto kernel = panel_qr_kernel<T, NB, LPC, RPT, false>;
    const int blocks = (m + CH - 1) / CH;
    int size = 1;
    while (size < blocks) size *= 2;
    cudaError_t e;
    if (size > 8 && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3(NB * LPC);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, m, nb, P, lda, tau, Y, ldy, (PanelGrid<T, NB> *)nullptr, pw);
}

// *done = false (and nothing launched) where the grid does not fit in
// 1 / `share` of the device's co-resident capacity
template <class T, int NB, int LPC, int RPT>
cudaError_t launch_grid(int m, int nb, T *P, long long lda, T *tau, T *Y, long long ldy, void *part, int sms,
                        int share, PanelWait pw, cudaStream_t st, bool *done)
{
    constexpr int CH = LPC * RPT;
    auto kernel = panel_qr_kernel<T, NB, LPC, RPT, true>;
    int blocks = (m + CH - 1) / CH, per_sm = 0;
    *done = false;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, NB * LPC, 0);
    if (e != cudaSuccess) return e;
    if ((long long)blocks * share > (long long)per_sm * sms) return cudaSuccess;
    if ((e = cudaMemsetAsync(part, 0, 256, st)) != cudaSuccess) return e;
    PanelGrid<T, NB> *gx = (PanelGrid<T, NB> *)part;
    void *args[] = {&m, &nb, &P, &lda, &tau, &Y, &ldy, &gx, &pw};
    *done = true;
    return cudaLaunchCooperativeKernel((const void *)kernel, dim3(blocks), dim3(NB * LPC), args, 0, st);
}

template <class T>
cudaError_t panel_qr_t(int m, int nb, T *P, long long lda, T *tau, T *Y, long long ldy, void *part, const PanelWait &pw,
                       cudaStream_t st, bool *done)
{
    constexpr bool Z = sizeof(T) == 16;
    *done = true;
    if (nb <= 32) {
        if (m <= 32 * kClusterMax) return launch_cluster<T, 32, 8, 4>(m, nb, P, lda, tau, Y, ldy, pw, st);
        if (m <= 64 * kClusterMax) return launch_cluster<T, 32, 8, 8>(m, nb, P, lda, tau, Y, ldy, pw, st);
        if (m <= 128 * kClusterMax) return launch_cluster<T, 32, 8, 16>(m, nb, P, lda, tau, Y, ldy, pw, st);
    } else {
        if (m <= 32 * kClusterMax) return launch_cluster<T, 64, 4, 8>(m, nb, P, lda, tau, Y, ldy, pw, st);
        if (m <= 64 * kClusterMax) return launch_cluster<T, 64, 4, 16>(m, nb, P, lda, tau, Y, ldy, pw, st);
        if (!Z && m <= 128 * kClusterMax) return launch_cluster<T, 64, Z ? 4 : 8, 16>(m, nb, P, lda, tau, Y, ldy, pw, st);
    }
    *done = false;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    int dev = 0, sms = 0, coop = 0;
    cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess || cap != cudaStreamCaptureStatusNone) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (!coop) return cudaSuccess;
    // half of the co-resident capacity, so that work on other streams keeps
    // room beside it; the tallest panels (over 9728 rows real, 4864 complex)
    // may take all of it
    if (nb <= 32) {
        e = launch_grid<T, 32, 8, 16>(m, nb, P, lda, tau, Y, ldy, part, sms, 2, pw, st, done);
        if (e != cudaSuccess || *done) return e;
        return launch_grid<T, 32, 8, 16>(m, nb, P, lda, tau, Y, ldy, part, sms, 1, pw, st, done);
    }
    e = launch_grid<T, 64, 4, 16>(m, nb, P, lda, tau, Y, ldy, part, sms, 2, pw, st, done);
    if (e != cudaSuccess || *done) return e;
    return launch_grid<T, 64, 4, Z ? 16 : 32>(m, nb, P, lda, tau, Y, ldy, part, sms, 1, pw, st, done);
}

// T (nb x nb upper triangular) of the block reflector I - Y T Y^H is the
// inverse of the triangle with diagonal 1/tau and the strict upper part of
// G = Y^H Y, so its columns are independent: x_j = tau_j, then for i = j-1 .. 0
// x_i = -tau_i sum_{q > i} G_iq x_q (zero where tau_i is zero).  One block per
// column; its first warp keeps the pending sums of R rows per lane, and each
// x_i found is added into all of them: a chain of nb short steps, where the
// forward recurrence over columns by one block took 50 us for nb = 32 and 501 us
// for nb = 64 complex (now 9 and 41 us).  The other warps stage the next columns of G.
constexpr int kTMax = 256;   // widest block reflector
constexpr int kTCols = 16;   // columns of G staged at a time

// R: rows per lane (32 R >= nb)
template <class T, int R>
__global__ void __launch_bounds__(128) panel_t_kernel(int nb, const T *__restrict__ G, long long ldg,
                                                      const T *__restrict__ tau, T *__restrict__ Tm, long long ldt)
{
    constexpr int LDG = 32 * R;
    extern __shared__ __align__(16) unsigned char dyn[];
    T *Gs = (T *)dyn;                         // two stages of kTCols columns, rows above the diagonal
    const int j = blockIdx.x, lane = threadIdx.x & 31;
    const bool worker = threadIdx.x < 32;
    auto stage = [&](int c) {
        T *S = Gs + (c & 1) * kTCols * LDG;
        constexpr int NE = kTCols * LDG / 128, CH = NE < 16 ? NE : 16;
        for (int e0 = 0; e0 < NE; e0 += CH) {   // CH loads in flight per thread
            T g[CH];
#pragma unroll
            for (int u = 0; u < CH; u++) {
                const int e = threadIdx.x + 128 * (e0 + u), col = c * kTCols + e / LDG, r = e % LDG;
                zero_of(g[u]);
                if (col <= j && r < col) g[u] = G[(long long)col * ldg + r];
            }
#pragma unroll
            for (int u = 0; u < CH; u++) S[threadIdx.x + 128 * (e0 + u)] = g[u];
        }
    };
    T s[R], x[R], nt[R];                      // pending sums, results and -tau of rows lane + 32 u
#pragma unroll
    for (int u = 0; u < R; u++) {
        const int r = lane + 32 * u;
        zero_of(s[u]);
        zero_of(x[u]);
        zero_of(nt[u]);
        if (r < nb) nt[u] = scale(tau[r], -1.0);
        if (r == j) x[u] = tau[r];
    }
    const int last = j / kTCols;
    stage(last);
    __syncthreads();
    for (int c = last; c >= 0; c--) {
        if (c > 0) stage(c - 1);              // while the first warp works on c
        if (worker) {
            const T *S = Gs + (c & 1) * kTCols * LDG;
            for (int i = min(j, c * kTCols + kTCols - 1); i >= c * kTCols; i--) {
                const int src = i & 31, ui = i >> 5;
                T xi;
                zero_of(xi);
#pragma unroll
                for (int u = 0; u < R; u++)
                    if (u == ui) {
                        if (i < j) {
                            const T v = mul(nt[u], s[u]);
                            if (lane == src) x[u] = v;
                            xi = v;
                        } else {
                            xi = x[u];
                        }
                    }
                xi = lane_of(xi, src);
                const T *g = S + (i - c * kTCols) * LDG;
#pragma unroll
                for (int u = 0; u < R; u++)   // the rows above i
                    if (u <= ui && lane + 32 * u < i) s[u] = mad(g[lane + 32 * u], xi, s[u]);
            }
        }
        __syncthreads();
    }
    if (!worker) return;
#pragma unroll
    for (int u = 0; u < R; u++) {
        const int r = lane + 32 * u;
        if (r < nb) Tm[(long long)j * ldt + r] = x[u];
    }
}

template <class T, int R>
cudaError_t launch_panel_t_as(int nb, const T *G, long long ldg, const T *tau, T *Tm, long long ldt, cudaStream_t st)
{
    const size_t smem = (size_t)2 * kTCols * 32 * R * sizeof(T);
    cudaError_t e = cudaFuncSetAttribute(panel_t_kernel<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    panel_t_kernel<T, R><<<nb, 128, smem, st>>>(nb, G, ldg, tau, Tm, ldt);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_panel_t(int nb, const T *G, long long ldg, const T *tau, T *Tm, long long ldt, cudaStream_t st)
{
    if (nb < 1) return cudaSuccess;
    if (nb <= 32) return launch_panel_t_as<T, 1>(nb, G, ldg, tau, Tm, ldt, st);
    if (nb <= 64) return launch_panel_t_as<T, 2>(nb, G, ldg, tau, Tm, ldt, st);
    if (nb <= 128) return launch_panel_t_as<T, 4>(nb, G, ldg, tau, Tm, ldt, st);
    if (nb <= kTMax) return launch_panel_t_as<T, 8>(nb, G, ldg, tau, Tm, ldt, st);
    return cudaErrorInvalidValue;
}

// Explicit reflectors of `np` consecutive panels of nb columns each, side by
// side (m x np nb, ldy): panel p's reflectors start at row p nb, its QR'd
// form lies at P + p (nb lda + nb) (the diagonal blocks below one another).
template <class T>
__global__ void __launch_bounds__(256) panels_explicit_y(int m, int nb, int np, const T *__restrict__ P, long long lda,
                                                         T *__restrict__ Y, long long ldy)
{
    const long long total = (long long)m * nb * np;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e / m), r = (int)(e - (long long)c * m);
        T y;
        zero_of(y);
        if (r == c) one_of(y);       // column c of the group has its unit entry in row c
        else if (r > c) y = P[(long long)c * lda + r];
        Y[(long long)c * ldy + r] = y;
    }
}

}  // namespace

cudaError_t panels_y(int is_complex, int m, int nb, int np, const double *P, long long lda, double *Y, long long ldy,
                     cudaStream_t st)
{
    const unsigned blocks = (unsigned)std::min(1184LL, ((long long)m * nb * np + 255) / 256);
    if (is_complex)
        panels_explicit_y<Zc><<<blocks, 256, 0, st>>>(m, nb, np, (const Zc *)P, lda, (Zc *)Y, ldy);
    else
        panels_explicit_y<double><<<blocks, 256, 0, st>>>(m, nb, np, P, lda, Y, ldy);
    return cudaGetLastError();
}

// T of the panel's block reflector from G = Y^H Y (nb x nb, ldg; the strict
// upper part is read) and tau
cudaError_t panel_t(int nb, const double *G, long long ldg, const double *tau, double *T, long long ldt,
                    cudaStream_t st)
{
    return launch_panel_t<double>(nb, G, ldg, tau, T, ldt, st);
}

cudaError_t zpanel_t(int nb, const double *G, long long ldg, const double *tau, double *T, long long ldt, cudaStream_t st)
{
    return launch_panel_t<Zc>(nb, (const Zc *)G, ldg, (const Zc *)tau, (Zc *)T, ldt, st);
}

// Bytes of the exchange area a panel of m rows may need (`part`).
size_t panel_part_bytes(int m, int is_complex)
{
    const size_t blocks = ((size_t)m + 63) / 64;
    return 256 + (size_t)2 * 64 * (blocks + 1) * (is_complex ? 16 : 8);
}

// QR of the m x nb panel P (lda, nb <= 64) and, where Y is not null, its
// explicit reflectors (ldy).  *done = false: nothing was done, the panel is
// too tall for one co-resident grid (or for a cluster, under capture).
// `status`: a device word that receives GB_ERR_TIMEOUT when a wait gives up, or
// null.
cudaError_t panel_qr_resident(int is_complex, int m, int nb, double *P, long long lda, double *tau, double *Y,
                              long long ldy, void *part, int *status, cudaStream_t st, bool *done)
{
    PanelWait pw;
    pw.status = status;
    if (is_complex) return panel_qr_t<Zc>(m, nb, (Zc *)P, lda, (Zc *)tau, (Zc *)Y, ldy, part, pw, st, done);
    return panel_qr_t<double>(m, nb, P, lda, tau, Y, ldy, part, pw, st, done);
}

}  // namespace gb

extern "C" {

// Fault-injection hook of the tests (not in the header): a panel of which
// block 0 does not arrive at column `hold`, with waits of wait_ns.
int gb_test_panel_hold(int is_complex, int m, int nb, double *P, double *tau, double *Y, void *part, long long wait_ns,
                       int hold, int *status, void *stream)
{
    gb::PanelWait pw;
    pw.ns = wait_ns;
    pw.status = status;
    pw.hold = hold;
    bool done = false;
    const cudaStream_t st = (cudaStream_t)stream;
    const cudaError_t e =
        is_complex ? gb::panel_qr_t<gb::Zc>(m, nb, (gb::Zc *)P, m, (gb::Zc *)tau, (gb::Zc *)Y, m, part, pw, st, &done)
                   : gb::panel_qr_t<double>(m, nb, P, m, tau, Y, m, part, pw, st, &done);
    return e == cudaSuccess && done ? GB_OK : GB_ERR_CUDA;
}

}  // extern "C"
