// Band -> tridiagonal reduction by bulge chasing on the device (the second
// step of the two-stage reduction, Sec. 2), emitting the reflectors in the
// layout trans_ev_tridi_to_band consumes.
//
// Sweep s generates H(s,k), k = 0, 1, ..., from the column it annihilates
// (column s for k = 0, the first column of the previous bulge otherwise) and
// applies it from both sides, all in the lower triangle.  With R_k the rows
// of H(s,k) (0-based s+k*b .. s+k*b+len-1), step k of a sweep is
//   O(s,k)  the off-diagonal block rows R_k x columns R_{k-1}: multiply by
//           H(s,k-1) from the right, generate H(s,k) from the first column,
//           multiply by it from the left (k = 0: the source column alone);
//   D(s,k)  the diagonal block R_k x R_k: symmetric two-sided update.
// The working matrix is kept in lower band storage of width 2b (entries up
// to 2b-1 below the diagonal, where the bulges live), in a workspace.
//
// What bounds it: the chain of sweeps.  O(s,k) needs O(s-1,k), D(s-1,k) and,
// for its last entry only, the beta of H(s-1,k+1); D(s,k) needs D(s-1,k),
// O(s-1,k+1) and the first entry of D(s-1,k+1).  So sweep s trails sweep s-1
// by one O step and the generation of the next reflector, and the stage
// takes n times that.  One SM issues two FP64 multiply-adds per clock, so a
// step's 12 b^2 flops of arithmetic per flop pair cost several microseconds
// on one SM; a sweep therefore runs on a cluster of C + CD blocks:
//   * ranks 0 .. C-1 hold b/C rows of O each.  The right product is local to
//     a row; the column sums x^T A (x the raw source column, A's own first
//     column giving x^T x) are exchanged once per step through distributed
//     shared memory, and every rank derives tau, the scale and v from them:
//     v^T a_j = a_0j + scale * sum_{i>0} x_i a_ij;
//   * ranks C .. C+CD-1 receive x as well and update D (rows dealt round
//     robin); with CD = 2 they exchange their parts of D v.
// Each block has 256 computing threads, four loader warps that wait for the
// flags of sweep s-1 and stage the next block in shared memory while the
// current one is worked on, and one publisher warp that makes the stores
// visible and raises this sweep's flags, so that neither the loads nor the
// fences sit on the chain.
//
// Measured on a GB300 (whole stage, before: one block of 256 threads per
// sweep with a lag of three tasks; now): real n = 512, nbw = 32: 15.1 -> 4.2 ms;
// nbw = 64: n = 2048 82 -> 23.5, 8192 339 -> 119, 16384 684 -> 348; complex
// n = 512, nbw = 32: 46 -> 6.9; nbw = 64: n = 2048 322 -> 50, 8192 1351 -> 325.
//
// Sweeps are taken by ticket in increasing s by a persistent grid of
// clusters, so every wait targets a smaller ticket, which a resident cluster
// holds: no deadlock at any residency.  All waits are bounded; a cluster in
// which a wait gave up finishes its sweep without waiting for flags, so that
// no block touches the shared memory of one that has left.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "elpa_gb300.h"
#include "layout.cuh"
#include "reduction.cuh"
#include "tcgen05.cuh"
#include "trans_ev_kernels.cuh"

#include <vector>

namespace gb {

namespace cg = cooperative_groups;

namespace {

constexpr int kMain = 256;       // computing threads of a block
constexpr int kLoaders = 128;    // threads 256 .. 383
constexpr int kChaseThreads = kMain + kLoaders + 32;  // and the publisher warp
constexpr int kFlags = 4;        // ints per sweep: reflectors generated, O parts done, D parts done, unused

__device__ __forceinline__ int ld_acq(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_rel(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void red_rel(int *p, int v)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void main_sync()
{
    __syncwarp();
    asm volatile("bar.sync 1, 256;" ::: "memory");
}
__device__ __forceinline__ void loader_sync()
{
    __syncwarp();
    asm volatile("bar.sync 2, 128;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(void *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc5::smem_addr(bar)) : "memory");
}

struct ChaseState {
    int ticket;
    int abort;
    int error;
};

// One problem of a batched chase: its working band and reflector arrays and
// its progress flags (kFlags ints per sweep).
struct ChaseProblem {
    int n, b;
    void *W;
    long long ldw;
    void *hh_v, *hh_tau;
    int *progress;
};

// Lower band storage of width 2b: A(i,j), i >= j, at W[(i-j) + j*ldw];
// reads go to L2 (entries written by other SMs).
template <class T>
struct Band {
    T *W;
    long long ldw;
    __device__ __forceinline__ T *at(int i, int j) const { return W + (i - j) + (long long)j * ldw; }
};

// ---- one block's shared memory ---------------------------------------------

template <class T, int BM, int C, int CD>
struct ChaseGeo {
    static constexpr int S = C + CD;              // blocks of a cluster
    static constexpr int RW = BM / C;             // O rows of a rank
    static constexpr int RD = BM / CD;            // D rows of a rank
    static constexpr int LD = BM + 4;             // entries per staged row
    static constexpr int NO = 2;                  // staged O blocks
    static constexpr int ND = sizeof(T) == 16 ? 1 : 2;  // staged D blocks
    static constexpr int TPR = kMain / RW;        // threads per O row (right product)
    static constexpr int TPC = kMain / BM;        // threads per O column (left product)
    static constexpr int TPD = kMain / RD;        // threads per D row
    static constexpr int NG = BM / 16;            // 16-row groups of the column sums
    static constexpr int NGR = RW / 16;           // of a rank
    static constexpr int OBUF = RW * LD, DBUF = RD * LD;
    static constexpr size_t STAGE = sizeof(T) * (size_t)(NO * OBUF > ND * DBUF ? NO * OBUF : ND * DBUF);
    static_assert(TPR >= 1 && TPR <= 32 && TPC >= 1 && TPC <= 8 && TPR <= 16 && TPD <= 16, "threads of a row or column share a warp");
    static_assert(S <= 8 && RW * S <= kMain && BM <= 64, "cluster and mailbox sizes");
};

template <class T, int BM, int C>
struct ChaseShared {
    T mx[2][BM];        // mailbox: the source column x
    T ms[2][BM / 16][BM];   // partial column sums sum_{i>0} conj(x_i) a_ij by 16-row group
    T ma[2][BM];        // row 0 of the block
    T mp[2][BM];        // tau D v (D ranks)
    T v[2][BM];         // v(s,k) by step parity
    T w[BM], sum[BM], q[BM];
    T tau, scal, kk;
    double beta[2];
    unsigned long long full[2], empty[2], xo[2], xd, gen[2], st[2];
    int sweep[2], abort;
};

template <class T, int BM, int C, int CD>
constexpr size_t chase_smem()
{
    return ChaseGeo<T, BM, C, CD>::STAGE + sizeof(ChaseShared<T, BM, C>) + 16;
}

// A wait gave up: tell the launch (other clusters stop too) and this block.
__device__ __forceinline__ void chase_give_up(ChaseState *state, int *abort)
{
    atomicExch(&state->error, GB_ERR_TIMEOUT);
    atomicExch(&state->abort, 1);
    *(volatile int *)abort = 1;
}

// mbarrier wait of any thread, bounded
__device__ __forceinline__ void chase_wait(void *bar, uint32_t parity, long long timeout_ns, ChaseState *state,
                                           int *abort)
{
    const uint32_t a = tc5::smem_addr(bar);
    if (mbar_try_cluster(a, parity)) return;
    const unsigned long long t0 = now_ns();
    for (long long i = 1; i < (1ll << 40); i++) {
        if (mbar_try_cluster(a, parity)) return;
        if ((i & 63) == 0 && (long long)(now_ns() - t0) > timeout_ns) break;
    }
    chase_give_up(state, abort);
}

// one loader thread: wait until a flag of sweep s-1 reaches `need`
__device__ __forceinline__ void chase_flag(const int *flag, int need, long long timeout_ns, ChaseState *state,
                                           int *abort)
{
    if (ld_acq(flag) >= need) return;
    const unsigned long long t0 = now_ns();
    for (long long i = 1;; i++) {
        if (ld_acq(flag) >= need) return;
        if ((i & 15) == 0) {
            if (*(volatile int *)&state->abort) break;
            if ((long long)(now_ns() - t0) > timeout_ns) {
                chase_give_up(state, abort);
                return;
            }
            __nanosleep(20);
        }
    }
    *(volatile int *)abort = 1;
}

// ---- a cluster: sweeps by ticket --------------------------------------------

// Next sweep (and problem) of the launch: one problem, or many of them with
// ticket t = sweep 1 + t / count of problem t % count.
struct ChaseWork {
    int count, smax;                 // problems, and the most sweeps of any
    ChaseProblem one;                // the problem, where there is no table
    const ChaseProblem *table;
};

template <class T, int BM, int C, int CD>
__global__ void __launch_bounds__(kChaseThreads, 1)
chase_kernel(ChaseWork work, ChaseState *state, long long timeout_ns)
{
    using G = ChaseGeo<T, BM, C, CD>;
    constexpr int LD = G::LD, RW = G::RW;
    extern __shared__ __align__(16) unsigned char chase_dyn[];
    T *stage = (T *)chase_dyn;
    ChaseShared<T, BM, C> &sm = *(ChaseShared<T, BM, C> *)(chase_dyn + G::STAGE);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const bool is_o = rank < C;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nbuf = is_o ? G::NO : G::ND;
    const int bufsz = is_o ? G::OBUF : G::DBUF;
    // peers' waits last as long as their flag waits may
    const long long wait_ns = 2 * timeout_ns;

    if (tid == 0) {
        sm.abort = 0;
        for (int i = 0; i < 2; i++) {
            tc5::mbar_init(tc5::smem_addr(&sm.full[i]), kLoaders);
            tc5::mbar_init(tc5::smem_addr(&sm.empty[i]), kMain + 1);
            tc5::mbar_init(tc5::smem_addr(&sm.xo[i]), is_o ? C + CD : C);
            tc5::mbar_init(tc5::smem_addr(&sm.gen[i]), 1);
            tc5::mbar_init(tc5::smem_addr(&sm.st[i]), kMain);
        }
        tc5::mbar_init(tc5::smem_addr(&sm.xd), CD);
        tc5::mbar_init_fence();
    }
    cluster.sync();
    // a D rank has consumed nothing yet: credit for the O ranks' first step
    if (!is_o && tid < C) mbar_arrive_remote(&sm.xo[0], tid);

    uint32_t kk = 0;       // steps so far, over all sweeps of this cluster
    uint32_t nxd = 0;      // exchanges of D v so far
    const long long total = (long long)work.count * work.smax;
    for (int it = 0;; it++) {
        if (rank == 0 && tid == 0) {
            const long long t = atomicAdd(&state->ticket, 1);
            const int put = (t >= total || *(volatile int *)&state->abort) ? -1 : (int)t;
            for (int r = 0; r < G::S; r++) cluster.map_shared_rank(&sm.sweep[it & 1], r)[0] = put;
        }
        __syncwarp();
        cluster.sync();
        const int t = sm.sweep[it & 1];
        if (t < 0) break;
        const ChaseProblem pr = work.table ? work.table[t % work.count] : work.one;
        const int s = 1 + t / work.count;
        const int n = pr.n, b = pr.b;
        if (s > n - 1) continue;
        const Band<T> A{(T *)pr.W, pr.ldw};
        const int nk = sweep_count(n, b, s);
        const int nkp = (s > 1) ? sweep_count(n, b, s - 1) : 0;
        const long long first = sweep_first(n, b, s);
        int *mine = pr.progress + (size_t)kFlags * (s - 1);
        const int *prev = mine - kFlags;

        if (tid < kMain && is_o) {
            // ================= O: right product, reflector, left product
            const int i0 = rank * RW;
            bool active = false;                      // H(s,k-1) is not the identity
            T ptau;
            zero_of(ptau);
            for (int k = 0; k < nk; k++, kk++) {
                const int r = s + k * b, len = min(b, n - r);
                const int c = (k == 0) ? s - 1 : r - b;
                const int ncols = (k == 0) ? 1 : b;
                const int par = kk & 1;
                T *B = stage + (kk % G::NO) * G::OBUF;
                chase_wait(&sm.full[kk % G::NO], (kk / G::NO) & 1, wait_ns, state, &sm.abort);
                if (active) {
                    const int row = tid / G::TPR, part = tid % G::TPR;
                    const T *vp = sm.v[par ^ 1];
                    constexpr int NA = 16 / G::TPR;
                    T e[BM / G::TPR], acc[NA];
#pragma unroll
                    for (int u = 0; u < NA; u++) zero_of(acc[u]);
#pragma unroll
                    for (int u = 0; u < BM / G::TPR; u++) {
                        e[u] = B[row * LD + part + G::TPR * u];
                        acc[u % NA] = mad(e[u], vp[part + G::TPR * u], acc[u % NA]);
                    }
                    const T y = mul(ptau, tree_sum<16, G::TPR>(acc));
#pragma unroll
                    for (int u = 0; u < BM / G::TPR; u++)
                        B[row * LD + part + G::TPR * u] = nmad(y, conj_of(vp[part + G::TPR * u]), e[u]);
                }
                main_sync();
                // column sums with the raw source column (the block's first)
                const int col = tid / G::TPC, cp = tid % G::TPC;
                T e[RW / G::TPC];
                {
                    constexpr int NE = 16 / G::TPC, NA = 8 / G::TPC;
#pragma unroll
                    for (int g = 0; g < G::NGR; g++) {
                        T acc[NA];
#pragma unroll
                        for (int u = 0; u < NA; u++) zero_of(acc[u]);
#pragma unroll
                        for (int u = 0; u < NE; u++) {
                            const int i = 16 * g + cp + G::TPC * u;
                            e[g * NE + u] = B[i * LD + col];
                            if (i0 + i > 0) acc[u % NA] = madc(B[i * LD], e[g * NE + u], acc[u % NA]);
                        }
                        const T sum = tree_sum<8, G::TPC>(acc);
                        T *to = &sm.ms[par][rank * G::NGR + g][col];
                        for (int d = cp; d < C; d += G::TPC) cluster.map_shared_rank(to, d)[0] = sum;
                        if (col == 0 && cp < CD) cluster.map_shared_rank(to, C + cp)[0] = sum;
                    }
                    if (rank == 0) {
                        const T a0 = B[col];
                        for (int d = cp; d < C; d += G::TPC) cluster.map_shared_rank(&sm.ma[par][col], d)[0] = a0;
                        if (col == 0 && cp < CD) cluster.map_shared_rank(&sm.ma[par][0], C + cp)[0] = a0;
                    }
                    if (tid < RW * G::S)
                        cluster.map_shared_rank(&sm.mx[par][i0 + tid % RW], tid / RW)[0] = B[(tid % RW) * LD];
                }
                main_sync();
                if (tid < G::S) {
                    asm volatile("fence.acq_rel.cluster;" ::: "memory");
                    mbar_arrive_remote(&sm.xo[par], tid);
                }
                chase_wait(&sm.xo[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                // every rank: the reflector, and the sums over ranks
                if (warp == 0) {
                    double ss = 0.0;
                    for (int q = 0; q < G::NG; q++) ss += re_of(sm.ms[par][q][0]);
                    const auto h = reflector(sm.ma[par][0], ss);
                    if (lane == 0) {
                        sm.tau = h.tau;
                        sm.scal = h.scal;
                        sm.beta[par] = h.beta;
                        mbar_arrive(&sm.gen[par]);
                    }
                } else if (tid >= 64 && tid < 64 + BM) {
                    T t2;
                    zero_of(t2);
                    for (int q = 0; q < G::NG; q++) t2 = add(t2, sm.ms[par][q][tid - 64]);
                    sm.sum[tid - 64] = t2;
                }
                main_sync();
                const T tau = sm.tau, scal = sm.scal;
                if (tid < BM) {
                    T vi;
                    if (tid == 0) one_of(vi);
                    else vi = mul(sm.mx[par][tid], scal);   // scal = 0 where tau = 0; x = 0 past len
                    sm.v[par][tid] = vi;
                } else if (tid >= 128 && tid < 128 + BM) {
                    // w_j = conj(tau) v^H a_j
                    const int j = tid - 128;
                    sm.w[j] = mul(conj_of(tau), mad(conj_of(scal), sm.sum[j], sm.ma[par][j]));
                }
                main_sync();
                const bool act = !is_zero(tau);
                {
                    const T wj = sm.w[col];
                    if (col < ncols) {
#pragma unroll
                        for (int u = 0; u < RW / G::TPC; u++) {
                            const int gi = i0 + cp + G::TPC * u;   // e[u]'s row: the groups follow each other
                            if (gi < len) {
                                if (col > 0) {
                                    *A.at(r + gi, c + col) = act ? nmad(sm.v[par][gi], wj, e[u]) : e[u];
                                } else if (gi > 0) {     // the annihilated column (its beta: the publisher)
                                    T z;
                                    zero_of(z);
                                    *A.at(r + gi, c) = act ? z : e[u];
                                }
                            }
                        }
                    }
                }
                mbar_arrive(&sm.st[par]);
                mbar_arrive(&sm.empty[kk % G::NO]);
                active = act;
                ptau = tau;
            }
        } else if (tid < kMain) {
            // ================= D: symmetric two-sided update
            const int dr = rank - C;
            for (int k = 0; k < nk; k++, kk++) {
                const int r = s + k * b, len = min(b, n - r);
                const int par = kk & 1;
                const long long idx = first + k;
                chase_wait(&sm.xo[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                if (warp == 0) {
                    double ss = 0.0;
                    for (int q = 0; q < G::NG; q++) ss += re_of(sm.ms[par][q][0]);
                    const auto h = reflector(sm.ma[par][0], ss);
                    if (lane == 0) {
                        sm.tau = h.tau;
                        sm.scal = h.scal;
                    }
                }
                main_sync();
                const T tau = sm.tau;
                if (tid < BM) {
                    T vi;
                    if (tid == 0) one_of(vi);
                    else vi = mul(sm.mx[par][tid], sm.scal);
                    sm.v[0][tid] = vi;
                    if (dr == 0 && tid < b) ((T *)pr.hh_v)[idx * b + tid] = vi;
                }
                if (dr == 0 && tid == 64) ((T *)pr.hh_tau)[idx] = tau;
                main_sync();
                // the mailbox is consumed: credit for the O ranks' next step
                if (tid < C) mbar_arrive_remote(&sm.xo[par ^ 1], tid);
                T *B = stage + (kk % G::ND) * G::DBUF;
                chase_wait(&sm.full[kk % G::ND], (kk / G::ND) & 1, wait_ns, state, &sm.abort);
                if (!is_zero(tau)) {
                    const int rr = tid / G::TPD, part = tid % G::TPD;
                    const int i = dr + CD * rr;                     // this thread's row of D
                    const T *v = sm.v[0];
                    const int pp = nxd & 1;
                    constexpr int NA = 16 / G::TPD;
                    T e[BM / G::TPD], acc[NA];
#pragma unroll
                    for (int u = 0; u < NA; u++) zero_of(acc[u]);
#pragma unroll
                    for (int u = 0; u < BM / G::TPD; u++) {
                        e[u] = B[rr * LD + part + G::TPD * u];
                        acc[u % NA] = mad(e[u], v[part + G::TPD * u], acc[u % NA]);
                    }
                    const T pi = mul(tau, tree_sum<16, G::TPD>(acc));
                    if (part < CD) cluster.map_shared_rank(&sm.mp[pp][i], C + part)[0] = pi;
                    main_sync();
                    if (CD > 1) {
                        if (tid < CD) {
                            asm volatile("fence.acq_rel.cluster;" ::: "memory");
                            mbar_arrive_remote(&sm.xd, C + tid);
                        }
                        chase_wait(&sm.xd, nxd & 1, wait_ns, state, &sm.abort);
                    }
                    nxd++;
                    // K = conj(tau)/2 v^H p, q = p - K v
                    if (warp == 0) {
                        T a[1];
                        zero_of(a[0]);
                        for (int j = lane; j < BM; j += 32) a[0] = madc(v[j], sm.mp[pp][j], a[0]);
                        const T vp = tree_sum<32, 32>(a);
                        if (lane == 0) sm.kk = mul(scale(conj_of(tau), 0.5), vp);
                    }
                    main_sync();
                    if (tid < BM) sm.q[tid] = nmad(sm.kk, v[tid], sm.mp[pp][tid]);
                    main_sync();
                    const T vi = v[i], qi = sm.q[i];
#pragma unroll
                    for (int u = 0; u < BM / G::TPD; u++) {
                        const int j = part + G::TPD * u;
                        if (j <= i && i < len)
                            *A.at(r + i, r + j) = nmad(vi, conj_of(sm.q[j]), nmad(qi, conj_of(v[j]), e[u]));
                    }
                }
                mbar_arrive(&sm.st[par]);
                mbar_arrive(&sm.empty[kk % G::ND]);
            }
        } else if (tid < kMain + kLoaders) {
            // ================= loaders: stage the next block
            const int lt = tid - kMain;
            for (int k = 0; k < nk; k++, kk++) {
                const int r = s + k * b, len = min(b, n - r);
                T *B = stage + (kk % nbuf) * bufsz;
                if (kk >= (uint32_t)nbuf)
                    chase_wait(&sm.empty[kk % nbuf], (kk / nbuf - 1) & 1, wait_ns, state, &sm.abort);
                const int upto = is_o ? min(k + 1, nkp) : min(k + 2, nkp);
                if (lt == 0 && s > 1 && !*(volatile int *)&sm.abort) {
                    chase_flag(prev + 1, C * upto, timeout_ns, state, &sm.abort);
                    chase_flag(prev + 2, CD * upto, timeout_ns, state, &sm.abort);
                }
                loader_sync();
                if (is_o) {
                    const int i0 = rank * RW;
                    const int c = (k == 0) ? s - 1 : r - b;
                    const int ncols = (k == 0) ? 1 : b;
                    // rows run along the band's contiguous index
                    constexpr int NU = RW * BM / kLoaders, CH = NU < 8 ? NU : 8;
#pragma unroll 1
                    for (int u0 = 0; u0 < NU; u0 += CH) {   // CH loads in flight per thread
                        T x[CH];
#pragma unroll
                        for (int u = 0; u < CH; u++) {
                            const int e = lt + kLoaders * (u0 + u), col = e / RW, i = e % RW;
                            zero_of(x[u]);
                            const bool corner = col == ncols - 1 && i0 + i == b - 1;   // beta of H(s-1,k+1): below
                            if (col < ncols && i0 + i < len && !corner) x[u] = ld_cg(A.at(r + i0 + i, c + col));
                        }
#pragma unroll
                        for (int u = 0; u < CH; u++) {
                            const int e = lt + kLoaders * (u0 + u), col = e / RW, i = e % RW;
                            B[i * LD + col] = x[u];
                        }
                    }
                    const int ci = b - 1 - i0;
                    if (len == b && ci >= 0 && ci < RW) {
                        loader_sync();
                        if (lt == 0) {
                            if (s > 1 && !*(volatile int *)&sm.abort)
                                chase_flag(prev, min(k + 2, nkp), timeout_ns, state, &sm.abort);
                            B[ci * LD + ncols - 1] = ld_cg(A.at(r + b - 1, c + ncols - 1));
                        }
                    }
                } else {
                    // the lower triangle, columns j and BM-1-j paired into runs of BM+1 entries
                    const int dr = rank - C;
                    constexpr int N2 = BM / 2 * (BM + 1), NU = (N2 + kLoaders - 1) / kLoaders, CH = 9;
#pragma unroll 1
                    for (int u0 = 0; u0 < NU; u0 += CH) {
                        T x[CH];
#pragma unroll
                        for (int u = 0; u < CH; u++) {
                            const int e = lt + kLoaders * (u0 + u);
                            const int q = e / (BM + 1), t2 = q + e % (BM + 1);   // row of column q, or past its end
                            const int j = t2 < BM ? q : BM - 1 - q, i = t2 < BM ? t2 : t2 - BM + j;
                            zero_of(x[u]);
                            if (e < N2 && i < len) x[u] = ld_cg(A.at(r + i, r + j));   // j <= i
                        }
#pragma unroll
                        for (int u = 0; u < CH; u++) {
                            const int e = lt + kLoaders * (u0 + u);
                            const int q = e / (BM + 1), t2 = q + e % (BM + 1);
                            const int j = t2 < BM ? q : BM - 1 - q, i = t2 < BM ? t2 : t2 - BM + j;
                            if (e < N2) {
                                if (i % CD == dr) B[(i / CD) * LD + j] = x[u];
                                if (j % CD == dr && i != j) B[(j / CD) * LD + i] = conj_of(x[u]);
                            }
                        }
                    }
                }
                mbar_arrive(&sm.full[kk % nbuf]);
            }
        } else if (lane == 0) {
            // ================= publisher: beta, fences and flags
            for (int k = 0; k < nk; k++, kk++) {
                const int par = kk & 1;
                if (is_o) {
                    chase_wait(&sm.gen[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                    if (rank == 0 && !*(volatile int *)&sm.abort) {
                        const int r = s + k * b, c = (k == 0) ? s - 1 : r - b;
                        T z;
                        zero_of(z);
                        *(double *)&z = sm.beta[par];
                        *A.at(r, c) = z;
                        st_rel(mine, k + 1);
                    }
                }
                chase_wait(&sm.st[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                if (!*(volatile int *)&sm.abort) {
                    __threadfence();
                    red_rel(mine + (is_o ? 1 : 2), 1);
                }
                mbar_arrive(&sm.empty[kk % nbuf]);
            }
        } else {
            kk += nk;
        }
    }
    __syncwarp();
    cluster.sync();   // no block leaves while a peer may still reach its shared memory
}

template <class T>
__global__ void __launch_bounds__(256) band_init(int n, int b, const T *__restrict__ AB, long long ldab,
                                                 T *__restrict__ W, long long ldw)
{
    const long long total = (long long)n * ldw;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        long long j = e / ldw, d = e - j * ldw;
        T z;
        zero_of(z);
        W[e] = (d <= b && j + d < n) ? AB[d + j * ldab] : z;
    }
}

template <class T>
__global__ void __launch_bounds__(256) band_extract(int n, const T *__restrict__ W, long long ldw,
                                                    double *__restrict__ dd, double *__restrict__ ee)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        dd[j] = re_of(W[(long long)j * ldw]);
        if (j < n - 1) ee[j] = re_of(W[1 + (long long)j * ldw]);
    }
}

}  // namespace

// Workspace: [256-byte head {ticket, abort, error}][progress: kFlags ints per
// sweep] then, 256-byte aligned, the 2b x n working band.
static size_t flags_bytes(int n) { return (256 + (size_t)n * kFlags * sizeof(int) + 255) & ~(size_t)255; }

size_t band_to_tridi_workspace_bytes(int n, int b)
{
    size_t band = 2 * (size_t)b * (size_t)n * sizeof(double);
    return flags_bytes(n) + ((band + 255) & ~(size_t)255);
}

size_t band_to_tridi_workspace_bytes_z(int n, int b)
{
    size_t band = 2 * (size_t)b * (size_t)n * 2 * sizeof(double);
    return flags_bytes(n) + ((band + 255) & ~(size_t)255);
}

// Sweeps that can be in flight at once: sweep s trails sweep s-1 by one O
// step and the generation of the next reflector, somewhat more than one step
// of its nk(1); further clusters would only poll, holding SM slots that
// concurrent work on other streams could use.
static int chase_active(int n, int b)
{
    const int nk1 = (n - 1 + b - 1) / b;
    return max(1, min(n - 1, (2 * nk1 + 2) / 3 + 2));
}

template <class T, int BM, int C, int CD>
static cudaError_t chase_launch_as(const ChaseWork &work, long long active, int sms, ChaseState *state,
                                   long long timeout_ns, cudaStream_t st)
{
    using G = ChaseGeo<T, BM, C, CD>;
    constexpr size_t smem = chase_smem<T, BM, C, CD>();
    auto kernel = chase_kernel<T, BM, C, CD>;
    // opt in to the large dynamic shared memory (cheap; per device, so every call)
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // at most two blocks per SM
    const long long clusters = max(1LL, min(active, 2LL * sms / G::S));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * G::S));
    cfg.blockDim = dim3(kChaseThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G::S;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, work, state, timeout_ns);
}

// `active`: sweeps in flight over all problems; bmax: the widest band.
// Real, b > 32: clusters of 6 (4 row parts of O, 2 of D: 11.5 us a sweep at
// n = 2048) while those of the sweeps in flight fit the SMs, else clusters of
// 3 (14.5 us a sweep at n = 8192, where clusters of 6 would leave half of the
// sweeps without SMs).  b <= 32 has a quarter of the work a step: clusters of
// 3 (8.1 us a sweep); complex steps have four times the work: 6 from b = 33.
static cudaError_t chase_launch(const ChaseWork &work, long long active, int bmax, int is_complex, ChaseState *state,
                                long long timeout_ns, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaError_t err;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return err;
    if (is_complex) {
        if (bmax <= 32) return chase_launch_as<Zc, 32, 2, 1>(work, active, sms, state, timeout_ns, st);
        return chase_launch_as<Zc, 64, 4, 2>(work, active, sms, state, timeout_ns, st);
    }
    if (bmax <= 32) return chase_launch_as<double, 32, 2, 1>(work, active, sms, state, timeout_ns, st);
    if (active * 6 <= sms) return chase_launch_as<double, 64, 4, 2>(work, active, sms, state, timeout_ns, st);
    return chase_launch_as<double, 64, 2, 1>(work, active, sms, state, timeout_ns, st);
}

static ChaseWork chase_one(int n, int b, void *W, void *hh_v, void *hh_tau, int *progress)
{
    ChaseWork w{};
    w.count = 1;
    w.smax = n - 1;
    w.one = ChaseProblem{n, b, W, 2LL * b, hh_v, hh_tau, progress};
    return w;
}

cudaError_t band_to_tridi_prepare_z(int n, int b, const double *AB, int ldab, void *ws, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    char *flags = (char *)ws;
    Zc *W = (Zc *)(flags + flags_bytes(n));
    cudaError_t err = cudaMemsetAsync(flags, 0, flags_bytes(n), st);
    if (err != cudaSuccess) return err;
    band_init<Zc><<<1024, 256, 0, st>>>(n, b, (const Zc *)AB, ldab, W, ldw);
    return cudaGetLastError();
}

cudaError_t band_to_tridi_finish_z(int n, int b, const void *ws, double *d, double *e, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    const Zc *W = (const Zc *)((const char *)ws + flags_bytes(n));
    band_extract<Zc><<<64, 256, 0, st>>>(n, W, ldw, d, e);
    return cudaGetLastError();
}

cudaError_t band_to_tridi_z(int n, int b, const double *AB, int ldab, double *d, double *e, double *hh_v,
                            double *hh_tau, void *ws, long long timeout_ns, cudaStream_t st)
{
    char *flags = (char *)ws;
    cudaError_t err = band_to_tridi_prepare_z(n, b, AB, ldab, ws, st);
    if (err != cudaSuccess) return err;
    if (n > 1) {
        const ChaseWork w = chase_one(n, b, flags + flags_bytes(n), hh_v, hh_tau, (int *)(flags + 256));
        if ((err = chase_launch(w, chase_active(n, b), b, 1, (ChaseState *)flags, timeout_ns, st)) != cudaSuccess)
            return err;
    }
    return band_to_tridi_finish_z(n, b, ws, d, e, st);
}

cudaError_t band_to_tridi_prepare_d(int n, int b, const double *AB, int ldab, void *ws, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    char *flags = (char *)ws;
    double *W = (double *)(flags + flags_bytes(n));
    cudaError_t err = cudaMemsetAsync(flags, 0, flags_bytes(n), st);
    if (err != cudaSuccess) return err;
    band_init<double><<<1024, 256, 0, st>>>(n, b, AB, ldab, W, ldw);
    return cudaGetLastError();
}

cudaError_t band_to_tridi_finish_d(int n, int b, const void *ws, double *d, double *e, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    const double *W = (const double *)((const char *)ws + flags_bytes(n));
    band_extract<double><<<64, 256, 0, st>>>(n, W, ldw, d, e);
    return cudaGetLastError();
}

cudaError_t band_to_tridi_d(int n, int b, const double *AB, int ldab, double *d, double *e, double *hh_v,
                            double *hh_tau, void *ws, size_t ws_bytes, long long timeout_ns, cudaStream_t st)
{
    (void)ws_bytes;
    char *flags = (char *)ws;
    cudaError_t err = band_to_tridi_prepare_d(n, b, AB, ldab, ws, st);
    if (err != cudaSuccess) return err;
    if (n > 1) {
        const ChaseWork w = chase_one(n, b, flags + flags_bytes(n), hh_v, hh_tau, (int *)(flags + 256));
        if ((err = chase_launch(w, chase_active(n, b), b, 0, (ChaseState *)flags, timeout_ns, st)) != cudaSuccess)
            return err;
    }
    return band_to_tridi_finish_d(n, b, ws, d, e, st);
}

size_t chase_batched_table_bytes(int count) { return 256 + (((size_t)count * sizeof(ChaseProblem) + 255) & ~(size_t)255); }

// The chases of `count` problems in one persistent launch, in two calls on
// one stream: band_to_tridi_chase_batched_upload_d writes the launch's state
// word (ticket, abort, error; read it with gb_trans_ev_query) and the problem
// table into `table` (device, chase_batched_table_bytes(count)), from the
// host (a copy from pageable memory waits for the stream's earlier work, so
// issue it before that work); band_to_tridi_chase_batched_d launches once
// band_to_tridi_prepare_d has run on every problem's workspace ws[i].
cudaError_t band_to_tridi_chase_batched_upload_d(int count, const int *n, const int *b, void *const *ws,
                                                 double *const *hh_v, double *const *hh_tau, void *table,
                                                 cudaStream_t st)
{
    if (count < 1) return cudaSuccess;
    std::vector<ChaseProblem> host((size_t)count);
    for (int i = 0; i < count; i++) {
        char *flags = (char *)ws[i];
        host[i] = ChaseProblem{n[i], b[i], flags + flags_bytes(n[i]), 2LL * b[i], hh_v[i], hh_tau[i],
                               (int *)(flags + 256)};
    }
    cudaError_t err = cudaMemsetAsync(table, 0, 256, st);
    if (err != cudaSuccess) return err;
    // from pageable memory: staged before the call returns, so `host` may go
    return cudaMemcpyAsync((char *)table + 256, host.data(), host.size() * sizeof(ChaseProblem),
                           cudaMemcpyHostToDevice, st);
}

cudaError_t band_to_tridi_chase_batched_d(int count, const int *n, const int *b, void *table, long long timeout_ns,
                                          cudaStream_t st)
{
    return band_to_tridi_chase_batched(count, n, b, table, timeout_ns, st, 0);
}

cudaError_t band_to_tridi_chase_batched(int count, const int *n, const int *b, void *table, long long timeout_ns,
                                        cudaStream_t st, int is_complex)
{
    int smax = 0, bmax = 1;
    long long active = 0;
    for (int i = 0; i < count; i++) {
        smax = max(smax, n[i] - 1);
        bmax = max(bmax, b[i]);
        if (n[i] > 1) active += chase_active(n[i], b[i]);
    }
    if (count < 1 || smax < 1) return cudaSuccess;
    ChaseWork w{};
    w.count = count;
    w.smax = smax;
    w.table = (const ChaseProblem *)((char *)table + 256);
    return chase_launch(w, active, bmax, is_complex, (ChaseState *)table, timeout_ns, st);
}

}  // namespace gb
