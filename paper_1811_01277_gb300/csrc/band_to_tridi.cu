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
// What bounds it: the chain of sweeps.  O(s,k) shares all but its last column
// and row with O(s-1,k); the last column is the first of D(s-1,k), and its last
// entry the beta of H(s-1,k+1).  The last row is zero but for that entry: its
// columns were annihilated by H(s-m,k+1), m >= 2, so it is not loaded, the zeros
// are never stored, and nothing has to wait for those blocks, one step ahead of
// the ones whose flags O(s,k) looks at.  D(s,k) shares all but its last row with
// D(s-1,k); that row is the first of O(s-1,k+1) and, on the diagonal, the first
// entry of D(s-1,k+1).  So sweep s trails sweep s-1 by one O step and one hop of those few
// entries, and the stage takes n times that.  One SM issues two FP64
// multiply-adds per clock, so a step's arithmetic (4 b^2 multiply-adds in O, 2 b^2
// and more in D) costs several microseconds on one SM; a sweep therefore runs
// on a cluster of C + CD blocks:
//   * ranks 0 .. C-1 hold b/C rows of O each.  The right product is local to
//     a row; the column sums x^T A (x the raw source column, A's own first
//     column giving x^T x) are exchanged once per step as asynchronous stores
//     into the peers' shared memory that count on their mbarriers, and every
//     rank derives tau, the scale and v from them: v^T a_j = a_0j + scale *
//     sum_{i>0} x_i a_ij.  128 threads keep this chain; another 128 take the
//     left product and the stores, while the chain is at the next block;
//   * ranks C .. C+CD-1 receive x as well and update D (rows dealt round
//     robin), D x before the reflector's scalars are known; with CD = 2 they
//     exchange their parts of D v.
// Each block also has four loader warps, which wait for the flags of sweep s-1
// and stage the next block in shared memory while the current one is worked on,
// and one publisher warp, which raises this sweep's flags.  The few entries on
// the chain (betas, first columns of D) skip the flags: they pass through slots
// in global memory that say themselves whether they are full.
//
// Measured on a GB300 (whole stage; before: one block of 256 threads per sweep
// with a lag of three tasks; then: clusters with every block behind flags; now):
// real n = 512, nbw = 32: 15.1, 4.2, 3.3 ms; nbw = 64: n = 2048 82, 23.5, 17.9;
// 8192 339, 119, 99; 16384 684, 348, 292; complex n = 512, nbw = 32: 46, 6.9,
// 6.9; nbw = 64: n = 2048 322, 50, 39; 8192 1351, 325, 310.  At n = 2048 an O
// step's chain is 3.3 us (2.0 from the block's arrival to the exchanged sums, 1.2
// for the reflector and v), a hop 3.4 us and the lag 8.6 us: jitter adds to both.
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
constexpr int kChain = 128;      // O blocks: threads 0 .. 127 keep the chain, 128 .. 255 finish the blocks
constexpr int kLoaders = 128;    // threads 256 .. 383
constexpr int kChaseThreads = kMain + kLoaders + 32;  // and the publisher warp
constexpr int kFlags = 8;        // ints per sweep: the steps each block of its cluster has stored (one 32-byte sector)
// The few entries that two sweeps meet at, the betas and the first columns of
// the D blocks, pass from a sweep to the next through slots that say themselves
// whether they are full (this signalling NaN is no result of arithmetic), so
// that no fence, flag or second load stands between a value and its reader.
constexpr unsigned long long kEmpty = 0x7ff4c0de00be7a00ull;

__device__ __forceinline__ int ld_acq(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void st_rel(int *p, int v)
{
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void main_sync()   // the computing threads of a D block
{
    __syncwarp();
    asm volatile("bar.sync 1, 256;" ::: "memory");
}
__device__ __forceinline__ void chain_sync()  // the chain's threads of an O block
{
    __syncwarp();
    asm volatile("bar.sync 3, 128;" ::: "memory");
}
// D blocks: the publisher warp hands the reflector's scalars to the others
__device__ __forceinline__ void scalars_give()
{
    __syncwarp();
    asm volatile("bar.arrive 4, 288;" ::: "memory");
}
__device__ __forceinline__ void scalars_take()
{
    __syncwarp();
    asm volatile("bar.sync 4, 288;" ::: "memory");
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

// One problem of a batched chase: its working band and reflector arrays, its
// progress flags (kFlags ints per sweep) and its slots, for odd and for even
// sweeps: a beta per step, and b entries per step for the first column of D.  A
// slot is emptied by its reader, sweep s+1, before its next writer, sweep s+2,
// can be there.
struct ChaseProblem {
    int n, b;
    void *W;
    long long ldw;
    void *hh_v, *hh_tau;
    int *progress;
    unsigned long long *betas, *firsts;
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
    static constexpr int TPR = kChain / RW;       // threads per O row (right product)
    static constexpr int TPC = kChain / BM;       // threads per O column (column sums, left product)
    static constexpr int TPD = kMain / RD;        // threads per D row
    static constexpr int NG = BM / 16;            // 16-row groups of the column sums
    static constexpr int NGR = RW / 16;           // of a rank
    static constexpr int OBUF = RW * LD, DBUF = RD * LD;
    static constexpr size_t STAGE = sizeof(T) * (size_t)(NO * OBUF > ND * DBUF ? NO * OBUF : ND * DBUF);
    // bytes of a step's messages: column sums, row 0 and the source column to
    // an O rank; the source column, its own sums and its first entry to a D rank
    static constexpr uint32_t O_BYTES = (uint32_t)sizeof(T) * (NG * BM + 2 * BM);
    static constexpr uint32_t D_BYTES = (uint32_t)sizeof(T) * (BM + NG + 1);
    static constexpr uint32_t P_BYTES = (uint32_t)sizeof(T) * BM;
    static_assert(TPR >= 1 && TPC >= 1 && TPC <= 8 && TPR <= 16 && TPD <= 16, "threads of a row or column share a warp");
    static_assert(S <= kFlags && RW * S <= kChain && BM <= 64 && RW % 16 == 0, "cluster and mailbox sizes");
};

template <class T, int BM, int C>
struct ChaseShared {
    T mx[2][BM];            // mailbox: the source column x
    T ms[2][BM / 16][BM];   // partial column sums sum_{i>0} conj(x_i) a_ij by 16-row group
    T ma[2][BM];            // row 0 of the block
    T mp[2][BM];            // tau D v (D ranks)
    T v[2][BM], w[2][BM];   // v(s,k) and conj(tau) v^H A by step parity
    T tau[2], scal[2];
    T sum[BM], q[BM], kk;
    unsigned long long full[2], empty[2], xo[2], xd[2], vw[2], st[2];
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

// A loader warp waits until every block of sweep s-1 has stored its part (lane
// r looks at block r's flag: need_o steps of the O blocks, need_d of the D
// blocks).  One flag per block: blocks may be two steps apart, so a sum
// over them would not say that each is there.
template <int C, int CD>
__device__ __forceinline__ void chase_flags(const int *prev, int need_o, int need_d, long long timeout_ns,
                                            ChaseState *state, int *abort)
{
    const int lane = threadIdx.x & 31;
    const int need = lane < C ? need_o : lane < C + CD ? need_d : 0;
    auto there = [&]() { return __all_sync(0xffffffffu, need == 0 || ld_acq(prev + lane) >= need); };
    if (there()) return;
    const unsigned long long t0 = now_ns();
    for (long long i = 1;; i++) {
        if (there()) return;
        if ((i & 15) == 0) {
            const bool stop = *(volatile int *)&state->abort != 0;
            const bool late = (long long)(now_ns() - t0) > timeout_ns;
            if (__any_sync(0xffffffffu, late)) {
                if (lane == 0) chase_give_up(state, abort);
                break;
            }
            if (__any_sync(0xffffffffu, stop)) break;
        }
    }
    *(volatile int *)abort = 1;
}

// one loader thread: the value in `slot`, which is emptied
__device__ __forceinline__ double take(unsigned long long *slot, long long timeout_ns, ChaseState *state, int *abort)
{
    unsigned long long v = ld_relaxed(slot);
    if (v == kEmpty) {
        const unsigned long long t0 = now_ns();
        for (long long i = 1; (v = ld_relaxed(slot)) == kEmpty; i++) {
            if ((i & 15) == 0) {
                if (*(volatile int *)&state->abort) break;
                if ((long long)(now_ns() - t0) > timeout_ns) {
                    chase_give_up(state, abort);
                    break;
                }
            }
        }
        if (v == kEmpty) {
            *(volatile int *)abort = 1;
            return 0.0;
        }
    }
    st_relaxed(slot, kEmpty);
    return __longlong_as_double((long long)v);
}
__device__ __forceinline__ void take_entry(double &x, unsigned long long *slots, int i, long long timeout_ns,
                                           ChaseState *state, int *abort)
{
    x = take(slots + i, timeout_ns, state, abort);
}
__device__ __forceinline__ void take_entry(Zc &x, unsigned long long *slots, int i, long long timeout_ns,
                                           ChaseState *state, int *abort)
{
    x.re = take(slots + 2 * i, timeout_ns, state, abort);
    x.im = take(slots + 2 * i + 1, timeout_ns, state, abort);
}
__device__ __forceinline__ void put_entry(unsigned long long *slots, int i, double x)
{
    st_relaxed(slots + i, (unsigned long long)__double_as_longlong(x));
}
__device__ __forceinline__ void put_entry(unsigned long long *slots, int i, Zc x)
{
    put_entry(slots, 2 * i, x.re);
    put_entry(slots, 2 * i + 1, x.im);
}

// |x|^2 below the source column's first entry, from its sums over groups
template <int NG, class T>
__device__ __forceinline__ double group_sum(const T *ms, int stride)
{
    double t = re_of(ms[0]) + re_of(ms[stride]);
    if (NG == 4) t += re_of(ms[2 * stride]) + re_of(ms[3 * stride]);
    return t;
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
__global__ void __launch_bounds__(kChaseThreads, sizeof(T) == 16 ? 1 : 2)
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
            tc5::mbar_init(tc5::smem_addr(&sm.full[i]), kLoaders / 32);
            tc5::mbar_init(tc5::smem_addr(&sm.empty[i]), (is_o ? kChain : kMain) / 32 + 1);
            tc5::mbar_init(tc5::smem_addr(&sm.xo[i]), is_o ? 1 + CD : 1);
            tc5::mbar_init(tc5::smem_addr(&sm.xd[i]), 1);
            tc5::mbar_init(tc5::smem_addr(&sm.vw[i]), 1);
            tc5::mbar_init(tc5::smem_addr(&sm.st[i]), (is_o ? kChain : kMain) / 32);
        }
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
        const int nk1 = sweep_count(n, b, 1);
        unsigned long long *betas = pr.betas + (size_t)(s & 1) * nk1, *betas_prev = pr.betas + (size_t)(~s & 1) * nk1;
        constexpr int words = sizeof(T) / 8;
        unsigned long long *firsts = pr.firsts + (size_t)(s & 1) * nk1 * b * words;
        unsigned long long *firsts_prev = pr.firsts + (size_t)(~s & 1) * nk1 * b * words;

        if (is_o && tid < kChain) {
            // ================= O, the chain: right product, column sums, reflector
            const int i0 = rank * RW;
            bool active = false;                      // H(s,k-1) is not the identity
            T ptau;
            zero_of(ptau);
            for (int k = 0; k < nk; k++, kk++) {
                const int par = kk & 1;
                T *B = stage + (kk % G::NO) * G::OBUF;
                if (tid == 0) mbar_expect(&sm.xo[par], G::O_BYTES);
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
                chain_sync();
                // the source column (the block's first) and row 0 as they are
                // now, then the column sums with the raw source column
                if (tid < RW * G::S)
                    send(&sm.mx[par][i0 + tid % RW], B[(tid % RW) * LD], &sm.xo[par], tid / RW);
                const int col = tid / G::TPC, cp = tid % G::TPC;
                if (rank == 0) {
                    const T a0 = B[col];
                    for (int d = cp; d < C; d += G::TPC) send(&sm.ma[par][col], a0, &sm.xo[par], d);
                    if (col == 0)
                        for (int d = cp; d < CD; d += G::TPC) send(&sm.ma[par][0], a0, &sm.xo[par], C + d);
                }
                constexpr int NE = 16 / G::TPC, NB8 = 8 / G::TPC;
#pragma unroll
                for (int g = 0; g < G::NGR; g++) {
                    T acc[NB8];
#pragma unroll
                    for (int u = 0; u < NB8; u++) zero_of(acc[u]);
#pragma unroll
                    for (int u = 0; u < NE; u++) {
                        const int i = 16 * g + cp + G::TPC * u;
                        if (i0 + i > 0) acc[u % NB8] = madc(B[i * LD], B[i * LD + col], acc[u % NB8]);
                    }
                    const T sum = tree_sum<8, G::TPC>(acc);
                    T *to = &sm.ms[par][rank * G::NGR + g][col];
                    for (int d = cp; d < C; d += G::TPC) send(to, sum, &sm.xo[par], d);
                    if (col == 0)
                        for (int d = cp; d < CD; d += G::TPC) send(to, sum, &sm.xo[par], C + d);
                }
                chase_wait(&sm.xo[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                // every rank: the reflector, and the sums over groups
                if (warp == 0) {
                    const auto h = reflector(sm.ma[par][0], group_sum<G::NG>(&sm.ms[par][0][0], BM));
                    if (lane == 0) {
                        sm.tau[par] = h.tau;
                        sm.scal[par] = h.scal;
                        // beta: final where k = 0 (the subdiagonal of T), else on
                        // to the next sweep, whose last entry of O(s+1,k-1) it is
                        if (rank == 0) {
                            if (k > 0) {
                                st_relaxed(betas + k, (unsigned long long)__double_as_longlong(h.beta));
                            } else {
                                T z;
                                zero_of(z);
                                *(double *)&z = h.beta;
                                *A.at(s, s - 1) = z;
                            }
                        }
                    }
                } else if (tid < 32 + BM) {
                    const int j = tid - 32;
                    T t2 = sm.ms[par][0][j];
                    for (int q = 1; q < G::NG; q++) t2 = add(t2, sm.ms[par][q][j]);
                    sm.sum[j] = t2;
                }
                chain_sync();
                const T tau = sm.tau[par], scal = sm.scal[par];
                if (tid < BM) {
                    T vi;
                    if (tid == 0) one_of(vi);
                    else vi = mul(sm.mx[par][tid], scal);   // scal = 0 where tau = 0; x = 0 past len
                    sm.v[par][tid] = vi;
                } else if (tid >= 64 && tid < 64 + BM) {
                    // w_j = conj(tau) v^H a_j
                    const int j = tid - 64;
                    sm.w[par][j] = mul(conj_of(tau), mad(conj_of(scal), sm.sum[j], sm.ma[par][j]));
                }
                chain_sync();
                if (tid == 0) mbar_arrive(&sm.vw[par]);
                active = !is_zero(tau);
                ptau = tau;
            }
        } else if (is_o && tid < kMain) {
            // ================= O, the finish: left product and stores, while
            // the chain is at the next block
            const int i0 = rank * RW, ft = tid - kChain;
            const int col = ft / G::TPC, cp = ft % G::TPC;
            for (int k = 0; k < nk; k++, kk++) {
                const int r = s + k * b, len = min(b, n - r);
                const int c = (k == 0) ? s - 1 : r - b;
                const int ncols = (k == 0) ? 1 : b;
                const int par = kk & 1;
                const T *B = stage + (kk % G::NO) * G::OBUF;
                chase_wait(&sm.vw[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                const bool act = !is_zero(sm.tau[par]);
                if (col < ncols) {
                    const T wj = sm.w[par][col];
#pragma unroll
                    for (int u = 0; u < RW / G::TPC; u++) {
                        const int i = cp + G::TPC * u, gi = i0 + i;
                        if (gi < len) {
                            const T e = B[i * LD + col];
                            // (the annihilated column stays unstored: its beta went its own
                            // way, and later sweeps know the zeros)
                            if (col > 0) *A.at(r + gi, c + col) = act ? nmad(sm.v[par][gi], wj, e) : e;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&sm.st[par]);
                    mbar_arrive(&sm.empty[kk % G::NO]);
                }
            }
        } else if (tid < kMain) {
            // ================= D: symmetric two-sided update
            const int dr = rank - C;
            const int rr = tid / G::TPD, part = tid % G::TPD;
            const int i = dr + CD * rr;                     // this thread's row of D
            // entry i of the first column: row 0 is the last entry of D(s+1,k-1),
            // the others the last column of O(s+1,k); D(s,0)'s first entry is final
            auto to_next = [&](int row, int k, T x) {
                if (row > 0 || k > 0) put_entry(firsts + (size_t)k * b * words, row, x);
                else *A.at(s, s) = x;
            };
            for (int k = 0; k < nk; k++, kk++) {
                const int r = s + k * b, len = min(b, n - r);
                const int par = kk & 1;
                const long long idx = first + k;
                const T *B = stage + (kk % G::ND) * G::DBUF;
                if (tid == 0) mbar_expect(&sm.xo[par], G::D_BYTES);
                chase_wait(&sm.full[kk % G::ND], (kk / G::ND) & 1, wait_ns, state, &sm.abort);
                chase_wait(&sm.xo[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                // D x over x's entries past the first, while the publisher warp
                // has the reflector's scalars: D v = D e_0 + scale D x
                constexpr int NA = 16 / G::TPD;
                T e[BM / G::TPD], acc[NA];
#pragma unroll
                for (int u = 0; u < NA; u++) zero_of(acc[u]);
#pragma unroll
                for (int u = 0; u < BM / G::TPD; u++) {
                    const int j = part + G::TPD * u;
                    e[u] = B[rr * LD + j];
                    if (j > 0) acc[u % NA] = mad(e[u], sm.mx[par][j], acc[u % NA]);
                }
                const T dx = tree_sum<16, G::TPD>(acc);
                scalars_take();
                const T tau = sm.tau[par], scal = sm.scal[par];
                const bool act = !is_zero(tau);
                if (tid < BM) {
                    T vi;
                    if (tid == 0) one_of(vi);
                    else vi = mul(sm.mx[par][tid], scal);
                    sm.v[0][tid] = vi;
                    if (dr == 0 && tid < b) ((T *)pr.hh_v)[idx * b + tid] = vi;
                }
                if (dr == 0 && tid == 64) ((T *)pr.hh_tau)[idx] = tau;
                const int pp = nxd & 1;
                if (act) {
                    if (CD > 1 && tid == 0) mbar_expect(&sm.xd[pp], G::P_BYTES);
                    const T pi = mul(tau, mad(scal, dx, B[rr * LD]));
                    if (CD == 1) {
                        if (part == 0) sm.mp[pp][i] = pi;
                    } else if (part < CD) {
                        send(&sm.mp[pp][i], pi, &sm.xd[pp], C + part);
                    }
                }
                main_sync();
                // the mailbox is consumed: credit for the O ranks' next step
                if (tid < C) mbar_arrive_remote(&sm.xo[par ^ 1], tid);
                if (act) {
                    if (CD > 1) chase_wait(&sm.xd[pp], (nxd >> 1) & 1, wait_ns, state, &sm.abort);
                    nxd++;
                    const T *v = sm.v[0];
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
                        if (j <= i) e[u] = nmad(vi, conj_of(sm.q[j]), nmad(qi, conj_of(v[j]), e[u]));
                        if (u == 0 && part == 0 && i < len) to_next(i, k, e[0]);
                    }
                    if (i < len)
#pragma unroll
                        for (int u = 0; u < BM / G::TPD; u++) {
                            const int j = part + G::TPD * u;
                            if (j > 0 && j <= i) *A.at(r + i, r + j) = e[u];
                        }
                } else if (part == 0 && i < len) {
                    to_next(i, k, e[0]);
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&sm.st[par]);
                    mbar_arrive(&sm.empty[kk % G::ND]);
                }
            }
        } else if (tid < kMain + kLoaders) {
            // ================= loaders: stage the next block
            const int lt = tid - kMain;
            for (int k = 0; k < nk; k++, kk++) {
                const int r = s + k * b, len = min(b, n - r);
                T *B = stage + (kk % nbuf) * bufsz;
                if (kk >= (uint32_t)nbuf)
                    chase_wait(&sm.empty[kk % nbuf], (kk / nbuf - 1) & 1, wait_ns, state, &sm.abort);
                // O(s,k): O(s-1,k), whose successor shares all but the last column
                // and row; D(s,k): D(s-1,k), and the first row of O(s-1,k+1)
                if (lt < 32 && s > 1 && !__any_sync(0xffffffffu, *(volatile int *)&sm.abort))
                    chase_flags<C, CD>(prev, min(is_o ? k + 1 : k + 2, nkp), is_o ? 0 : min(k + 1, nkp), timeout_ns, state,
                                       &sm.abort);
                loader_sync();
                if (is_o) {
                    const int i0 = rank * RW;
                    const int c = (k == 0) ? s - 1 : r - b;
                    const int ncols = (k == 0) ? 1 : b;
                    // from the band: all but the last column, which follows below,
                    // and the last row (zero up to there); the first sweep loads both
                    const int lcols = s > 1 ? ncols - 1 : ncols, lrows = s > 1 ? min(len, b - 1) : len;
                    // rows run along the band's contiguous index
                    constexpr int NU = RW * BM / kLoaders, CH = NU < 8 ? NU : 8;
#pragma unroll 1
                    for (int u0 = 0; u0 < NU; u0 += CH) {   // CH loads in flight per thread
                        T x[CH];
#pragma unroll
                        for (int u = 0; u < CH; u++) {
                            const int e = lt + kLoaders * (u0 + u), col = e / RW, i = e % RW;
                            zero_of(x[u]);
                            if (col < lcols && i0 + i < lrows) x[u] = ld_cg(A.at(r + i0 + i, c + col));
                        }
#pragma unroll
                        for (int u = 0; u < CH; u++) {
                            const int e = lt + kLoaders * (u0 + u), col = e / RW, i = e % RW;
                            B[i * LD + col] = x[u];
                        }
                    }
                    // the last column: the first column of D(s-1,k) from its
                    // second entry on, and the beta of H(s-1,k+1)
                    if (s > 1) {
                        loader_sync();
                        if (lt < RW && i0 + lt < len && !*(volatile int *)&sm.abort) {
                            T x;
                            zero_of(x);
                            if (i0 + lt == b - 1)
                                *(double *)&x = take(betas_prev + k + 1, timeout_ns, state, &sm.abort);
                            else
                                take_entry(x, firsts_prev + (size_t)k * b * words, i0 + lt + 1, timeout_ns, state, &sm.abort);
                            B[lt * LD + ncols - 1] = x;
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
                            const bool corner = s > 1 && j == b - 1;   // D(s-1,k+1)'s first entry: below
                            if (e < N2 && i < len && !corner) x[u] = ld_cg(A.at(r + i, r + j));   // j <= i
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
                    if (s > 1 && len == b && (b - 1) % CD == dr) {
                        loader_sync();
                        if (lt == 0 && !*(volatile int *)&sm.abort) {
                            T x;
                            take_entry(x, firsts_prev + (size_t)(k + 1) * b * words, 0, timeout_ns, state, &sm.abort);
                            B[((b - 1) / CD) * LD + b - 1] = x;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.full[kk % nbuf]);
            }
        } else {
            // ================= publisher warp: fences and flags; in D
            // blocks the reflector's scalars too
            for (int k = 0; k < nk; k++, kk++) {
                const int par = kk & 1;
                if (!is_o) {
                    chase_wait(&sm.xo[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                    const auto h = reflector(sm.ma[par][0], group_sum<G::NG>(&sm.ms[par][0][0], BM));
                    if (lane == 0) {
                        sm.tau[par] = h.tau;
                        sm.scal[par] = h.scal;
                    }
                    scalars_give();
                }
                if (lane == 0) {
                    chase_wait(&sm.st[par], (kk >> 1) & 1, wait_ns, state, &sm.abort);
                    // (the release orders the block's stores, seen through the
                    // barrier, before the flag)
                    if (!*(volatile int *)&sm.abort) st_rel(mine + rank, k + 1);
                    mbar_arrive(&sm.empty[kk % nbuf]);
                }
                __syncwarp();
            }
        }
    }
    __syncwarp();
    cluster.sync();   // no block leaves while a peer may still reach its shared memory
}

template <class T>
__global__ void __launch_bounds__(256) band_init(int n, int b, const T *__restrict__ AB, long long ldab,
                                                 T *__restrict__ W, long long ldw,
                                                 unsigned long long *__restrict__ slots, size_t nslots)
{
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nslots; e += (size_t)gridDim.x * blockDim.x)
        slots[e] = kEmpty;
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
// sweep][slots: 2 nk(1) betas, 2 nk(1) b entries of one or two words] then,
// 256-byte aligned, the 2b x n working band.
static size_t progress_bytes(int n) { return (256 + (size_t)n * kFlags * sizeof(int) + 255) & ~(size_t)255; }
static size_t slot_words(int n, int b, int words)
{
    const size_t nk1 = ((size_t)n + b - 1) / b;
    return 2 * nk1 + 2 * nk1 * b * words;
}
static size_t flags_bytes(int n, int b, int words)
{
    return progress_bytes(n) + ((slot_words(n, b, words) * 8 + 255) & ~(size_t)255);
}
static ChaseProblem chase_problem(int n, int b, int words, void *ws, void *hh_v, void *hh_tau)
{
    char *flags = (char *)ws;
    unsigned long long *slots = (unsigned long long *)(flags + progress_bytes(n));
    return ChaseProblem{n,      b,      flags + flags_bytes(n, b, words), 2LL * b, hh_v, hh_tau, (int *)(flags + 256), slots,
                        slots + 2 * (((size_t)n + b - 1) / b)};
}

size_t band_to_tridi_workspace_bytes(int n, int b)
{
    size_t band = 2 * (size_t)b * (size_t)n * sizeof(double);
    return flags_bytes(n, b, 1) + ((band + 255) & ~(size_t)255);
}

size_t band_to_tridi_workspace_bytes_z(int n, int b)
{
    size_t band = 2 * (size_t)b * (size_t)n * 2 * sizeof(double);
    return flags_bytes(n, b, 2) + ((band + 255) & ~(size_t)255);
}

// Sweeps that can be in flight at once: sweep s trails sweep s-1 by about two
// of its nk(1) steps; further clusters would only poll, holding SM slots that
// concurrent work on other streams could use (n = 2048: 17.8 ms with 16 clusters,
// 17.6 with 19, 19.7 with 30).
static int chase_active(int n, int b)
{
    const int nk1 = (n - 1 + b - 1) / b;
    return max(1, min(n - 1, (nk1 + 1) / 2 + 3));
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
// Real, b > 32: clusters of 6 (4 row parts of O, 2 of D) up to twice the
// sweeps that find SMs: n = 2048 17.6 ms against 22.8 with clusters of 3, 4096
// 42.5 against 46.0, 8192 99.8 against 124; beyond that (n = 16384) clusters of 3,
// which keep twice the sweeps in flight.  b <= 32 has a quarter of the work a
// step: clusters of 3; complex steps have four times the work: 6 from b = 33.
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
    if (active * 6 <= 4LL * sms) return chase_launch_as<double, 64, 4, 2>(work, active, sms, state, timeout_ns, st);
    return chase_launch_as<double, 64, 2, 1>(work, active, sms, state, timeout_ns, st);
}

static ChaseWork chase_one(const ChaseProblem &problem)
{
    ChaseWork w{};
    w.count = 1;
    w.smax = problem.n - 1;
    w.one = problem;
    return w;
}

cudaError_t band_to_tridi_prepare_z(int n, int b, const double *AB, int ldab, void *ws, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    char *flags = (char *)ws;
    Zc *W = (Zc *)(flags + flags_bytes(n, b, 2));
    cudaError_t err = cudaMemsetAsync(flags, 0, progress_bytes(n), st);
    if (err != cudaSuccess) return err;
    band_init<Zc><<<1024, 256, 0, st>>>(n, b, (const Zc *)AB, ldab, W, ldw,
                                        (unsigned long long *)(flags + progress_bytes(n)), slot_words(n, b, 2));
    return cudaGetLastError();
}

cudaError_t band_to_tridi_finish_z(int n, int b, const void *ws, double *d, double *e, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    const Zc *W = (const Zc *)((const char *)ws + flags_bytes(n, b, 2));
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
        const ChaseWork w = chase_one(chase_problem(n, b, 2, ws, hh_v, hh_tau));
        if ((err = chase_launch(w, chase_active(n, b), b, 1, (ChaseState *)flags, timeout_ns, st)) != cudaSuccess)
            return err;
    }
    return band_to_tridi_finish_z(n, b, ws, d, e, st);
}

cudaError_t band_to_tridi_prepare_d(int n, int b, const double *AB, int ldab, void *ws, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    char *flags = (char *)ws;
    double *W = (double *)(flags + flags_bytes(n, b, 1));
    cudaError_t err = cudaMemsetAsync(flags, 0, progress_bytes(n), st);
    if (err != cudaSuccess) return err;
    band_init<double><<<1024, 256, 0, st>>>(n, b, AB, ldab, W, ldw, (unsigned long long *)(flags + progress_bytes(n)), slot_words(n, b, 1));
    return cudaGetLastError();
}

cudaError_t band_to_tridi_finish_d(int n, int b, const void *ws, double *d, double *e, cudaStream_t st)
{
    const long long ldw = 2LL * b;
    const double *W = (const double *)((const char *)ws + flags_bytes(n, b, 1));
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
        const ChaseWork w = chase_one(chase_problem(n, b, 1, ws, hh_v, hh_tau));
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
                                                 int is_complex, cudaStream_t st)
{
    if (count < 1) return cudaSuccess;
    std::vector<ChaseProblem> host((size_t)count);
    for (int i = 0; i < count; i++) {
        host[i] = chase_problem(n[i], b[i], is_complex ? 2 : 1, ws[i], hh_v[i], hh_tau[i]);
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
