// FP64-accurate products on the tcgen05 tensor cores: the eight-digit form of
// dgemm_sliced.cuh, C = alpha A B^T + beta C for operands cut into balanced
// base-256 FP16 digit planes.
//
// Scheme: each entry is a 64-bit fixed-point value against its row's power of
// two (|x| <= 2^62), cut into eight digits d_s in [-128, 127], exact in FP16.
// The 36 digit pairs s + t <= 7 accumulate in FP32, one accumulator per level
// l = s + t, over at most 128 values of k: (l + 1) 128 2^14 <= 2^24, so every
// sum is exact.  The dropped levels, the first of them seven pairs of up to
// 2^14 a value of k, lie below 7.1 k 2^-62 of the row maxima's product; with digits
// of random signs about 2^-62 sqrt(k), where 56-bit digits left 2^-57 sqrt(k).
//
// One CTA owns a 128 x 64 tile of C: 8 levels x 64 columns of FP32 fill the
// 512 columns of tensor memory.  One MMA per A plane s and half of the levels:
// its B operand spans the planes t that land there along N (planes follow each
// other in shared memory at one 8-row stride), 12 MMAs per K step of 16.
//   * The levels are worked on in two halves, 0-3 and 4-7.  In the last 32
//     values of k of a group of 128 the low half is issued first, so that it
//     is folded while the high half multiplies; the high half is folded while
//     the next group's low half multiplies.
//   * Operands lie in global memory in blocks of 128 rows x 32 k, 64 KB, in
//     the order of the MMA's canonical K-major layout (no swizzle), so a stage
//     is one bulk copy for A and eight (one 4 KB piece per plane) for B; two
//     stages of 96 KB.
//   * 8 warps fold levels into a 96-bit integer per entry and write C; one
//     warp copies, one issues MMAs.  The grid is persistent: the next tile's
//     MMAs run under this tile's epilogue.
//   * The epilogue assembles the FP64 result with integer operations, rounded
//     once (two FP64 lanes per clock and SM would make conversions in FP64 as
//     long as the MMAs of a whole group); only alpha and beta other than +-1,
//     0 cost FP64 operations, beta = 1 one addition.
//
// What bounds it: 36 x 2 m n k FP16 flops at the tensor rate for long k; HBM
// traffic of C and of the digit planes (16 bytes per entry) for k <= 128.
// Measured on a GB300 (whole calls, slicing included; before: the same scheme
// on bf16 mma.sync, 43 pairs of 7-bit digits): 8192^3 139.8 -> 22.8 ms (48.2
// TFLOP/s of FP64, 0.90 of the tensor rate over 36), 4096^3 17.9 -> 3.2 ms,
// 3001 x 1777 x 4099 6.14 -> 1.29 ms; the n = 16320 panel products of a
// solver: symmetric x 64 columns 9.0 -> 2.3 ms (1.4 of it slicing, HBM-bound),
// rank-128 update 7.9 -> 1.8 ms; 64 x 4096, k = 16384 2.3 -> 0.78 ms.  Error
// against 64-bit references 1.2e-15 to 3.0e-15, as before.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "dgemm_sliced.cuh"
#include "elpa_gb300.h"
#include "mma_bf16.cuh"
#include "slice_views.cuh"
#include "tcgen05.cuh"

namespace gb {

namespace {

constexpr int kTM = 128, kTN = 64, kTK = 32;   // tile of C, and k of a stage
constexpr int kGroup = 4;                      // stages per exact sum: 128 values of k
constexpr int kPl = 8;                         // digit planes
constexpr uint32_t kPlaneBytes = kTM * kTK * 2;          // a plane of a block: 8 KB
constexpr uint32_t kBlockBytes = kPl * kPlaneBytes;      // a 128 x 32 block: 64 KB
constexpr uint32_t kBPlane = kTN * kTK * 2;              // the B tile's part of a plane: 4 KB
constexpr uint32_t kStageBytes = kBlockBytes + kPl * kBPlane;
constexpr uint32_t kSbo = kTK / 8 * 128;                 // bytes between 8-row groups
constexpr int kFoldWarps = 8;                  // two per lane quarter, kCols columns each
constexpr int kCols = kTN / (kFoldWarps / 4);
constexpr int kThreads5 = (kFoldWarps + 4) * 32; // copies, MMAs, two idle warps (registers are dealt by fours)
constexpr size_t kSmem5 = 2 * (size_t)kStageBytes + 1024;
constexpr long long kWaitNs = 4000000000ll;
constexpr unsigned long long kBias = 0x8080808080808080ull;

// round(x 2^(62 - e)) for |x| < 2^e, to nearest, from the bit pattern
__device__ __forceinline__ long long fixed62(double x, int e)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((u >> 52) & 0x7ff);
    if (ex == 0) return 0;                              // subnormals read as zero
    const unsigned long long M = (u & 0xfffffffffffffull) | (1ull << 52);
    const int sh = ex - 1075 + 62 - e;                  // at most 9
    unsigned long long r;
    if (sh >= 0) r = M << sh;
    else if (sh > -54) r = (M + (1ull << (-sh - 1))) >> -sh;
    else r = 0;
    return (u >> 63) ? -(long long)r : (long long)r;
}

// FP16 pair of the balanced digits in byte bi of a and b (biased bytes):
// 0x6400 | m is 1024 + m, minus 1152
__device__ __forceinline__ uint32_t digits_of(uint32_t a, uint32_t b, int bi)
{
    const uint32_t sel = (uint32_t)bi | ((uint32_t)bi << 4) | ((uint32_t)(4 + bi) << 8) | ((uint32_t)(4 + bi) << 12);
    const uint32_t r = (__byte_perm(a, b, sel) & 0x00ff00ffu) | 0x64006400u;
    const __half2 h = __hsub2(*(const __half2 *)&r, __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480)));
    return *(const uint32_t *)&h;
}

// Row exponent from the high word of the row's largest magnitude (0 for rows
// of zeros and subnormals, which read as zero).  A row with a NaN or an infinity
// gets an exponent far beyond the others: its digits are zeros, and the epilogue
// knows its results for NaN.
constexpr int kNonFinite = 1 << 20;
__device__ __forceinline__ int exponent_of(uint32_t hi)
{
    return hi >= 0x7ff00000u ? kNonFinite : (hi >> 20) ? (int)(hi >> 20) - 1022 : 0;
}

__device__ __forceinline__ uint32_t abs_hi(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// Digits of a 32 x 32 tile at (r0, k0), entry (r, k) at t[r * sr + k * sk]:
// 128 threads (`tid`), thread (r, q) cuts eight consecutive k and stores 16
// bytes per plane; a plane's part of the tile is 2 KB contiguous.
__device__ __forceinline__ void cut_tile(int tid, const double *t, int sr, int sk, int r0, int k0, int rows, int KC,
                                         int e, unsigned char *__restrict__ planes)
{
    // consecutive threads: the 8 rows of a core matrix, then its neighbour along k
    const int g = tid >> 5, q = (tid >> 3) & 3, r = (g << 3) | (tid & 7);
    const int row = r0 + r;
    if (row >= rows) return;
    uint32_t w[kPl][4];
#pragma unroll
    for (int p = 0; p < 4; p++) {
        const unsigned long long y0 = (unsigned long long)fixed62(t[r * sr + (q * 8 + 2 * p) * sk], e) + kBias;
        const unsigned long long y1 = (unsigned long long)fixed62(t[r * sr + (q * 8 + 2 * p + 1) * sk], e) + kBias;
#pragma unroll
        for (int s = 0; s < 4; s++) w[s][p] = digits_of((uint32_t)(y0 >> 32), (uint32_t)(y1 >> 32), 3 - s);
#pragma unroll
        for (int s = 4; s < 8; s++) w[s][p] = digits_of((uint32_t)y0, (uint32_t)y1, 7 - s);
    }
    unsigned char *base = planes + ((size_t)(row >> 7) * KC + (k0 >> 5)) * kBlockBytes +
                          (size_t)((row & 127) >> 3) * kSbo + q * 128 + (row & 7) * 16;
#pragma unroll
    for (int s = 0; s < kPl; s++) *(uint4 *)(base + s * kPlaneBytes) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

__device__ __forceinline__ int cut_row(int tid) { return ((tid >> 5) << 3) | (tid & 7); }

// High words of the row maxima, 32 rows x `span` values of k a block.
__global__ void __launch_bounds__(256) tc5_rowmax(int view, const double *__restrict__ src, long long ld, int R, int K,
                                                  int span, uint32_t *__restrict__ rmax)
{
    __shared__ uint32_t red[8][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int r0 = blockIdx.y * 32, kb = blockIdx.x * span, ke = min(K, kb + span);
    if (view == kViewRow || view == kViewZExpandN || view == kViewZRowConj) {   // r runs along memory
        uint32_t m = 0;
        if (r0 + tx < R)
            for (int k = kb + ty; k < ke; k += 8) m = max(m, abs_hi(view_at(view, src, ld, r0 + tx, k)));
        red[ty][tx] = m;
        __syncthreads();
        if (ty == 0) {
            for (int i = 1; i < 8; i++) m = max(m, red[i][tx]);
            if (r0 + tx < R && m) atomicMax(rmax + r0 + tx, m);
        }
    } else if (view == kViewSym) {
        // the stored triangle only: an entry counts for its row and its column
        uint32_t m = 0;
        if (kb <= r0 + 31)
            for (int k = kb + ty; k < min(ke, r0 + 32); k += 8) {
                const int r = r0 + tx;
                const uint32_t v = (r < R && r >= k) ? abs_hi(src[r + (long long)k * ld]) : 0u;
                m = max(m, v);
                const uint32_t c = __reduce_max_sync(0xffffffffu, v);
                if (tx == 0 && c) atomicMax(rmax + k, c);
            }
        red[ty][tx] = m;
        __syncthreads();
        if (ty == 0) {
            for (int i = 1; i < 8; i++) m = max(m, red[i][tx]);
            if (r0 + tx < R && m) atomicMax(rmax + r0 + tx, m);
        }
    } else {
        for (int i = ty; i < 32; i += 8) {
            const int r = r0 + i;
            uint32_t m = 0;
            if (r < R)
                for (int k = kb + tx; k < ke; k += 32) m = max(m, abs_hi(view_at(view, src, ld, r, k)));
            m = __reduce_max_sync(0xffffffffu, m);
            if (tx == 0 && r < R && m) atomicMax(rmax + r, m);
        }
    }
}

// Digits of 32 rows x `chunks` chunks of 32 k a block, the row maxima known.  A
// symmetric view reads each stored tile once and writes it and its mirror image.
__global__ void __launch_bounds__(256) tc5_slice(int view, const double *__restrict__ src, long long ld, int R, int K,
                                                 int rows, int KC, int chunks, const uint32_t *__restrict__ rmax,
                                                 unsigned char *__restrict__ planes, int *__restrict__ e_out)
{
    __shared__ double t[32][33];
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int r0 = blockIdx.y * 32;
    if (blockIdx.x == 0 && tid < 32) e_out[r0 + tid] = r0 + tid < R ? exponent_of(rmax[r0 + tid]) : 0;
    for (int c = 0; c < chunks; c++) {
        const int k0 = (blockIdx.x * chunks + c) * 32;
        if (k0 >= KC * 32 || (view == kViewSym && k0 > r0)) break;
        load_tile(view, src, ld, R, K, r0, k0, t);
        __syncthreads();
        if (view == kViewSym) {
            const int half = tid & 127, i = cut_row(half);
            if (tid < 128) {
                cut_tile(half, &t[0][0], 33, 1, r0, k0, rows, KC, r0 + i < R ? exponent_of(rmax[r0 + i]) : 0, planes);
            } else if (k0 != r0) {
                cut_tile(half, &t[0][0], 1, 33, k0, r0, rows, KC, k0 + i < R ? exponent_of(rmax[k0 + i]) : 0, planes);
            }
        } else if (tid < 128) {
            const int i = cut_row(tid);
            cut_tile(tid, &t[0][0], 33, 1, r0, k0, rows, KC, r0 + i < R ? exponent_of(rmax[r0 + i]) : 0, planes);
        }
        __syncthreads();
    }
}

// Short rows (K <= 160): a block takes all k of its 32 rows, maxima first,
// then digits (the second read comes from L2): one launch instead of three.
// The view is a template argument: a short kernel's time is latency, and a
// switch per load adds to it (A^T B of 100 x 100 x 100 51.7 -> 43.6 us a call).
template <int view>
__global__ void __launch_bounds__(256) tc5_slice_rows(const double *__restrict__ src, long long ld, int R, int K,
                                                      int rows, int KC, unsigned char *__restrict__ planes,
                                                      int *__restrict__ e_out)
{
    __shared__ double t[2][32][33];
    __shared__ uint32_t red[8][33];
    __shared__ int ex[32];
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 32 + tx;
    const int r0 = blockIdx.x * 32;
    uint32_t m = 0;
    if (view == kViewRow || view == kViewZExpandN || view == kViewZRowConj) {
        if (r0 + tx < R)
            for (int k = ty; k < K; k += 8) m = max(m, abs_hi(view_at(view, src, ld, r0 + tx, k)));
        red[ty][tx] = m;
        __syncthreads();
        if (ty == 0) {
            for (int i = 1; i < 8; i++) m = max(m, red[i][tx]);
            ex[tx] = exponent_of(m);
        }
    } else {
        uint32_t row[4] = {0, 0, 0, 0};   // (all rows' loads before the first reduction)
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (r0 + ty + 8 * q < R)
                for (int k = tx; k < K; k += 32) row[q] = max(row[q], abs_hi(view_at(view, src, ld, r0 + ty + 8 * q, k)));
#pragma unroll
        for (int q = 0; q < 4; q++) {
            m = __reduce_max_sync(0xffffffffu, row[q]);
            if (tx == 0) ex[ty + 8 * q] = exponent_of(m);
        }
    }
    __syncthreads();
    if (tid < 32) e_out[r0 + tid] = ex[tid];
    // two tiles at a time, 128 threads each
    for (int c = 0; c < KC; c += 2) {
        load_tile(view, src, ld, R, K, r0, c * 32, t[0]);
        if (c + 1 < KC) load_tile(view, src, ld, R, K, r0, (c + 1) * 32, t[1]);
        __syncthreads();
        const int h = tid >> 7;
        if (c + h < KC) cut_tile(tid & 127, &t[h][0][0], 33, 1, r0, (c + h) * 32, rows, KC, ex[cut_row(tid & 127)], planes);
        __syncthreads();
    }
}

// ---- the product ------------------------------------------------------------

struct ProductArgs {
    const unsigned char *A, *B;   // digit blocks: A rows are the MMA's M, B rows its N
    const int *ea, *eb;
    int KC;                       // 32-wide k chunks of both
    int m, n;                     // rows of A and of B used
    int tiles_m, tiles_n, splits, kc_split;
    long long tiles;              // tiles of C worked on, times splits
    double alpha, beta;
    double *C;
    long long ldc;
    int fill, swapped;            // swapped: entry (row of A, row of B) is C(row of B, row of A)
    double *part;                 // split-K partials (C's orientation, leading dimension rows of C)
    int *status;                  // null, or receives GB_ERR_TIMEOUT when a wait gives up
    long long wait_ns;            // limit of the waits
    uint32_t hold;                // for tests: a block's copies end after this many stages
};

struct Tile {
    int tm, tn, kc0, kc1, split;
};

// Tile number t of the launch.  All of C: supergroups of 16 row tiles,
// columns within, so that the tiles in flight share operand blocks in L2.
// Lower triangles: row by row (row tile i has 2i + 2 column tiles, Hermitian
// forms i + 1, the last row's perhaps cut off).
__device__ __forceinline__ Tile tile_of(const ProductArgs &p, long long t)
{
    const long long per = p.tiles / p.splits;
    Tile x;
    x.split = (int)(t / per);
    const int u = (int)(t - x.split * per);
    if (p.fill == kFillAll) {
        const int sg = u / (16 * p.tiles_n), first = sg * 16;
        const int rows = min(16, p.tiles_m - first), v = u - sg * 16 * p.tiles_n;
        x.tn = v / rows;
        x.tm = first + v % rows;
    } else {
        const long long f = p.fill == kFillLower ? 1 : 2;   // tiles before row i: i (i + 1) / f
        long long i = (long long)((sqrtf(1.0f + 4.0f * (float)f * (float)u) - 1.0f) * 0.5f);
        while (i > 0 && i * (i + 1) / f > u) i--;
        while ((i + 1) * (i + 2) / f <= u) i++;
        x.tm = (int)i;
        x.tn = (int)(u - i * (i + 1) / f);
    }
    x.kc0 = x.split * p.kc_split;
    x.kc1 = min(p.KC, x.kc0 + p.kc_split);
    return x;
}

struct Tc5Sync {
    unsigned long long full[2], empty[2], ready[2], freed[2];   // ready/freed: low and high levels
    uint32_t tmem;
    int abort;
};

__device__ __forceinline__ bool wait5(const unsigned long long *bar, uint32_t parity, Tc5Sync &sy, long long wait_ns)
{
    if (tc5::mbar_wait(tc5::smem_addr(bar), parity & 1, wait_ns)) return true;
    *(volatile int *)&sy.abort = 1;
    return false;
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ int f2i(uint32_t f) { return __float2int_rn(__uint_as_float(f)); }

// FP64 value of the 96-bit integer hi 2^32 + lo times 2^e, rounded once (ties
// to even), without branches so that several columns' chains interleave.
// *odd is set where the result is not normal (and not zero): scaled_odd then.
__device__ __forceinline__ double assemble(long long hi, uint32_t lo, int e, bool *odd)
{
    const uint32_t neg = (uint32_t)(hi >> 63);              // all ones for a negative value
    const uint32_t l = (lo ^ neg) - neg;
    unsigned long long h = (unsigned long long)(hi ^ (hi >> 63)) + ((neg && l == 0) ? 1 : 0);
    // leading bits to the top of 64, a mark for anything below them
    const bool small = (h >> 32) == 0;
    h = small ? (h << 32) | l : h;
    const uint32_t below = small ? 0u : l;
    const int z = __clzll((long long)h) & 63;               // at most 31 unless small
    const uint32_t rest = __funnelshift_l(0u, below, z);    // below << z (z <= 31)
    const uint32_t up = __funnelshift_l(below, 0u, z);      // below >> (32 - z), 0 for z = 0
    unsigned long long top = (h << z) | up | (rest != 0 ? 1u : 0u);
    const bool zero = h == 0;
    const uint32_t low = (uint32_t)top & 0x7ffu;
    unsigned long long mant = top >> 11;                    // 53 bits
    mant += (low + ((uint32_t)mant & 1u)) > 0x400u ? 1 : 0;
    // value = mant 2^(43 - z + e), 32 less where small; biased exponent of mant
    const int field = 43 - z + e - (small ? 32 : 0) + 1075;
    *odd = !zero && (field < 1 || field >= 2046);
    unsigned long long bits = ((unsigned long long)(uint32_t)(field - 1) << 52) + mant;
    bits = zero ? 0ull : bits;
    return __longlong_as_double((long long)(bits | ((unsigned long long)(neg & 0x80000000u) << 32)));
}

// The same by scalings, for results outside the normal range.  The integer is
// below 2^96 and e = ea + eb - 68 may go down to -2112, past the two factors of
// scale_by_pow2: from e = -1300 on every result is a zero (of its sign).
__device__ __noinline__ double scaled_odd(long long hi, uint32_t lo, int e)
{
    return scale_by_pow2((double)hi * 4294967296.0 + (double)lo, max(e, -1300));
}

__global__ void __launch_bounds__(kThreads5, 1) tc5_product(const ProductArgs p)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ Tc5Sync sy;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        sy.abort = 0;
        for (int i = 0; i < 2; i++) {
            tc5::mbar_init(tc5::smem_addr(&sy.full[i]), 1);
            tc5::mbar_init(tc5::smem_addr(&sy.empty[i]), 1);
            tc5::mbar_init(tc5::smem_addr(&sy.ready[i]), 1);
            tc5::mbar_init(tc5::smem_addr(&sy.freed[i]), kFoldWarps);
        }
        tc5::mbar_init_fence();
    }
    if (warp == 0) tc5::tmem_alloc(tc5::smem_addr(&sy.tmem), 512);
    tc5::fence_before_sync();
    __syncthreads();
    tc5::fence_after_sync();
    const uint32_t tmem = *(volatile uint32_t *)&sy.tmem;

    // registers: 168 a thread at launch (3 warpgroups, 504 in all); the two
    // folding warpgroups take 216 each, the third keeps 56
    if (warp >= kFoldWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == kFoldWarps) {
            // ---- copies
            if (lane == 0) {
                uint32_t q = 0;
                bool ok = true;
                for (long long t = blockIdx.x; ok && t < p.tiles; t += gridDim.x) {
                    const Tile x = tile_of(p, t);
                    const unsigned char *ga = p.A + ((size_t)x.tm * p.KC) * kBlockBytes;
                    const unsigned char *gb_ = p.B + ((size_t)(x.tn >> 1) * p.KC) * kBlockBytes + (x.tn & 1) * kBPlane;
                    for (int kc = x.kc0; kc < x.kc1; kc++, q++) {
                        const int st = q & 1;
                        if (q == p.hold || (q >= 2 && !wait5(&sy.empty[st], (q >> 1) - 1, sy, p.wait_ns))) {
                            ok = false;
                            break;
                        }
                        const uint32_t bar = tc5::smem_addr(&sy.full[st]);
                        const uint32_t sa = tc5::smem_addr(smem + st * kStageBytes);
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kStageBytes)
                                     : "memory");
                        bulk_copy(sa, ga + (size_t)kc * kBlockBytes, kBlockBytes, bar);
#pragma unroll
                        for (int s = 0; s < kPl; s++)
                            bulk_copy(sa + kBlockBytes + s * kBPlane, gb_ + (size_t)kc * kBlockBytes + s * kPlaneBytes, kBPlane,
                                      bar);
                    }
                }
                // no copy may be in flight when the block leaves
                for (uint32_t i = q < 2 ? 0 : q - 2; i < q; i++)
                    tc5::mbar_wait(tc5::smem_addr(&sy.full[i & 1]), (i >> 1) & 1, kWaitNs);
            }
        } else if (warp == kFoldWarps + 1) {
            // ---- MMAs (the warp together, an elected lane issuing: see tcgen05.cuh)
            {
                uint32_t q = 0, grp = 0;
                bool ok = true;
                auto wait_all = [&](auto *bar, uint32_t n) { return __all_sync(0xffffffffu, wait5(bar, n, sy, p.wait_ns)) != 0; };
                auto mmas = [&](uint32_t st, bool high, bool first) {
                    if (!tc5::elect_one()) return;
                    const uint32_t sa = tc5::smem_addr(smem + st * kStageBytes);
                    const uint64_t da = tc5::smem_desc(sa, 128, kSbo), db = tc5::smem_desc(sa + kBlockBytes, 128, kSbo);
#pragma unroll
                    for (int ks = 0; ks < kTK / 16; ks++) {
#pragma unroll
                        for (int s = 0; s < kPl; s++) {
                            // levels [4 high, 4 high + 4): planes t0 .. t1 of B
                            const int t0 = high ? (s < 4 ? 4 - s : 0) : 0, t1 = high ? 7 - s : 3 - s;
                            if (t1 < t0) continue;
                            const uint64_t a = da + (uint64_t)((s * kPlaneBytes + ks * 256) >> 4);
                            const uint64_t b = db + (uint64_t)((t0 * kBPlane + ks * 256) >> 4);
                            // s = 0 writes all four levels of a half first
                            tc5::mma_smem_a(tmem + kTN * (s + t0), a, b, tc5::idesc_f16_f32(kTM, kTN * (t1 - t0 + 1)),
                                            (first && ks == 0 && s == 0) ? 0u : 1u);
                        }
                    }
                };
                for (long long t = blockIdx.x; ok && t < p.tiles; t += gridDim.x) {
                    const Tile x = tile_of(p, t);
                    for (int kc = x.kc0; ok && kc < x.kc1; kc += kGroup, grp++) {
                        const int ns = min(kGroup, x.kc1 - kc), first = min(ns, 2);
                        if (grp > 0 && !wait_all(&sy.freed[0], grp - 1)) { ok = false; break; }
                        tc5::fence_after_sync();
                        for (int c = 0; c < first && ok; c++) {
                            if (!wait_all(&sy.full[(q + c) & 1], (q + c) >> 1)) { ok = false; break; }
                            tc5::fence_after_sync();
                            mmas((q + c) & 1, false, c == 0);
                            __syncwarp();
                            if (c == ns - 1 && tc5::elect_one()) tc5::commit(tc5::smem_addr(&sy.ready[0]));
                        }
                        if (!ok) break;
                        if (grp > 0 && !wait_all(&sy.freed[1], grp - 1)) { ok = false; break; }
                        tc5::fence_after_sync();
                        for (int c = 0; c < first; c++) {
                            mmas((q + c) & 1, true, c == 0);
                            __syncwarp();
                            if (tc5::elect_one()) tc5::commit(tc5::smem_addr(&sy.empty[(q + c) & 1]));
                        }
                        for (int c = first; c < ns; c++) {
                            if (!wait_all(&sy.full[(q + c) & 1], (q + c) >> 1)) { ok = false; break; }
                            tc5::fence_after_sync();
                            mmas((q + c) & 1, false, false);
                            __syncwarp();
                            if (c == ns - 1 && tc5::elect_one()) tc5::commit(tc5::smem_addr(&sy.ready[0]));
                            mmas((q + c) & 1, true, false);
                            __syncwarp();
                            if (tc5::elect_one()) tc5::commit(tc5::smem_addr(&sy.empty[(q + c) & 1]));
                        }
                        if (!ok) break;
                        if (tc5::elect_one()) tc5::commit(tc5::smem_addr(&sy.ready[1]));
                        q += ns;
                    }
                }
                // every MMA is complete before tensor memory is given back: the
                // fold warps have waited for the last group; after a failure,
                // wait here (bounded)
                if (!ok) {
                    if (tc5::elect_one()) tc5::commit(tc5::smem_addr(&sy.empty[q & 1]));
                    for (long long i = 0; i < 100000; i++) __nanosleep(100);
                }
            }
        }
    } else {
        // ---- folds and the epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int quarter = warp & 3, c0 = (warp >> 2) * kCols;
        const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16) + c0;
        uint32_t grp = 0;
        bool bad = false;   // a wait gave up: this tile and the block's later ones are NaN
        for (long long t = blockIdx.x; t < p.tiles; t += gridDim.x) {
            const Tile x = tile_of(p, t);
            long long hi[kCols];
            uint32_t lo[kCols];
#pragma unroll
            for (int j = 0; j < kCols; j++) {
                hi[j] = 0;
                lo[j] = 0;
            }
            const int r = x.tm * kTM + quarter * 32 + lane, cb = x.tn * kTN + c0;
            const bool sw = p.swapped != 0;
            const long long rs = sw ? p.ldc : 1, cs = sw ? 1 : p.ldc;
            auto wanted = [&](int c) {
                return r < p.m && c < p.n && !(p.fill == kFillLower && r < c) && !(p.fill == kFillZLower && (r >> 1) < c);
            };
            // C's old entries, on their way while the tensor cores work
            double old[kCols];
#pragma unroll
            for (int j = 0; j < kCols; j++) old[j] = 0.0;
            // (a tile wholly inside C needs no tests, and its loads go out together)
            const bool inside = (x.tm + 1) * kTM <= p.m && (x.tn + 1) * kTN <= p.n &&
                                (p.fill == kFillAll || (p.fill == kFillLower && x.tm * kTM >= (x.tn + 1) * kTN) ||
                                 (p.fill == kFillZLower && x.tm * (kTM / 2) >= (x.tn + 1) * kTN));
            if (!p.part && p.beta != 0.0) {
                const double *src = p.C + r * rs + cb * cs;
                if (inside) {
#pragma unroll
                    for (int j = 0; j < kCols; j++) old[j] = __ldcg(src + j * cs);
                } else {
#pragma unroll
                    for (int j = 0; j < kCols; j++)
                        if (wanted(cb + j)) old[j] = src[j * cs];
                }
            }
            for (int kc = x.kc0; kc < x.kc1 && !bad; kc += kGroup, grp++) {
                wait5(&sy.ready[0], grp, sy, p.wait_ns);
                tc5::fence_after_sync();
#pragma unroll
                for (int h = 0; h < kCols / 8; h++) {
                    uint32_t a[4][8];
#pragma unroll
                    for (int l = 0; l < 4; l++) tc5::ld_x8(tl + kTN * l + 8 * h, a[l]);
                    tc5::wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        // L0 2^8 + L1 below 2^30, L2 2^8 + L3 below 2^31
                        const int p0 = f2i(a[0][j]) * 256 + f2i(a[1][j]), p1 = f2i(a[2][j]) * 256 + f2i(a[3][j]);
                        hi[8 * h + j] += (long long)p0 * 65536 + p1;
                    }
                }
                tc5::fence_before_sync();
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc5::smem_addr(&sy.freed[0])) : "memory");
                wait5(&sy.ready[1], grp, sy, p.wait_ns);
                tc5::fence_after_sync();
#pragma unroll
                for (int h = 0; h < kCols / 8; h++) {
                    uint32_t a[4][8];
#pragma unroll
                    for (int l = 0; l < 4; l++) tc5::ld_x8(tl + kTN * (4 + l) + 8 * h, a[l]);
                    tc5::wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        long long s = (long long)f2i(a[0][j]) * 256 + f2i(a[1][j]);
                        s = s * 65536 + ((long long)f2i(a[2][j]) * 256 + f2i(a[3][j]));
                        s += lo[8 * h + j];
                        lo[8 * h + j] = (uint32_t)s;
                        hi[8 * h + j] += s >> 32;
                    }
                }
                tc5::fence_before_sync();
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc5::smem_addr(&sy.freed[1])) : "memory");
                bad = *(volatile int *)&sy.abort != 0;
            }
            // entry (r, c) of A B^T times 2^(ea + eb - 68)
            const int er = r < p.m ? p.ea[r] - 68 : 0;
            double *out = p.C + r * rs;
            long long ocs = cs;
            if (p.part) {   // split-K: C's orientation, leading dimension its rows
                const long long rows = sw ? p.n : p.m;
                out = p.part + (size_t)x.split * p.m * p.n + (sw ? r * rows : (long long)r);
                ocs = sw ? 1 : rows;
            }
#pragma unroll
            for (int h = 0; h < kCols / 8; h++) {
                double v[8];
                bool any = false;
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    bool odd;
                    const int c = cb + 8 * h + j;
                    const int e = er + __ldg(p.eb + min(c, p.n - 1));
                    v[j] = assemble(hi[8 * h + j], lo[8 * h + j], e, &odd);
                    any |= odd || e > kNonFinite / 2;
                }
                if (any) {
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        bool odd;
                        const int e = er + __ldg(p.eb + min(cb + 8 * h + j, p.n - 1));
                        assemble(hi[8 * h + j], lo[8 * h + j], e, &odd);
                        if (odd) v[j] = scaled_odd(hi[8 * h + j], lo[8 * h + j], e);
                        // (alpha = 0 asks for no product)
                        if (e > kNonFinite / 2) v[j] = p.alpha == 0.0 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
                    }
                }
                if (bad) {
#pragma unroll
                    for (int j = 0; j < 8; j++) v[j] = __longlong_as_double(0x7ff8000000000000ll);
                }
                if (!p.part) {
                    if (p.alpha == -1.0) {
#pragma unroll
                        for (int j = 0; j < 8; j++) v[j] = -v[j];
                    } else if (p.alpha != 1.0) {
#pragma unroll
                        for (int j = 0; j < 8; j++) v[j] *= p.alpha;
                    }
                    if (p.beta == 1.0) {
#pragma unroll
                        for (int j = 0; j < 8; j++) v[j] += old[8 * h + j];
                    } else if (p.beta != 0.0) {
#pragma unroll
                        for (int j = 0; j < 8; j++) v[j] = fma(p.beta, old[8 * h + j], v[j]);
                    }
                }
                if (inside) {
#pragma unroll
                    for (int j = 0; j < 8; j++) out[(cb + 8 * h + j) * ocs] = v[j];
                } else {
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int c = cb + 8 * h + j;
                        if (p.fill == kFillZLower && (r >> 1) == c && (r & 1)) v[j] = 0.0;   // Hermitian diagonal
                        if (wanted(c)) out[c * ocs] = v[j];
                    }
                }
            }
        }
    }
    tc5::fence_before_sync();
    __syncthreads();
    if (tid == 0 && sy.abort && p.status) atomicExch(p.status, GB_ERR_TIMEOUT);
    if (warp == 0) {
        tc5::fence_after_sync();
        tc5::tmem_dealloc(tmem, 512);
    }
}

}  // namespace

size_t tc5_planes_bytes(int R, int K)
{
    const size_t Rb = ((size_t)(R > 0 ? R : 1) + kTM - 1) / kTM, KC = ((size_t)(K > 0 ? K : 1) + kTK - 1) / kTK;
    return Rb * KC * kBlockBytes;
}

int tc5_rows_padded(int R) { return (std::max(R, 1) + kTM - 1) / kTM * kTM; }

cudaError_t tc5_slice_matrix(SliceView view, int R, int K, const double *src, long long ld, uint32_t *rmax,
                             uint16_t *planes, int *e, cudaStream_t st)
{
    const int KC = (std::max(K, 1) + kTK - 1) / kTK;
    // rows past R are never needed: they only meet outputs that are not stored
    const int rows = (std::max(R, 1) + 31) / 32 * 32;
    const dim3 block(32, 8);
    // one launch where a block's rows are short (10 us for 512 blocks at K = 64;
    // 33 us at K = 512, where the three launches of the tiled form are faster)
    if (K <= 160 && view != kViewSym) {
        auto run = [&](auto kernel) {
            kernel<<<rows / 32, block, 0, st>>>(src, ld, R, K, rows, KC, (unsigned char *)planes, e);
        };
        switch (view) {
        case kViewRow: run(tc5_slice_rows<kViewRow>); break;
        case kViewCol: run(tc5_slice_rows<kViewCol>); break;
        case kViewZExpandN: run(tc5_slice_rows<kViewZExpandN>); break;
        case kViewZExpandC: run(tc5_slice_rows<kViewZExpandC>); break;
        case kViewZHermExpand: run(tc5_slice_rows<kViewZHermExpand>); break;
        default: run(tc5_slice_rows<kViewZRowConj>); break;
        }
        return cudaGetLastError();
    }
    cudaError_t err = cudaMemsetAsync(rmax, 0, (size_t)rows * sizeof(uint32_t), st);
    if (err != cudaSuccess) return err;
    // A block's chunks of k are a chain of loads, so they go to blocks of their
    // own until other blocks hide the chain, at about 32 blocks an SM.  Symmetric
    // n x n times 64 columns, one chunk a block against eight (maxima) and four
    // (digits): n = 200 52.8 and 69.2 us, 1000 73.9 and 90.4, 2000 107 and 141; transposed
    // operands 200 52.9 and 65.1, 2500 151 and 152, 4000 282 and 237.
    int dev = 0, sms = 0;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return err;
    const long long tiles = (long long)KC * (rows / 32);
    const int chunks = tiles <= 32LL * sms ? 1 : 4;
    // (maxima of long rows: blocks of more k, two an SM, for fewer atomics)
    const int span = view == kViewSym && chunks == 1 ? 32 : 32 * (int)std::min(8LL, std::max(1LL, tiles / (2 * sms)));
    tc5_rowmax<<<dim3((K + span - 1) / span, rows / 32), block, 0, st>>>((int)view, src, ld, R, K, span, rmax);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    tc5_slice<<<dim3((KC + chunks - 1) / chunks, rows / 32), block, 0, st>>>((int)view, src, ld, R, K, rows, KC, chunks, rmax,
                                                                             (unsigned char *)planes, e);
    return cudaGetLastError();
}

// C = alpha A B^T + beta C for two digit-plane operands; arguments checked by
// sliced_gemm.
cudaError_t tc5_gemm(const SlicedOp &A, const SlicedOp &B, int m, int n, double alpha, double beta, double *C,
                     long long ldc, int fill, double *work, size_t work_elems, cudaStream_t st, int *status,
                     long long wait_ns, int hold)
{
    int dev = 0, sms = 148;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    // the tile's 128 rows run along the longer side where C is short and wide
    // (m <= 64 would leave half of every MMA's rows empty)
    const bool sw = fill == kFillAll && ((m + kTM - 1) / kTM) * ((n + kTN - 1) / kTN) > ((n + kTM - 1) / kTM) * ((m + kTN - 1) / kTN);
    ProductArgs p{};
    const SlicedOp &M = sw ? B : A, &N = sw ? A : B;
    p.A = (const unsigned char *)M.planes;
    p.B = (const unsigned char *)N.planes;
    p.ea = M.e;
    p.eb = N.e;
    p.m = sw ? n : m;
    p.n = sw ? m : n;
    p.KC = (std::max(A.K, 1) + kTK - 1) / kTK;
    p.tiles_m = (p.m + kTM - 1) / kTM;
    p.tiles_n = (p.n + kTN - 1) / kTN;
    long long tiles = (long long)p.tiles_m * p.tiles_n;
    if (fill != kFillAll) {
        tiles = 0;
        for (int i = 0; i < p.tiles_m; i++) tiles += std::min(p.tiles_n, fill == kFillLower ? 2 * i + 2 : i + 1);
    }
    // split the reduction when the tiles alone cannot fill the device, in
    // parts of at least four exact sums (512 values of k)
    int splits = 1;
    p.kc_split = p.KC;
    if (tiles < sms && work) {
        splits = (int)(sms / tiles);
        splits = std::min(splits, std::max(1, p.KC / (4 * kGroup)));
        while (splits > 1 && (size_t)splits * m * n > work_elems) splits--;
    }
    if (splits > 1) {
        p.kc_split = ((p.KC + splits - 1) / splits + kGroup - 1) / kGroup * kGroup;
        splits = (p.KC + p.kc_split - 1) / p.kc_split;
    }
    p.splits = splits;
    p.tiles = tiles * splits;
    p.alpha = alpha;
    p.beta = beta;
    p.C = C;
    p.ldc = ldc;
    p.fill = fill;
    p.swapped = sw;
    p.part = splits > 1 ? work : nullptr;
    p.status = status;
    p.wait_ns = wait_ns > 0 ? wait_ns : kWaitNs;
    p.hold = hold >= 0 ? (uint32_t)hold : 0xffffffffu;
    // opt in to the large dynamic shared memory (cheap; per device, so every call)
    if ((e = cudaFuncSetAttribute(tc5_product, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem5)) != cudaSuccess)
        return e;
    tc5_product<<<(unsigned)std::min<long long>(p.tiles, sms), kThreads5, kSmem5, st>>>(p);
    if ((e = cudaGetLastError()) != cudaSuccess || splits == 1) return e;
    return sliced_reduce_launch(m, n, splits, work, alpha, beta, C, ldc, fill, st);
}

}  // namespace gb
