// trans_ev_tridi_to_band on the tcgen05 tensor cores (the default for real
// data with nbw in {16, 32, 64}).
//
// Schedule (as in the other pipelines): work item (g, c) = all tiles of
// sweep group g (NB sweeps: 32 for nbw = 64, else 16) for column block c
// (128 columns); items take tickets in batches of column blocks, groups
// descending, so every dependency wait targets an item that is already
// running; tile k of group g waits until group g+1 has published
// min(k+1, K_{g+1}) tiles.  All waits are bounded.
//
// Tile algebra (Sec. 3.1's blocked Householder aggregation): the tile's NB
// reflectors, applied last sweep first, multiply to I - V T V^T, with V the
// (b+NB-1) x NB parallelogram of reflectors and T upper triangular; with
// U = V T (V's columns scaled to unit length, U's by the inverse factors),
//     Z_win <- Z_win - U (V^T Z_win).
// Both products run on the tensor cores, transposed so that the 128
// eigenvector columns are the MMA's M dimension:
//     W^T  (128 x NB)  = Z_win^T (128 x LP) . V   (LP x NB)
//     dZ^T (128 x LP)  = W^T     (128 x NB) . U^T (NB x LP)
//
// Exact FP64-accurate arithmetic from FP16 digits:
//  * Z is per-column 64-bit fixed point for the whole call (tc_fixed.cuh),
//    |Zi| < 2^61.  V and U rows are fixed point against per-row powers of
//    two, |Vi|, |Ui| <= 2^62.
//  * Every 64-bit value x is cut into eight balanced base-256 digits
//    d_s in [-128, 127] (s = 0 most significant): with y = x +
//    0x8080808080808080 (mod 2^64), d_s = byte_{7-s}(y) - 128, and
//    x = sum_s d_s 256^(7-s).  Each digit is exact in FP16.
//  * Digit products of level l = s + t <= 8 (43 pairs) accumulate in FP32 in
//    TMEM, one accumulator per level.  A level sums at most 8 pairs x K
//    products of magnitude <= 2^14: for the first product K = LP <= 96,
//    below 2^24 (exact); for the second K = NB <= 32, and because the top
//    digits are bounded by 32 (W) and 64 (U), below 2^22 (exact, and
//    convertible by one floating-point addition).  The dropped levels
//    (>= 9) are below 2^-69 of the products' scale.
//  * One MMA per digit plane s of the A operand: its B operand spans the
//    other operand's planes t = 0 .. 8-s along N (the planes follow each
//    other in shared memory at the same 8-row stride), so plane t's product
//    lands in the accumulator of level s+t.  9 MMAs per K step instead of 43.
//  * Levels are folded into 64-bit integers (one rounding per entry) and the
//    update Zi -= dZi is an integer subtraction.
//
// Data movement per tile (b = 64, NB = 32, LP = 96):
//  * the tile record is a V part (V digit planes in the MMA's canonical
//    K-major layout, 48 KB) and a U part (U^T digit planes by 16-row
//    chunks, the exponents of V's columns and U's rows; 48.5 KB), built
//    once per tile by tc5_tile_prep; each part arrives by cp.async.bulk on its
//    own mbarrier, requested as soon as the previous tile no longer needs the
//    buffer;
//  * the window (LP rows x 128 columns, int64) lives in shared memory; the
//    64 new rows come from global memory through L2, NB-1 rows carry over
//    where they are (the window turns in its slots);
//  * Z's digit planes are cut by the threads straight into TMEM (tcgen05.st)
//    and are the A operand of the first product, W's digit planes the A
//    operand of the second.
// TMEM (512 columns): Z digits of ZR K steps in turn [0, 64 ZR), W levels [64
// ZR, + 9 NB); then W digits [0, 64 NB/16) and the dZ levels of two 16-row
// chunks [64 NB/16, + 2 9 16).
//
// What bounds it: 16 thousand digit cuts and as many folds a tile on the
// integer pipe, in 16 warps (one block per SM: the window and the record fill
// shared memory), against 8 thousand clocks of MMAs.  So the 16 warps do nothing
// else: a driver warp issues the MMAs of a K step or chunk as soon as the
// workers have arrived there (named barriers on which only the driver waits),
// a flags' warp publishes stored tiles, looks for the next one's rows and
// makes what a fold needs besides its sums.  A tile of n = 8192, nev =
// 4096 takes 25.8 thousand clocks (34.3 with everything in the same 16 warps and
// K steps and chunks in series): cuts and the first product 6.1, folding
// and cutting W 3.2, the second product and its folds 10.1, loads and
// stores 5.0.  Whole calls: n = 16384, nev = 4096 261 -> 184 ms; complex n = 4096,
// nev = 1228 37.1 -> 20.5; n = nev = 1024, nbw = 32 (a chain of 64 groups) 1.24 -> 0.91.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "elpa_gb300.h"
#include "layout.cuh"
#include "mma_bf16.cuh"
#include "tc_fixed.cuh"
#include "tcgen05.cuh"
#include "trans_ev_kernels.cuh"

namespace gb {

namespace {

constexpr int kCols5 = 128;       // eigenvector columns per work item (the MMA's M)
constexpr int kWork5 = 512;       // 16 working warps: four per TMEM lane quarter (and per SM sub-partition)
constexpr int kThreads5 = kWork5 + 128;  // and a warpgroup of which one warp is the driver (MMAs, record
                                 // copies) and one has the flags; it gives registers to the workers: 96 at launch, then 64 and 104
constexpr int kHandOver = kWork5 + 32;  // threads at the barriers from workers to driver
constexpr int kInStep = kWork5 + 64;    // and at the tile's barriers: with the flags' warp too
constexpr int kPlanes = 8;        // balanced base-256 digits of a 64-bit value
constexpr int kLevels5 = 9;       // digit-pair levels 0..8
constexpr int kColumnBatch5 = 8;  // 128-column blocks per ticket batch (2 and 4 re-read the records more, 16 gains nothing)
constexpr int kTmemCols = 512;
constexpr unsigned long long kDigitBias = 0x8080808080808080ull;
constexpr long long kMbarTimeoutNs = 2000000000ll;  // an MMA batch or a record copy takes microseconds

// RF = 1: real data.  RF = 2: complex data in its real form (interleaved
// re/im storage of Z read as a real column of 2n rows; every complex entry
// of V and U expanded to a 2 x 2 real block), so the tile is a real tile of
// 2 NB reflector columns over a window of 2 (b + NB - 1) rows.
template <int B, int RF>
struct Geo {
    static constexpr int NB = RF == 2 ? 8 : (B == 64 ? 32 : 16);  // sweeps per tile
    static constexpr int NBC = RF * NB;                 // reflector columns of the real form (W's N)
    static constexpr int ADV = RF * B;                  // window rows advanced per tile
    static constexpr int LC = B + NB - 1;               // window rows of the data (complex rows for RF = 2)
    static constexpr int L = RF * LC;                   // window rows of the real form
    static constexpr int CARRY = L - ADV;               // rows carried from tile to tile
    static constexpr int LP = (L + 15) / 16 * 16;       // padded to the MMA's K step
    static constexpr int KSTEPS = LP / 16;              // K steps of the first product
    static constexpr int KD = NBC / 16;                 // K steps of the second
    // tile record: V part [8 planes][NBC rows q][LP] and U part [chunks of
    // NCH rows][8 planes][rows][NBC] + eV[NBC] + eU[LP], canonical K-major
    static constexpr int VPLANE = NBC * LP * 2;
    static constexpr int VBYTES = kPlanes * VPLANE;
    static constexpr int UBYTES = kPlanes * LP * NBC * 2;
    static constexpr int U_EV = UBYTES;
    static constexpr int U_EU = UBYTES + NBC * 4;
    static constexpr int UPART = (UBYTES + (NBC + LP) * 4 + 127) / 128 * 128;
    static constexpr int REC = VBYTES + UPART;
    static constexpr int SBO_V = 16 * LP;               // bytes between 8-row groups of V (N = q)
    static constexpr int SBO_U = 16 * NBC;              // bytes between 8-row groups of U^T (N = j)
    // window: [128 columns][ZROW] int64, ZROW = 2 mod 4 so that a warp's
    // 16-byte accesses to one row pair of 32 columns are conflict-free
    static constexpr int ZROW = LP + 2;
    // dZ row chunks of 16 rows (N = 16 rows x up to 8 U planes), two in tensor
    // memory at once: one is folded while the next one's products run
    static constexpr int NCH = 16;
    static constexpr int CHUNKS = LP / NCH;
    static constexpr int DZBUF = kLevels5 * NCH;        // TMEM columns of a chunk's levels
    // TMEM columns
    static constexpr int WLEV = kLevels5 * NBC;                     // W level accumulators
    static constexpr int ZR = (kTmemCols - WLEV) / 64 < KSTEPS ? (kTmemCols - WLEV) / 64 : KSTEPS;
    static constexpr int T_ZD = 0;
    static constexpr int T_WACC = 64 * ZR;
    static constexpr int T_WD = 0;
    static constexpr int T_DZ = 64 * KD;
    // shared memory
    static constexpr int S_V = 0;
    static constexpr int S_U = VBYTES;
    static constexpr int S_Z = REC;
    static constexpr int S_FC = S_Z + kCols5 * ZROW * 8;     // the folds' constants: V's reflectors, U's rows
    static constexpr int S_BAR = S_FC + (NBC + LP) * 16;    // 6 + ZR mbarriers, TMEM base
    // at least 116 KB, so that shared memory alone keeps the kernel at one
    // CTA per SM: every CTA allocates all 512 TMEM columns
    static constexpr int SMEM = (S_BAR + 128) > 116 * 1024 ? (S_BAR + 128) : 116 * 1024;
    static_assert(ZR >= 1 && T_WACC + WLEV <= kTmemCols, "Z digits and W levels fit in TMEM");
    static_assert(T_DZ + 2 * DZBUF <= kTmemCols, "W digits and two chunks of dZ levels fit in TMEM");
    static_assert(ADV % 8 == 0 && CHUNKS >= 2, "window units stay whole when the window turns");
    // level bounds per K with the top digits bounded by 32 (Z, W) and 64
    // (V, U): at most 7 x 2^14 + 32 128 + 128 64 (level 7) or 7 x 2^14 (level 8)
    static_assert(LP * (7 * 128 * 128) < (1 << 24), "W level sums stay exact in FP32");
    static_assert(NBC * (7 * 128 * 128) < (1 << 22), "dZ level sums stay below 2^22");
    // levels of W that stay below 2^22: a column of V has ADV nonzero rows, and
    // level l < 8 has l - 1 inner pairs
    static constexpr int w_level(int l) { return ADV * (l == 8 ? 7 * 16384 : l == 0 ? 2048 : (l - 1) * 16384 + 4096 + 8192); }
    static constexpr int WMAGIC = w_level(8) < (1 << 22) && w_level(7) < (1 << 22) ? 9 : w_level(4) < (1 << 22) ? 5 : 3;
    static_assert(w_level(2) < (1 << 22), "W levels 0..2 stay below 2^22");
    static_assert(LP % 16 == 0 && NBC % 16 == 0 && NB <= B && CARRY <= ADV, "tile shape");
    static_assert(VBYTES % 128 == 0 && REC % 128 == 0 && S_Z % 16 == 0, "record alignment");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// ---- digits ----------------------------------------------------------------

// FP16 pair (low half from a, high half from b) of the balanced digits held
// in byte `bi` of a and of b (biased bytes: digit = byte - 128).  0x6400|m is
// the FP16 value 1024 + m for 0 <= m < 1024, so subtracting 1152 is exact.
__device__ __forceinline__ uint32_t digit_pair(uint32_t a, uint32_t b, int bi)
{
    const uint32_t sel = (uint32_t)bi | ((uint32_t)bi << 4) | ((uint32_t)(4 + bi) << 8) | ((uint32_t)(4 + bi) << 12);
    const uint32_t r = (__byte_perm(a, b, sel) & 0x00ff00ffu) | 0x64006400u;
    const __half2 h = __hsub2(*(const __half2 *)&r, __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480)));
    return *(const uint32_t *)&h;
}

// the eight digit planes of the pair (x0, x1): out[s] holds plane s
__device__ __forceinline__ void cut_pair(long long x0, long long x1, uint32_t (&out)[kPlanes])
{
    const unsigned long long y0 = (unsigned long long)x0 + kDigitBias;
    const unsigned long long y1 = (unsigned long long)x1 + kDigitBias;
    const uint32_t a_hi = (uint32_t)(y0 >> 32), a_lo = (uint32_t)y0;
    const uint32_t b_hi = (uint32_t)(y1 >> 32), b_lo = (uint32_t)y1;
#pragma unroll
    for (int s = 0; s < 4; s++) out[s] = digit_pair(a_hi, b_hi, 3 - s);
#pragma unroll
    for (int s = 4; s < 8; s++) out[s] = digit_pair(a_lo, b_lo, 7 - s);
}

// Folds of nine exact level sums, sum_l L_l 2^(50 - 8 l + e) rounded once:
// with hi = sum_{l<4} L_l 2^(8(3-l)) and lo = sum_{l>=4} L_l 2^(8(8-l)) it is
// hi 2^(26+e) + lo 2^(e-14) (mod 2^64; the result fits since it is a
// fixed-point entry).  These are 16 thousand folds a tile on the integer pipe,
// so what depends on the exponent alone is made once a tile, by the flags' warp.
//
// An FP32 level sum x (an integer, |x| < 2^22) plus 1.5 2^23 has the bit
// pattern 0x4B400000 + x.  Two such patterns combine with one multiply-add
// into the unsigned 32-bit value L_a 2^8 + L_b + kPairBias (no wrap: |L_a 2^8 +
// L_b| < 2^30 + 2^22 and kPairBias lies between that and 2^32 less that), and
// unsigned wide multiply-adds go on from there without sign extensions; the
// biases leave as one 64-bit constant of hi and one of lo.
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr uint32_t kPairBias = 0x4B400000u * 257u;    // mod 2^32
constexpr unsigned long long kHiBias = (unsigned long long)kPairBias * 65537ull;
constexpr unsigned long long kLoBias =                // nine magic patterns
    (unsigned long long)kPairBias * ((1ull << 24) + 256ull) + (unsigned long long)kMagicBits;
constexpr unsigned long long kLoBias4 = (unsigned long long)kMagicBits << 32;   // level 4 alone
static_assert(kPairBias > (1u << 30) + (1u << 22) && kPairBias < 0xffffffffu - (1u << 30) - (1u << 22), "pairs do not wrap");

// The constants of a row or reflector of exponent e: lo's bias and rounding,
// and the two shifts (s = 26 + e left, t = 14 - e right).  Exponents are at
// least -26 (below, a row would be held finer than half a unit of the result
// by 2^-27); above 13 (reflectors far from orthogonal) t <= 0 and the fold
// shifts lo left.
struct alignas(16) FoldConst {
    unsigned long long lo_add;
    int s, t;
};
constexpr int kMinExp = -26;
__device__ __forceinline__ FoldConst fold_const(int e, unsigned long long lo_bias)
{
    FoldConst f;
    f.s = 26 + e;
    f.t = 14 - e;
    f.lo_add = (e <= 13 ? 1ull << (13 - e) : 0ull) - lo_bias;
    return f;
}

__device__ __forceinline__ uint32_t magic_bits(uint32_t f)
{
    return __float_as_uint(__fadd_rn(__uint_as_float(f), 12582912.0f));
}

__device__ __forceinline__ unsigned long long wide(uint32_t a, uint32_t b, unsigned long long c)
{
    return (unsigned long long)a * b + c;
}

__device__ __forceinline__ long long fold_shift(unsigned long long hi, unsigned long long lo, FoldConst f)
{
    return (long long)(((hi - kHiBias) << f.s) + (unsigned long long)((long long)(lo + f.lo_add) >> f.t));
}

// level sums below 2^22, as magic bit patterns; FAR: the exponent may be above 13
template <bool FAR>
__device__ __forceinline__ long long fold9_bits(const uint32_t (&b)[kLevels5], FoldConst f)
{
    const uint32_t p0 = b[0] * 256u + b[1], p1 = b[2] * 256u + b[3];
    const uint32_t p2 = b[4] * 256u + b[5], p3 = b[6] * 256u + b[7];
    const unsigned long long hi = wide(p0, 65536u, p1);
    const unsigned long long lo = wide(p2, 1u << 24, wide(p3, 256u, b[8]));
    if (FAR && f.t <= 0)
        return (long long)((unsigned long long)shift_ll((long long)(hi - kHiBias), f.s) +
                           (unsigned long long)shift_ll((long long)(lo + f.lo_add), -f.t));
    return fold_shift(hi, lo, f);
}

// level sums (FP32) below 2^24 of which the first NM stay below 2^22 (a
// conversion runs at an eighth of an addition's rate).  Reflectors have unit
// length: no exponent is above 13.
template <int NM>
__device__ __forceinline__ long long fold9_big(const uint32_t (&f)[kLevels5], FoldConst c)
{
    uint32_t m[5];
#pragma unroll
    for (int l = 0; l < 5; l++)
        m[l] = l < NM ? magic_bits(f[l]) : kMagicBits + (uint32_t)__float2int_rn(__uint_as_float(f[l]));
    const unsigned long long hi = wide(m[0] * 256u + m[1], 65536u, m[2] * 256u + m[3]);
    const int l5 = __float2int_rn(__uint_as_float(f[5])), l6 = __float2int_rn(__uint_as_float(f[6]));
    const int l7 = __float2int_rn(__uint_as_float(f[7])), l8 = __float2int_rn(__uint_as_float(f[8]));
    const long long lo = (long long)l5 * (1 << 24) + ((long long)l6 * 65536 + ((long long)l7 * 256 + l8));
    return fold_shift(hi, (unsigned long long)lo + ((unsigned long long)m[4] << 32), c);
}

// round(x 2^(62 - e)) for |x| < 2^e, to nearest with ties to even: the row's
// fixed point (|result| <= 2^62), from the bit pattern with integer
// operations only (x = M 2^p, M the 53-bit significand; subnormals too)
__device__ __forceinline__ long long fixed_row(double x, int e)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((u >> 52) & 0x7ff);
    const unsigned long long M = (u & 0xfffffffffffffull) | (ex ? (1ull << 52) : 0ull);
    const int sh = (ex ? ex : 1) - 1075 + 62 - e;     // x 2^(62-e) = M 2^sh, sh <= 10
    unsigned long long r;
    if (sh >= 0) {
        r = M << sh;
    } else if (sh > -64) {
        const int k = -sh;
        r = M >> k;
        const unsigned long long rem = M & ((1ull << k) - 1), half = 1ull << (k - 1);
        if (rem > half || (rem == half && (r & 1))) r++;
    } else {
        r = 0;
    }
    return (u >> 63) ? -(long long)r : (long long)r;
}

// ---- per-tile records ------------------------------------------------------

// The digit planes of eight values that are neighbours along K: 16 bytes a plane
__device__ __forceinline__ void put_octet(unsigned char *dst, int plane_stride, const long long (&x)[8])
{
    uint32_t w[4][kPlanes];
#pragma unroll
    for (int i = 0; i < 4; i++) cut_pair(x[2 * i], x[2 * i + 1], w[i]);
#pragma unroll
    for (int t = 0; t < kPlanes; t++)
        *(uint4 *)(dst + t * plane_stride) = make_uint4(w[0][t], w[1][t], w[2][t], w[3][t]);
}

template <int B>
constexpr size_t prep_smem_bytes()
{
    using Gm = Geo<B, 1>;
    return (size_t)(2 * Gm::LP * (Gm::NB + 1) + Gm::NB * (Gm::NB + 1) + 3 * Gm::NB) * 8 + (size_t)(Gm::NB + Gm::LP) * 4;
}

template <int B>
constexpr size_t prep_smem_bytes_z()
{
    using Gm = Geo<B, 2>;
    return (size_t)(2 * Gm::LC * (Gm::NB + 1) + 2 * Gm::NB * (Gm::NB + 1) + Gm::NB) * 16 + (size_t)Gm::NB * 8 +
           (size_t)(Gm::NB + Gm::LC) * 4;
}

// The records of a real band (65 thousand tiles at n = 16384).  Bounded by the FP64
// pipe, two multiply-adds per clock and SM: 40 thousand clocks a tile for b = 64
// (Gram 13, substitution 24), 22.7 -> 14 ms at n = 16384 against a Gram matrix and
// a product V T with half of the lanes idle and T by a chain of 32 steps.
template <int B>
__global__ void __launch_bounds__(256, 2) tc5_tile_prep(int n, const double *__restrict__ hh_v,
                                                     const double *__restrict__ hh_tau,
                                                     const long long *__restrict__ off,
                                                     unsigned char *__restrict__ rec)
{
    using Gm = Geo<B, 1>;
    constexpr int L = Gm::L, LP = Gm::LP, NB = Gm::NB, NB1 = NB + 1;
    const int k = blockIdx.x, g = blockIdx.y;
    const int b = B;
    if (k >= group_tiles(n, b, NB, g)) return;
    extern __shared__ double psm[];
    double *V = psm;                      // [LP][NB1]
    double *U = V + LP * NB1;             // [LP][NB1]
    double *Gr = U + LP * NB1;            // [NB][NB1]
    double *tau = Gr + NB * NB1;          // [NB]
    double *nv = tau + NB;                // [NB] column norms of V, and their inverses
    double *rn = nv + NB;                 // [NB]
    int *seV = (int *)(rn + NB);          // [NB]
    int *seU = seV + NB;                  // [LP]
    const int s0 = 1 + g * NB;
    // reflector q of the tile occupies window rows q .. q+len-1 of column q
    for (int e = threadIdx.x; e < LP * NB; e += blockDim.x) {
        const int j = e / NB, q = e % NB;
        const int s = s0 + q;
        double val = 0.0;
        if (s <= n - 1 && s + k * b < n && j - q >= 0 && j - q < b && j < L) {
            const long long idx = sweep_first(n, b, s) + k;
            const int len = min(b, n - s - k * b);
            const double t = hh_tau[idx];
            const int i = j - q;
            if (t != 0.0 && i < len) val = (i == 0) ? 1.0 : hh_v[idx * b + i];
        }
        V[j * NB1 + q] = val;
    }
    if (threadIdx.x < NB) {
        const int s = s0 + threadIdx.x;
        tau[threadIdx.x] = (s <= n - 1 && s + k * b < n) ? hh_tau[sweep_first(n, b, s) + k] : 0.0;
    }
    __syncthreads();
    // Gram matrix (upper triangle): diagonals d and NB - d together make rows of
    // NB products of like length, so that no lane idles on the FP64 pipe
    for (int e = threadIdx.x; e < NB * (NB / 2 + 1); e += blockDim.x) {
        const int d = e / NB, i = e % NB;                    // d = 0: the squares
        const int p = i < NB - d ? i : i - (NB - d), q = i < NB - d ? i + d : p + NB - d;
        if (2 * d == NB && i >= NB / 2) continue;
        double a = 0.0;
        for (int j = q; j < min(p + b, LP); j++) a = fma(V[j * NB1 + p], V[j * NB1 + q], a);
        Gr[p * NB1 + q] = a;
    }
    __syncthreads();
    if (threadIdx.x < NB) {
        const double a = Gr[threadIdx.x * NB1 + threadIdx.x];
        nv[threadIdx.x] = a > 0.0 ? sqrt(a) : 1.0;
        rn[threadIdx.x] = a > 0.0 ? 1.0 / nv[threadIdx.x] : 1.0;
    }
    __syncthreads();
    // U T^{-1} = V with T^{-1} = D^{-1} + the strict upper part of V^T V (D the
    // taus), row by row: u_p = tau_p (v_p - sum_{q<p} u_q G_qp).  A thread keeps its
    // row's sums in registers; the rows take three warps, a different three from tile to
    // tile (each scheduler has a quarter of the FP64 pipe).  Then unit columns of V
    // (U rescaled to keep U V^T): |v_q^T z| <= ||z||, so W stays inside the
    // column's fixed-point range whatever tau is.
    unsigned char *ru = rec + ((size_t)off[g] + k) * Gm::REC + Gm::VBYTES;
    const int row = (int)((threadIdx.x + 32u * (blockIdx.x + blockIdx.y)) % blockDim.x);
    if (row < LP) {
        double a[NB] = {};   // sum_{q<p} u_q G_qp of the columns p to come
        unsigned long long m = 0;
#pragma unroll
        for (int p = 0; p < NB; p++) {
            const double v = V[row * NB1 + p], u = tau[p] * (v - a[p]);
#pragma unroll
            for (int q = p + 1; q < NB; q++) a[q] = fma(u, Gr[p * NB1 + q], a[q]);
            const double us = u * nv[p];
            const unsigned long long w = (unsigned long long)__double_as_longlong(us) & ~(1ull << 63);
            m = w > m ? w : m;
            U[row * NB1 + p] = us;
            V[row * NB1 + p] = v * rn[p];
        }
        seU[row] = max(exponent_above(m), kMinExp);
        ((int *)(ru + Gm::U_EU))[row] = seU[row];
    }
    __syncthreads();
    unsigned char *r = rec + ((size_t)off[g] + k) * Gm::REC;
    if (threadIdx.x < NB) {
        unsigned long long m = 0;
        for (int j = 0; j < LP; j++) {
            const unsigned long long u = (unsigned long long)__double_as_longlong(V[j * NB1 + threadIdx.x]) & ~(1ull << 63);
            m = u > m ? u : m;
        }
        seV[threadIdx.x] = max(exponent_above(m), kMinExp);
        ((int *)(ru + Gm::U_EV))[threadIdx.x] = seV[threadIdx.x];
    }
    __syncthreads();
    // digit planes in the canonical K-major layout of the B operands:
    // V (N = q, K = j), plane t: byte t VPLANE + (q/8) SBO_V + (j/8) 128 +
    // (q%8) 16 + (j%8) 2, so the planes follow each other along N at the same
    // 8-row stride (an MMA's B may span planes t0, t0+1, ...);
    // U^T (N = j, K = q), by chunks of 16 rows: chunk c = j/16 at c 16 SBO_U,
    // within it plane t at t (rows of the chunk / 8) SBO_U, then
    // (j%16/8) SBO_U + (q/8) 128 + (j%8) 16 + (q%8) 2 (again the planes of a
    // chunk contiguous along N)
    for (int e = threadIdx.x; e < NB * (LP / 8); e += blockDim.x) {
        const int q = e % NB, jo = e / NB;
        long long x[8];
#pragma unroll
        for (int i = 0; i < 8; i++) x[i] = fixed_row(V[(jo * 8 + i) * NB1 + q], seV[q]);
        put_octet(r + (q >> 3) * Gm::SBO_V + jo * 128 + (q & 7) * 16, Gm::VPLANE, x);
    }
    for (int e = threadIdx.x; e < LP * (NB / 8); e += blockDim.x) {
        const int j = e % LP, qo = e / LP;
        long long x[8];
#pragma unroll
        for (int i = 0; i < 8; i++) x[i] = fixed_row(U[j * NB1 + qo * 8 + i], seU[j]);
        put_octet(ru + j / Gm::NCH * Gm::NCH * Gm::SBO_U + ((j % Gm::NCH) >> 3) * Gm::SBO_U + qo * 128 +
                      (j & 7) * 16,
                  Gm::NCH / 8 * Gm::SBO_U, x);
    }
}

// Complex tile record: the complex V, T, U of the tile (the same forward
// recurrence with V^H), then their real forms: V's entry v at (row j,
// column q) becomes the 2 x 2 block [[re v, -im v], [im v, re v]] of
// V' (rows 2j+p, columns 2q+p'), so that (z^T V')_(2q+p') are the real and
// imaginary parts of (z^T conj(V))_q; U's entry u becomes, in the B operand
// of the second product (rows 2q+p', columns 2j+p), [[re u, im u],
// [-im u, re u]], so that (w'^T B)_(2j+p) are the parts of (w^T U^T)_j.
// Row exponents are shared by the two real rows of a complex row.
__device__ __forceinline__ double2 cmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
// conj(a) b + c
__device__ __forceinline__ double2 cfma_conj(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, fma(a.y, b.y, c.x)), fma(a.x, b.y, fma(-a.y, b.x, c.y)));
}

template <int B>
__global__ void __launch_bounds__(256) tc5_tile_prep_z(int n, const double2 *__restrict__ hh_v,
                                                       const double2 *__restrict__ hh_tau,
                                                       const long long *__restrict__ off,
                                                       unsigned char *__restrict__ rec)
{
    using Gm = Geo<B, 2>;
    constexpr int LC = Gm::LC, LP = Gm::LP, NB = Gm::NB, NB1 = NB + 1, NBC = Gm::NBC;
    const int k = blockIdx.x, g = blockIdx.y;
    const int b = B;
    if (k >= group_tiles(n, b, NB, g)) return;
    extern __shared__ double2 zsm[];
    double2 *V = zsm;                     // [LC][NB1]
    double2 *U = V + LC * NB1;            // [LC][NB1]
    double2 *T = U + LC * NB1;            // [NB][NB1]
    double2 *Gr = T + NB * NB1;           // [NB][NB1]
    double2 *tau = Gr + NB * NB1;         // [NB]
    double *nv = (double *)(tau + NB);    // [NB]
    int *seV = (int *)(nv + NB);          // [NB]
    int *seU = seV + NB;                  // [LC]
    const int s0 = 1 + g * NB;
    const double2 zero = make_double2(0.0, 0.0);
    for (int e = threadIdx.x; e < LC * NB; e += blockDim.x) {
        const int j = e / NB, q = e % NB;
        const int s = s0 + q;
        double2 val = zero;
        if (s <= n - 1 && s + k * b < n && j - q >= 0 && j - q < b) {
            const long long idx = sweep_first(n, b, s) + k;
            const int len = min(b, n - s - k * b);
            const double2 t = hh_tau[idx];
            const int i = j - q;
            if ((t.x != 0.0 || t.y != 0.0) && i < len) val = (i == 0) ? make_double2(1.0, 0.0) : hh_v[idx * b + i];
        }
        V[j * NB1 + q] = val;
    }
    if (threadIdx.x < NB) {
        const int s = s0 + threadIdx.x;
        tau[threadIdx.x] = (s <= n - 1 && s + k * b < n) ? hh_tau[sweep_first(n, b, s) + k] : zero;
    }
    __syncthreads();
    // Gram matrix v_p^H v_q (p < q), T by T(q,q) = tau_q,
    // T(0:q,q) = -tau_q T(0:q,0:q) V(:,0:q)^H v_q
    for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
        const int p = e / NB, q = e % NB;
        double2 a = zero;
        if (p < q)
            for (int j = q; j < min(p + b, LC); j++) a = cfma_conj(V[j * NB1 + p], V[j * NB1 + q], a);
        Gr[p * NB1 + q] = a;
    }
    __syncthreads();
    for (int q = 0; q < NB; q++) {
        if (threadIdx.x < NB) {
            const int i = threadIdx.x;
            double2 t = zero;
            if (i < q) {
                for (int p = i; p < q; p++) t = cfma(T[i * NB1 + p], Gr[p * NB1 + q], t);
                t = cmul(make_double2(-tau[q].x, -tau[q].y), t);
            } else if (i == q) {
                t = tau[q];
            }
            T[i * NB1 + q] = t;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < LC * NB; e += blockDim.x) {
        const int j = e / NB, q = e % NB;
        double2 a = zero;
        for (int p = max(0, j - b + 1); p <= min(q, j); p++) a = cfma(V[j * NB1 + p], T[p * NB1 + q], a);
        U[j * NB1 + q] = a;
    }
    if (threadIdx.x < NB) {
        const int q = threadIdx.x;
        double a = 0.0;
        for (int j = q; j < min(q + b, LC); j++) {
            const double2 v = V[j * NB1 + q];
            a = fma(v.x, v.x, fma(v.y, v.y, a));
        }
        nv[q] = sqrt(a);
        ((double *)Gr)[q] = a > 0.0 ? 1.0 / nv[q] : 0.0;  // the Gram matrix is no longer needed
    }
    __syncthreads();
    for (int e = threadIdx.x; e < LC * NB; e += blockDim.x) {
        const int j = e / NB, q = e % NB;
        if (nv[q] > 0.0) {
            const double2 v = V[j * NB1 + q], u = U[j * NB1 + q];
            const double rn = ((const double *)Gr)[q];
            V[j * NB1 + q] = make_double2(v.x * rn, v.y * rn);
            U[j * NB1 + q] = make_double2(u.x * nv[q], u.y * nv[q]);
        }
    }
    __syncthreads();
    unsigned char *r = rec + ((size_t)off[g] + k) * Gm::REC;
    unsigned char *ru = r + Gm::VBYTES;
    auto absbits = [](double x) { return (unsigned long long)__double_as_longlong(x) & ~(1ull << 63); };
    if (threadIdx.x < NB) {
        unsigned long long m = 0;
        for (int j = 0; j < LC; j++) {
            const double2 v = V[j * NB1 + threadIdx.x];
            m = max(m, max(absbits(v.x), absbits(v.y)));
        }
        seV[threadIdx.x] = max(exponent_above(m), kMinExp);
        ((int *)(ru + Gm::U_EV))[2 * threadIdx.x] = seV[threadIdx.x];
        ((int *)(ru + Gm::U_EV))[2 * threadIdx.x + 1] = seV[threadIdx.x];
    }
    for (int j = threadIdx.x; j < LP / 2; j += blockDim.x) {
        unsigned long long m = 0;
        if (j < LC)
            for (int q = 0; q < NB; q++) {
                const double2 u = U[j * NB1 + q];
                m = max(m, max(absbits(u.x), absbits(u.y)));
            }
        const int ev = max(exponent_above(m), kMinExp);
        if (j < LC) seU[j] = ev;
        ((int *)(ru + Gm::U_EU))[2 * j] = ev;
        ((int *)(ru + Gm::U_EU))[2 * j + 1] = ev;
    }
    __syncthreads();
    // V' (N = q' = 2q+p', K = j' = 2j+p) and the second product's B
    // (N = j', K = q'), in the layouts of the real record
    for (int e = threadIdx.x; e < NBC * (LP / 8); e += blockDim.x) {
        const int qq = e % NBC, jo = e / NBC, q = qq >> 1;
        long long x[8];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {      // the two real rows of complex row j
            const int j = jo * 4 + i / 2;
            const double2 v = j < LC ? V[j * NB1 + q] : zero;
            x[i] = fixed_row((qq & 1) ? -v.y : v.x, seV[q]);
            x[i + 1] = fixed_row((qq & 1) ? v.x : v.y, seV[q]);
        }
        put_octet(r + (qq >> 3) * Gm::SBO_V + jo * 128 + (qq & 7) * 16, Gm::VPLANE, x);
    }
    for (int e = threadIdx.x; e < LP * (NBC / 8); e += blockDim.x) {
        const int jj = e % LP, qo = e / LP, j = jj >> 1;
        const int ev = j < LC ? seU[j] : kMinExp;
        long long x[8];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const double2 u = j < LC ? U[j * NB1 + qo * 4 + i / 2] : zero;
            x[i] = fixed_row((jj & 1) ? u.y : u.x, ev);
            x[i + 1] = fixed_row((jj & 1) ? u.x : -u.y, ev);
        }
        put_octet(ru + jj / Gm::NCH * Gm::NCH * Gm::SBO_U + ((jj % Gm::NCH) >> 3) * Gm::SBO_U + qo * 128 + (jj & 7) * 16,
                  Gm::NCH / 8 * Gm::SBO_U, x);
    }
}

// ---- the main kernel ------------------------------------------------------

template <bool V>
struct Bool {
    static constexpr bool value = V;
};

struct Tc5Shared {
    int item;
    int far;        // some row's exponent is above 13
    int ready;      // the next tile's rows are there (looked up while this tile's dZ is folded)
};

// wait for an mbarrier phase; on giving up record the timeout
__device__ __forceinline__ bool tc5_wait(uint32_t bar, uint32_t parity, TcState *state)
{
    if (tc5::mbar_wait(bar, parity, kMbarTimeoutNs)) return true;
    tc_set_error(state, GB_ERR_TIMEOUT);
    atomicExch(&state->abort, 1);
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// the workers arrive at barrier `id`, the driver waits there for them
__device__ __forceinline__ void workers_arrive(int id)
{
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kHandOver) : "memory");
}
__device__ __forceinline__ void driver_takes(int id)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kHandOver) : "memory");
}
// workers, driver and flags' warp together: true (in all of them) if a wait of any gave up
__device__ __forceinline__ bool in_step(bool gave_up)
{
    uint32_t r;
    __syncwarp();
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, 15, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
                 : "=r"(r)
                 : "r"((uint32_t)gave_up), "n"(kInStep)
                 : "memory");
    return r != 0;
}

// n: the data's order (complex rows for RF = 2); Zi, ldz: the real form
// (ldz in 64-bit words, RF times the data's leading dimension)
template <int B, int RF>
__global__ void __launch_bounds__(kThreads5, 1)
pipeline_tc5(int n, int nev, long long *__restrict__ Zi, long long ldz, const unsigned char *__restrict__ rec,
             const long long *__restrict__ off, int G, int C, int CB, TcState *state, int *progress,
             long long spin_polls, long long timeout_ns, int hold_group)
{
    using Gm = Geo<B, RF>;
    constexpr int L = Gm::L, LP = Gm::LP, ZROW = Gm::ZROW, KSTEPS = Gm::KSTEPS, NB = Gm::NB, NBC = Gm::NBC;
    constexpr int ZR = Gm::ZR, KD = Gm::KD, ADV = Gm::ADV, CARRY = Gm::CARRY;
    const long long nrows = (long long)RF * n;             // rows of the real form
    extern __shared__ __align__(1024) unsigned char smem[];
    long long *Zs = (long long *)(smem + Gm::S_Z);
    const uint32_t bar_v = tc5::smem_addr(smem + Gm::S_BAR);
    const uint32_t bar_u = bar_v + 8;
    const uint32_t bar_dz = bar_v + 16;                     // two: one per chunk buffer
    const uint32_t bar_k = bar_v + 32;                      // one per K step of Z digits in tensor memory
    const uint32_t bar_end = bar_k + 8 * ZR, bar_fc = bar_end + 8;
    uint32_t *tmem_slot = (uint32_t *)(smem + Gm::S_BAR + 48 + 8 * ZR);
    const FoldConst *eV = (const FoldConst *)(smem + Gm::S_FC), *eU = eV + NBC;
    __shared__ Tc5Shared sh;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quarter = warp & 3, wq = warp >> 2;            // lane quarter, and which of its four warps
    const int col = quarter * 32 + lane;                    // this thread's column of the item (its TMEM lane)
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const int b = B;
    const bool lead = tid == kWork5;                        // the driver's thread that issues

    if (lead) {
        sh.item = atomicAdd(&state->ticket, 1);
        sh.ready = 0;
        tc5::mbar_init(bar_v, 1);
        tc5::mbar_init(bar_u, 1);
        tc5::mbar_init(bar_dz, 1);
        tc5::mbar_init(bar_end, 1);
        tc5::mbar_init(bar_fc, 1);
        tc5::mbar_init(bar_dz + 8, 1);
        for (int i = 0; i < ZR; i++) tc5::mbar_init(bar_k + 8 * i, 1);
        tc5::mbar_init_fence();
    }
    if (warp == 0) tc5::tmem_alloc(tc5::smem_addr(tmem_slot), kTmemCols);
    tc5::fence_before_sync();
    __syncthreads();
    tc5::fence_after_sync();
    constexpr uint32_t tmem = 0;   // all 512 columns are this block's, so they start at 0 (checked below)

    const int item = sh.item;
    const int batch = item / (G * CB);
    const int rem = item - batch * G * CB;
    const int cb = min(CB, C - batch * CB);
    const int g = G - 1 - rem / cb;
    const int c = batch * CB + rem % cb;
    const int s0 = 1 + g * NB;
    const int K = group_tiles(n, b, NB, g);
    const int Knext = (g + 1 < G) ? group_tiles(n, b, NB, g + 1) : 0;
    const int col0 = c * kCols5;
    const unsigned char *rec_g = rec + (size_t)off[g] * Gm::REC;

    int v_issued = 0, u_issued = 0;   // V and U parts requested so far (lead)
    if (tid == 0 && *(volatile uint32_t *)tmem_slot != tmem) {
        tc_set_error(state, GB_ERR_CUDA);
        atomicExch(&state->abort, 1);
    }
    bool gave_up = false;     // this thread's waits: the block leaves at the next barrier

    if (lead) {
        if (g + 1 != hold_group) st_release(progress + (long long)g * C + c, 0);
        tc5::bulk_load(tc5::smem_addr(smem + Gm::S_V), rec_g, Gm::VBYTES, bar_v);
        tc5::bulk_load(tc5::smem_addr(smem + Gm::S_U), rec_g + Gm::VBYTES, Gm::UPART, bar_u);
        v_issued = u_issued = 1;
    }
    bool loaded = false;      // the window already holds this tile's rows
    if (warp >= kWork5 / 32) {
        // ================= the driver: dependency flags, record copies, MMAs (the
        // other three warps of its warpgroup have nothing to do)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if (warp == kWork5 / 32 + 1) {
            // the flags: waits for group g+1, says whether the next tile's rows are
            // there, publishes a tile's rows as soon as they are stored (a fence
            // and a flag; on the driver's way they would hold up the products)
            const int *flag = progress + (long long)(g + 1) * C + c;
            for (int k = 0; k < K; k++) {
                if (!loaded) {
                    if (lane == 0) {
                        const int need = (g + 1 < G) ? min(k + 1, Knext) : 0;
                        unsigned long long t0 = 0;
                        long long polls = 0;
                        bool abort = false;
                        while (need > 0 && ld_acquire(flag) < need) {
                            if (*(volatile int *)&state->abort) { abort = true; break; }
                            if (polls == 0) t0 = now_ns();
                            if (++polls >= spin_polls || (long long)(now_ns() - t0) > timeout_ns) {
                                tc_set_error(state, GB_ERR_TIMEOUT);
                                atomicExch(&state->abort, 1);
                                abort = true;
                                break;
                            }
                            __nanosleep(64);
                        }
                        gave_up |= abort || *(volatile int *)&state->abort;
                    }
                    if (in_step(gave_up)) break;
                    in_step(false);   // the workers have loaded the window
                }
                // the folds' constants from the exponents in this tile's U part
                gave_up |= !tc5_wait(bar_u, (uint32_t)(k & 1), state);
                __syncwarp();
                const int *ex = (const int *)(smem + Gm::S_U + Gm::U_EV);   // eV, then eU
                FoldConst *fc = (FoldConst *)(smem + Gm::S_FC);
                bool far = false;
                for (int i = lane; i < NBC + LP; i += 32) {
                    const int e = ex[i];
                    far |= e > 13;
                    fc[i] = fold_const(e, i < NBC && Gm::WMAGIC != 9 ? kLoBias4 : kLoBias);
                }
                far = __any_sync(0xffffffffu, far);
                __syncwarp();   // every lane's constants before lane 0's arrival (a vote orders no memory)
                if (lane == 0) {
                    sh.far = far;
                    mbar_arrive(bar_fc);
                }
                __syncwarp();
                if (in_step(gave_up)) break;   // W's digits are there
                if (lane == 0) {
                    const int next = (g + 1 < G) ? min(k + 2, Knext) : 0;
                    bool there = k + 1 < K && (next == 0 || ld_acquire(flag) >= next);
                    if (k + 1 < K && !there) {   // once more when the last chunk's products are done
                        constexpr int q = (Gm::CHUNKS - 1) & 1, uses = (Gm::CHUNKS - q + 1) / 2;
                        gave_up |= !tc5_wait(bar_dz + 8 * q, (uint32_t)((k + 1) * uses - 1) & 1, state);
                        there = ld_acquire(flag) >= next;
                    }
                    sh.ready = there;
                }
                if (in_step(gave_up)) break;   // dZ is folded
                loaded = sh.ready != 0;
                in_step(false);                // the tile's final rows are stored
                // every thread's stores happen before this thread's fence and release
                // (barrier, then a cumulative release at GPU scope)
                if (lane == 0 && g + 1 != hold_group) {
                    __threadfence();
                    st_release(progress + (long long)g * C + c, k + 1);
                }
                if (lane == 0) gave_up |= *(volatile int *)&state->abort != 0;   // another block gave up
            }
        } else
        for (int k = warp == kWork5 / 32 ? 0 : K; k < K; k++) {
            const uint64_t vdesc = tc5::smem_desc(tc5::smem_addr(smem + Gm::S_V), 128, Gm::SBO_V);
            const uint64_t udesc = tc5::smem_desc(tc5::smem_addr(smem + Gm::S_U), 128, Gm::SBO_U);
            const bool more = k + 1 < K;
            if (!loaded) {
                if (in_step(gave_up)) break;
                in_step(false);   // the workers have loaded the window
            }
            // ---- W^T = Z^T V by K steps, each when the workers have cut its Z digits
#pragma unroll
            for (int kk = 0; kk < KSTEPS; kk++) {
                if (kk == 0) gave_up |= !tc5_wait(bar_v, (uint32_t)(k & 1), state);   // this tile's V planes
                driver_takes(1 + kk);
                // one MMA per Z digit plane s: B spans V planes 0 .. 8-s
                // along N, so plane t lands in level s+t (D columns T_WACC +
                // NB (s+t)); in the first K step level 8 is first written by
                // its own MMA (s = 1, t = 7), every other level by s = 0
                tc5::fence_after_sync();
                if (tc5::elect_one()) {
                    const int sl = kk % ZR;
                    const uint64_t b0 = vdesc + (uint64_t)((kk * 256) >> 4);
#pragma unroll
                    for (int s = 0; s < kPlanes; s++) {
                        const uint32_t a_t = tmem + Gm::T_ZD + sl * 64 + s * 8;
                        const int nt = s == 0 ? kPlanes : kLevels5 - s;          // planes t = 0 .. nt-1
                        if (kk == 0 && s == 1) {
                            tc5::mma_tmem_a(tmem + Gm::T_WACC + NBC * 8, a_t, b0 + (uint64_t)((7 * Gm::VPLANE) >> 4),
                                                 tc5::idesc_f16_f32(128, NBC), 0u);
                            tc5::mma_tmem_a(tmem + Gm::T_WACC + NBC, a_t, b0, tc5::idesc_f16_f32(128, NBC * 7), 1u);
                        } else {
                            tc5::mma_tmem_a(tmem + Gm::T_WACC + NBC * s, a_t, b0, tc5::idesc_f16_f32(128, NBC * nt),
                                                 (kk > 0 || s > 0) ? 1u : 0u);
                        }
                    }
                    tc5::commit(bar_k + 8 * sl);
                }
                __syncwarp();
            }
            {
                constexpr int sl = (KSTEPS - 1) % ZR, turns = (KSTEPS - sl + ZR - 1) / ZR;
                gave_up |= !tc5_wait(bar_k + 8 * sl, (uint32_t)(k * turns + (KSTEPS - 1) / ZR) & 1, state);
            }
            tc5::fence_after_sync();
            // the V buffer is free: request the next tile's V planes
            if (lead && more) {
                tc5::bulk_load(tc5::smem_addr(smem + Gm::S_V), rec_g + (size_t)(k + 1) * Gm::REC, Gm::VBYTES, bar_v);
                v_issued = k + 2;
            }
            if (in_step(gave_up)) break;   // W's digits are there
            // ---- dZ^T = W^T U^T by chunks of 16 rows (M 128, N = rows x planes, K NB)
#pragma unroll
            for (int ch = 0; ch < Gm::CHUNKS; ch++) {
                if (ch >= 2) driver_takes(1 + ch - 2);   // chunk ch - 2 is read, its buffer free
                // per W digit plane s and K step one MMA whose B spans the chunk's
                // U planes 0 .. 8-s along N (level l = s+t at D columns l N of the
                // chunk's buffer); level 8 first written alone (s = 1, t = 7)
                constexpr int N = Gm::NCH;
                tc5::fence_after_sync();
                constexpr uint32_t pstride = (uint32_t)(N / 8) * Gm::SBO_U;   // bytes between the chunk's planes
                const uint32_t dz = tmem + Gm::T_DZ + (ch & 1) * Gm::DZBUF;
                if (tc5::elect_one()) {
#pragma unroll
                    for (int kd = 0; kd < KD; kd++)
#pragma unroll
                        for (int s = 0; s < kPlanes; s++) {
                            const uint32_t a_t = tmem + Gm::T_WD + kd * 64 + s * 8;
                            const uint64_t b0 = udesc + (uint64_t)((ch * N * Gm::SBO_U + kd * 256) >> 4);
                            const int nt = s == 0 ? kPlanes : kLevels5 - s;
                            if (kd == 0 && s == 1) {
                                tc5::mma_tmem_a(dz + 8 * N, a_t, b0 + (uint64_t)((7 * pstride) >> 4),
                                                     tc5::idesc_f16_f32(128, N), 0u);
                                tc5::mma_tmem_a(dz + N, a_t, b0, tc5::idesc_f16_f32(128, 7 * N), 1u);
                            } else {
                                tc5::mma_tmem_a(dz + s * N, a_t, b0, tc5::idesc_f16_f32(128, nt * N),
                                                     (kd > 0 || s > 0) ? 1u : 0u);
                            }
                        }
                    tc5::commit(bar_dz + 8 * (ch & 1));
                }
                __syncwarp();
            }
            if (in_step(gave_up)) break;   // dZ is folded
            tc5::fence_after_sync();
            // the U part is consumed (planes by the MMAs, exponents by the folds):
            // request the next tile's
            if (lead && more) {
                tc5::fence_proxy_async_smem();
                tc5::bulk_load(tc5::smem_addr(smem + Gm::S_U), rec_g + (size_t)(k + 1) * Gm::REC + Gm::VBYTES, Gm::UPART,
                               bar_u);
                u_issued = k + 2;
            }
            loaded = sh.ready != 0;
            in_step(false);   // the tile's final rows are stored
        }
    } else {
        // ================= the workers
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        // The window turns in its LP slots: logical row j of tile k is in slot
        // (j + k ADV) mod LP, so carried rows stay where they are and new rows take
        // the slots of the rows that left.  (Rows L .. LP-1 hold what was there:
        // V's and U's digits are zero in them.)
        int base = 0;
        auto slot = [&](int j) { return j + base < LP ? j + base : j + base - LP; };
        uint32_t dz_phase = 0;          // bit q: the phase of chunk barrier q to wait for next
        constexpr int CW = kCols5 / (kWork5 / 32);  // columns per warp in loads and stores
        for (int k = 0; k < K; k++) {
            const long long row0 = (long long)RF * ((long long)s0 + (long long)k * b);
            if (!loaded) {
                if (in_step(gave_up)) break;   // group g+1 has stored this tile's rows
                // ---- window: new rows from global memory (through L2: rows written
                // by other SMs)
                const int jlo = (k == 0) ? 0 : CARRY;
                constexpr int H = (L + 31) / 32, CL = H > 3 ? CW / 2 : CW;   // passes of 32 rows, columns at once
#pragma unroll 1
                for (int i0 = 0; i0 < CW; i0 += CL) {
                    long long v[CL][H];
#pragma unroll
                    for (int i = 0; i < CL; i++) {
                        const int cc = warp * CW + i0 + i;
                        const long long *zc = Zi + (long long)(col0 + cc < nev ? col0 + cc : 0) * ldz;
#pragma unroll
                        for (int h = 0; h < H; h++) {
                            const int j = jlo + lane + 32 * h;
                            v[i][h] = (col0 + cc < nev && j < L && row0 + j < nrows) ? __ldcg(zc + row0 + j) : 0ll;
                        }
                    }
#pragma unroll
                    for (int i = 0; i < CL; i++)
#pragma unroll
                        for (int h = 0; h < H; h++) {
                            const int j = jlo + lane + 32 * h;
                            if (j < L) Zs[(warp * CW + i0 + i) * ZROW + slot(j)] = v[i][h];
                        }
                }
                in_step(false);
            }
            // ---- Z digits: four rows per warp of a lane quarter and K step, step kk
            // at columns (kk mod ZR) 64 + plane 8 + pair
            const long long *zc = Zs + col * ZROW;
#pragma unroll 1
            for (int kk = 0; kk < KSTEPS; kk++) {
                const int sl = kk % ZR, turns = (KSTEPS - sl + ZR - 1) / ZR;   // steps of a tile that take this place
                // the products that read the place before (commit k turns + kk / ZR - 1)
                if (kk >= ZR) gave_up |= !tc5_wait(bar_k + 8 * sl, (uint32_t)(k * turns + kk / ZR - 1) & 1, state);
                tc5::fence_after_sync();
                uint32_t w[kPlanes][2];
                const long long *zr = zc + slot(kk * 16 + wq * 4);
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const longlong2 z2 = *(const longlong2 *)(zr + 2 * p);
                    uint32_t d[kPlanes];
                    cut_pair(z2.x, z2.y, d);
#pragma unroll
                    for (int s = 0; s < kPlanes; s++) w[s][p] = d[s];
                }
#pragma unroll
                for (int s = 0; s < kPlanes; s++) tc5::st_x2(tmem + lane_off + Gm::T_ZD + sl * 64 + s * 8 + wq * 2, w[s]);
                tc5::wait_st();
                tc5::fence_before_sync();
                workers_arrive(1 + kk);
            }
            {
                constexpr int sl = (KSTEPS - 1) % ZR, turns = (KSTEPS - sl + ZR - 1) / ZR;
                gave_up |= !tc5_wait(bar_k + 8 * sl, (uint32_t)(k * turns + (KSTEPS - 1) / ZR) & 1, state);
            }
            tc5::fence_after_sync();
            // ---- fold W's levels (reflectors q0 .. q0+NB/4-1 of this column), cut
            // W into digit planes (TMEM: K step q/16, columns s*8 + (q%16)/2)
            gave_up |= !tc5_wait(bar_fc, (uint32_t)(k & 1), state);   // this tile's U part is there, its constants made
            {
                constexpr int QW = NBC / 4;
                const int q0 = wq * QW;
                uint32_t a[kLevels5][QW];
#pragma unroll
                for (int l = 0; l < kLevels5; l++) {
                    if constexpr (QW == 8) {
                        tc5::ld_x8(tmem + lane_off + Gm::T_WACC + NBC * l + q0, a[l]);
                    } else {
                        tc5::ld_x4(tmem + lane_off + Gm::T_WACC + NBC * l + q0, a[l]);
                    }
                }
                tc5::wait_ld();
                uint32_t wd[kPlanes][QW / 2];
#pragma unroll
                for (int p = 0; p < QW / 2; p++) {
                    long long wi[2];
#pragma unroll
                    for (int u = 0; u < 2; u++) {
                        uint32_t f[kLevels5];
#pragma unroll
                        for (int l = 0; l < kLevels5; l++) f[l] = Gm::WMAGIC == 9 ? magic_bits(a[l][2 * p + u]) : a[l][2 * p + u];
                        if constexpr (Gm::WMAGIC == 9) wi[u] = fold9_bits<false>(f, eV[q0 + 2 * p + u]);
                        else wi[u] = fold9_big<Gm::WMAGIC>(f, eV[q0 + 2 * p + u]);
                    }
                    uint32_t d[kPlanes];
                    cut_pair(wi[0], wi[1], d);
#pragma unroll
                    for (int s = 0; s < kPlanes; s++) wd[s][p] = d[s];
                }
                // (the W digits go to the Z-digit columns, dead since the W
                // products completed; the W levels stay untouched until the dZ
                // products, issued after the barrier below)
                const uint32_t wcol = Gm::T_WD + (q0 >> 4) * 64 + (q0 & 15) / 2;
#pragma unroll
                for (int s = 0; s < kPlanes; s++) {
                    if constexpr (QW == 8) {
                        tc5::st_x4(tmem + lane_off + wcol + s * 8, wd[s]);
                    } else {
                        tc5::st_x2(tmem + lane_off + wcol + s * 8, wd[s]);
                    }
                }
                tc5::wait_st();
            }
            tc5::fence_before_sync();
            if (in_step(gave_up)) break;
            // ---- dZ by chunks, folded into the window: Zs -= dZ
            const bool far = sh.far != 0;
#pragma unroll 1
            for (int ch = 0; ch < Gm::CHUNKS; ch++) {
                const int jb = ch * Gm::NCH + wq * (Gm::NCH / 4);
                gave_up |= !tc5_wait(bar_dz + 8 * (ch & 1), (dz_phase >> (ch & 1)) & 1, state);
                dz_phase ^= 1u << (ch & 1);
                tc5::fence_after_sync();
                // this thread: four rows of its column, all levels fetched in one
                // round of TMEM loads
                uint32_t a4[kLevels5][4];
#pragma unroll
                for (int l = 0; l < kLevels5; l++)
                    tc5::ld_x4(tmem + lane_off + Gm::T_DZ + (ch & 1) * Gm::DZBUF + l * Gm::NCH + wq * (Gm::NCH / 4), a4[l]);
                tc5::wait_ld();
                tc5::fence_before_sync();
                if (ch + 2 < Gm::CHUNKS) workers_arrive(1 + ch);
                long long *zw = Zs + col * ZROW + slot(jb);
                auto fold_rows = [&](auto FAR) {
#pragma unroll
                    for (int p = 0; p < 2; p++) {
                        const int j = jb + 2 * p;
                        if (j >= L) continue;
                        long long dz[2];
#pragma unroll
                        for (int u = 0; u < 2; u++) {
                            uint32_t bits[kLevels5];
#pragma unroll
                            for (int l = 0; l < kLevels5; l++) bits[l] = magic_bits(a4[l][2 * p + u]);
                            dz[u] = fold9_bits<FAR.value>(bits, eU[j + u]);
                        }
                        longlong2 *zp = (longlong2 *)(zw + 2 * p);
                        longlong2 z2 = *zp;
                        z2.x -= dz[0];
                        if (j + 1 < L) z2.y -= dz[1];
                        *zp = z2;
                    }
                };
                if (!far) fold_rows(Bool<false>{});
                else fold_rows(Bool<true>{});
            }
            tc5::fence_before_sync();   // this tile's TMEM reads precede the next tile's TMEM writes
            if (in_step(gave_up)) break;
            tc5::fence_after_sync();
            // ---- store the rows final for this group (all rows after the last
            // tile), and bring in the next tile's new rows if they are there: per
            // batch of the warp's columns the loads set out first, then the final
            // rows leave, then the new rows take their slots (the same warp's, so
            // no block barrier between the two).  HN > 2: two batches, to stay
            // within 128 registers
            constexpr int H = (L + 31) / 32, HN = (ADV + 31) / 32;
            constexpr int CS = HN > 2 ? CW / 2 : CW;
            loaded = sh.ready != 0;
            const int jhi = (k == K - 1) ? L : ADV;
            const int base_n = base + ADV % LP < LP ? base + ADV % LP : base + ADV % LP - LP;
            const int ncol = min(nev - col0 - warp * CW, CW);   // columns of this warp that there are
            long long *zg0 = Zi + (long long)(col0 + warp * CW) * ldz + row0 + lane;
            bool bad = false;
#pragma unroll 1
            for (int i0 = 0; i0 < CW; i0 += CS) {
                long long *zg = zg0 + i0 * ldz;
                long long vn[CS][HN];
                if (loaded) {
#pragma unroll
                    for (int h = 0; h < HN; h++) {
                        const bool ok = CARRY + lane + 32 * h < L && row0 + ADV + CARRY + lane + 32 * h < nrows;
#pragma unroll
                        for (int i = 0; i < CS; i++) {
                            vn[i][h] = 0;
                            if (ok && i0 + i < ncol) vn[i][h] = __ldcg(zg + i * ldz + ADV + CARRY + 32 * h);
                        }
                    }
                }
                // rows 32 h of several columns: shared-memory reads, then stores
#pragma unroll
                for (int h = 0; h < H; h++) {
                    if (32 * h >= jhi) break;
                    const bool ok = lane + 32 * h < jhi && row0 + lane + 32 * h < nrows;
                    const long long *zs = Zs + (warp * CW + i0) * ZROW + slot(min(lane + 32 * h, LP - 1));
                    long long v[CS];
#pragma unroll
                    for (int i = 0; i < CS; i++) v[i] = zs[i * ZROW];
                    if (ok) {
                        bool any = false;   // a high word at or beyond the limit: a cheap superset
#pragma unroll
                        for (int i = 0; i < CS; i++)
                            if (i0 + i < ncol) {
                                any |= (uint32_t)((int)(v[i] >> 32) + 0x1fffffff) >= 0x3fffffffu;
                                zg[i * ldz + 32 * h] = v[i];
                            }
                        if (any)
                            for (int i = 0; i < CS; i++) bad |= i0 + i < ncol && tc_out_of_range(v[i]);
                    }
                }
                if (loaded) {
                    __syncwarp();
#pragma unroll
                    for (int h = 0; h < HN; h++) {
                        const int j = CARRY + lane + 32 * h;   // its slot in the next tile's window
                        long long *zs = Zs + (warp * CW + i0) * ZROW + (j + base_n < LP ? j + base_n : j + base_n - LP);
                        if (j < L) {
#pragma unroll
                            for (int i = 0; i < CS; i++) zs[i * ZROW] = vn[i][h];
                        }
                    }
                }
            }
            if (bad) tc_set_error(state, GB_ERR_RANGE);
            base = base_n;
            in_step(false);
        }
    }
    // ---- leave: no copy or MMA of this CTA may still be in flight when its
    // TMEM is released (bounded waits; a timeout was already recorded)
    __syncthreads();
    if (warp == kWork5 / 32) {
        if (v_issued > 0) tc5::mbar_wait(bar_v, (uint32_t)((v_issued - 1) & 1), kMbarTimeoutNs);
        if (u_issued > 0) tc5::mbar_wait(bar_u, (uint32_t)((u_issued - 1) & 1), kMbarTimeoutNs);
        __syncwarp();
        if (tc5::elect_one()) tc5::commit(bar_end);   // after every MMA of this block (the same lane issued them all)
        tc5::mbar_wait(bar_end, 0, kMbarTimeoutNs);
    }
    tc5::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc5::fence_after_sync();
        tc5::tmem_dealloc(*(volatile uint32_t *)tmem_slot, kTmemCols);
    }
}

template <int B, int RF>
size_t tc5_bytes(int n, int nev)
{
    using Gm = Geo<B, RF>;
    const long long G = group_count(n, Gm::NB);
    const long long C = (nev + kCols5 - 1) / kCols5;
    long long tiles = 0;
    for (long long g = 0; g < G; g++) tiles += group_tiles(n, B, Gm::NB, (int)g);
    size_t o = 256 + (size_t)(G * C) * 4;                   // head + progress
    o = (o + 255) & ~(size_t)255;
    o += ((size_t)nev * 4 + 255) & ~(size_t)255;            // column scales
    o += ((size_t)(G + 1) * 8 + 255) & ~(size_t)255;        // tile offsets
    o += (size_t)tiles * Gm::REC;                           // tile records
    return o;
}

// Z, ldz: the data (complex entries interleaved for RF = 2, ldz in entries)
template <int B, int RF>
cudaError_t run_tc5(int n, int nev, const double *hh_v, const double *hh_tau, double *Z, long long ldz,
                    int column_batch, void *ws, size_t ws_bytes, long long spin_polls, long long timeout_ns,
                    int hold_group, cudaStream_t st)
{
    using Gm = Geo<B, RF>;
    const int G = group_count(n, Gm::NB);
    const int C = (nev + kCols5 - 1) / kCols5;
    if (G <= 0 || nev <= 0) return cudaSuccess;
    if (ws_bytes < tc5_bytes<B, RF>(n, nev)) return cudaErrorInvalidValue;
    char *base = (char *)ws;
    TcState *state = (TcState *)base;
    int *progress = (int *)(base + 256);
    size_t o = (256 + (size_t)G * C * 4 + 255) & ~(size_t)255;
    int *E = (int *)(base + o);
    o += ((size_t)nev * 4 + 255) & ~(size_t)255;
    long long *toff = (long long *)(base + o);
    o += ((size_t)(G + 1) * 8 + 255) & ~(size_t)255;
    unsigned char *rec = (unsigned char *)(base + o);

    cudaError_t e = cudaMemsetAsync(ws, 0, 256, st);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(progress, 0xff, (size_t)G * C * 4, st)) != cudaSuccess) return e;
    // the per-column fixed point works on the real form: 2n rows of a complex column
    const int nr = RF * n;
    const long long ldr = RF * ldz;
    const dim3 conv_grid((nr + 255) / 256 < 64 ? (nr + 255) / 256 : 64, nev < 65535 ? nev : 65535);
    tc_col_scale<<<(nev + 7) / 8, 256, 0, st>>>(nr, nev, Z, ldr, E, state);
    tc_convert<<<conv_grid, 256, 0, st>>>(nr, nev, Z, ldr, E, 1);
    tc_tile_offsets<<<1, 1, 0, st>>>(n, B, Gm::NB, G, toff);
    const dim3 prep_grid(group_tiles(n, B, Gm::NB, 0), G);
    if constexpr (RF == 1) {
        constexpr size_t prep_smem = prep_smem_bytes<B>();
        if ((e = cudaFuncSetAttribute(tc5_tile_prep<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)prep_smem)) !=
            cudaSuccess)
            return e;
        tc5_tile_prep<B><<<prep_grid, 256, prep_smem, st>>>(n, hh_v, hh_tau, toff, rec);
    } else {
        constexpr size_t prep_smem = prep_smem_bytes_z<B>();
        if ((e = cudaFuncSetAttribute(tc5_tile_prep_z<B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)prep_smem)) != cudaSuccess)
            return e;
        tc5_tile_prep_z<B><<<prep_grid, 256, prep_smem, st>>>(n, (const double2 *)hh_v, (const double2 *)hh_tau, toff,
                                                              rec);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(pipeline_tc5<B, RF>, cudaFuncAttributeMaxDynamicSharedMemorySize, Gm::SMEM)) !=
        cudaSuccess)
        return e;
    // Column blocks per ticket batch: at least kColumnBatch5, and as many as make a
    // batch's work (CB groups x tiles over the SMs) twice the chain of its
    // groups (a tile each, then the longest group's tiles), in equal batches:
    // n = 4096, 20 blocks: 10.0 ms in one batch, 11.5 in batches of 8; complex, 10
    // blocks: 25.1 against 36.2; n = 16384: 8 (218 ms; 32 blocks at once, which
    // re-read Z more, 220)
    int want = column_batch;
    if (want <= 0) {
        int dev = 0, sms = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        const long long Kmax = group_tiles(n, B, Gm::NB, 0);
        const long long chain = (4LL * sms * (G + Kmax) + (long long)G * Kmax - 1) / ((long long)G * Kmax);
        const long long least = chain > kColumnBatch5 ? chain : kColumnBatch5;
        const int batches = (int)(C / least > 1 ? C / least : 1);
        want = (C + batches - 1) / batches;
    }
    const int CB = C < want ? C : want;
    if ((e = mark_kernel_begin(st)) != cudaSuccess) return e;
    pipeline_tc5<B, RF><<<(unsigned)G * (unsigned)C, kThreads5, Gm::SMEM, st>>>(
        n, nev, (long long *)Z, ldr, rec, toff, G, C, CB, state, progress, spin_polls, timeout_ns, hold_group);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = mark_kernel_end(st)) != cudaSuccess) return e;
    tc_convert<<<conv_grid, 256, 0, st>>>(nr, nev, Z, ldr, E, 0);
    return cudaGetLastError();
}

}  // namespace

bool pipeline_tc5_supported(int b) { return b == 16 || b == 32 || b == 64; }

int pipeline_tc5_sweeps_per_tile(int b, int is_complex)
{
    if (is_complex) return Geo<64, 2>::NB;
    return b == 64 ? Geo<64, 1>::NB : Geo<16, 1>::NB;
}

size_t pipeline_tc5_workspace_bytes(int n, int b, int nev, int is_complex)
{
    if (n < 2 || nev < 1) return 256;
    if (is_complex) {
        if (b == 16) return tc5_bytes<16, 2>(n, nev);
        if (b == 32) return tc5_bytes<32, 2>(n, nev);
        return tc5_bytes<64, 2>(n, nev);
    }
    if (b == 16) return tc5_bytes<16, 1>(n, nev);
    if (b == 32) return tc5_bytes<32, 1>(n, nev);
    return tc5_bytes<64, 1>(n, nev);
}

cudaError_t pipeline_tc5_d(int n, int b, int nev, const double *hh_v, const double *hh_tau, double *Z, long long ldz,
                           int column_batch, void *ws, size_t ws_bytes, long long spin_polls, long long timeout_ns,
                           int hold_group, cudaStream_t st)
{
    if (b == 16)
        return run_tc5<16, 1>(n, nev, hh_v, hh_tau, Z, ldz, column_batch, ws, ws_bytes, spin_polls, timeout_ns,
                              hold_group, st);
    if (b == 32)
        return run_tc5<32, 1>(n, nev, hh_v, hh_tau, Z, ldz, column_batch, ws, ws_bytes, spin_polls, timeout_ns,
                              hold_group, st);
    if (b == 64)
        return run_tc5<64, 1>(n, nev, hh_v, hh_tau, Z, ldz, column_batch, ws, ws_bytes, spin_polls, timeout_ns,
                              hold_group, st);
    return cudaErrorInvalidValue;
}

cudaError_t pipeline_tc5_z(int n, int b, int nev, const double *hh_v, const double *hh_tau, double *Z, long long ldz,
                           int column_batch, void *ws, size_t ws_bytes, long long spin_polls, long long timeout_ns,
                           int hold_group, cudaStream_t st)
{
    if (b == 16)
        return run_tc5<16, 2>(n, nev, hh_v, hh_tau, Z, ldz, column_batch, ws, ws_bytes, spin_polls, timeout_ns,
                              hold_group, st);
    if (b == 32)
        return run_tc5<32, 2>(n, nev, hh_v, hh_tau, Z, ldz, column_batch, ws, ws_bytes, spin_polls, timeout_ns,
                              hold_group, st);
    if (b == 64)
        return run_tc5<64, 2>(n, nev, hh_v, hh_tau, Z, ldz, column_batch, ws, ws_bytes, spin_polls, timeout_ns,
                              hold_group, st);
    return cudaErrorInvalidValue;
}

}  // namespace gb
