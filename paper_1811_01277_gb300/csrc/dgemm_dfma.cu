// Tiled FP64 products on the DFMA pipe (see dgemm_dfma.cuh).
//
// One CTA of 256 threads computes a TS x TS tile of C, TS = 64 or 32; thread
// (tx, ty) owns rows tx + 16i and columns ty + 16j (i, j < TS/16), so the
// shared-memory reads of a k step are broadcasts without bank conflicts.  The
// reduction runs in steps of 512/TS: the next step's operand tiles are loaded
// from global memory into registers while the current step's DFMAs run from
// shared memory (double-buffered).  An FP64 FMA occupies a scheduler's narrow
// FP64 pipe for many cycles, so even a 2 x 2 register tile leaves the issue
// slots free for the loads and address arithmetic.
//
// What bounds it is FP64 issue, two FMAs per clock and SM, so the work has to
// reach every SM: the solver's panel products (b x b over a long reduction,
// m x b over a short one) take TS = 32 and reductions split down to 16 values
// of k (choose_shape).  Measured on a GB300 over the panels of an n = 1024,
// nbw = 32 solve (before: 64 x 64 tiles, splits of 64 and more): Y^T X 84 -> 12 us,
// A2 (Y T) 98 -> 25 us, Y T and X - Y M 44 -> 16 us a launch.
//
// Operand modes: N (as stored), T (transposed) and SYM (symmetric, lower
// triangle stored).  Each mode has its own thread-to-element mapping so that
// consecutive threads read consecutive addresses; a symmetric tile that
// crosses the diagonal is read element by element.
#include <cuda_runtime.h>

#include <stdint.h>

#include <algorithm>

#include "dgemm_dfma.cuh"
#include "elpa_gb300.h"

namespace gb {

namespace {

constexpr int NT = 256;
constexpr int MODE_N = 0, MODE_T = 1, MODE_SYM = 2;

struct Gemm {
    int m, n;                 // C is m x n
    int k, k2;                // reduction lengths of product 1 and (optional) product 2
    const double *A, *B;      // product 1: op(A) (m x k) op(B) (k x n)
    const double *A2, *B2;    // product 2, same modes, k2 long (k2 = 0: none)
    long long lda, ldb, lda2, ldb2;
    double *C;
    long long ldc;
    double alpha, beta;
    double *partial;          // split-K partials [splits][n][m] (splits > 1)
    int kchunk;               // reduction length per split (over both products), multiple of the k step
    int lower;                // 1: tiles with row tile >= column tile only, elements r >= c
    int tiles_m;
};

// op(A)(r, q) of a BM x BK tile at (r0, q0); 2 elements per thread.
template <int MODE, int TS>
__device__ __forceinline__ void load_a(const double *__restrict__ A, long long lda, int m, int kend, int r0, int q0,
                                       double (&v)[2], int (&sr)[2], int (&sq)[2])
{
    constexpr int BM = TS, BK = 512 / TS;
    const bool below = r0 >= q0 + BK - 1;       // every r >= q in the tile
    const bool above = r0 + BM - 1 < q0;        // every r < q in the tile
    const bool tmap = (MODE == MODE_T) || (MODE == MODE_SYM && above);
#pragma unroll
    for (int t = 0; t < 2; t++) {
        const int e = threadIdx.x + NT * t;
        int r, q;
        if (tmap) {
            q = e % BK;
            r = e / BK;
        } else {
            r = e % BM;
            q = e / BM;
        }
        sr[t] = r;
        sq[t] = q;
        const int gr = r0 + r, gq = q0 + q;
        double x = 0.0;
        if (gr < m && gq < kend) {
            if (MODE == MODE_N) x = A[(long long)gq * lda + gr];
            else if (MODE == MODE_T) x = A[(long long)gr * lda + gq];
            else if (below || (!above && gr >= gq)) x = A[(long long)gq * lda + gr];
            else x = A[(long long)gr * lda + gq];
        }
        v[t] = x;
    }
}

// op(B)(q, c) of a BK x BN tile at (q0, c0); 2 elements per thread.
template <int MODE, int TS>
__device__ __forceinline__ void load_b(const double *__restrict__ B, long long ldb, int n, int kend, int q0, int c0,
                                       double (&v)[2], int (&sq)[2], int (&sc)[2])
{
    constexpr int BN = TS, BK = 512 / TS;
    const bool below = q0 >= c0 + BN - 1;       // every q >= c
    const bool above = q0 + BK - 1 < c0;        // every q < c
    const bool cmap = (MODE == MODE_T) || (MODE == MODE_SYM && above);
#pragma unroll
    for (int t = 0; t < 2; t++) {
        const int e = threadIdx.x + NT * t;
        int q, c;
        if (cmap) {
            c = e % BN;
            q = e / BN;
        } else {
            q = e % BK;
            c = e / BK;
        }
        sq[t] = q;
        sc[t] = c;
        const int gq = q0 + q, gc = c0 + c;
        double x = 0.0;
        if (gq < kend && gc < n) {
            if (MODE == MODE_N) x = B[(long long)gc * ldb + gq];
            else if (MODE == MODE_T) x = B[(long long)gq * ldb + gc];
            else if (below || (!above && gq >= gc)) x = B[(long long)gc * ldb + gq];
            else x = B[(long long)gq * ldb + gc];
        }
        v[t] = x;
    }
}

template <int MA, int MB, int TS>
__global__ void __launch_bounds__(NT) dfma_gemm_kernel(Gemm g)
{
    constexpr int BM = TS, BN = TS, BK = 512 / TS, RT = TS / 16;
    __shared__ double As[2][BK][BM + 1];
    __shared__ double Bs[2][BK][BN + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    int ti, tj;
    if (g.lower) {  // blockIdx.x enumerates the lower tiles row by row
        const long long L = blockIdx.x;
        int i = (int)((sqrt(8.0 * (double)L + 1.0) - 1.0) * 0.5);
        while ((long long)(i + 1) * (i + 2) / 2 <= L) i++;
        while ((long long)i * (i + 1) / 2 > L) i--;
        ti = i;
        tj = (int)(L - (long long)i * (i + 1) / 2);
    } else {
        ti = blockIdx.x;
        tj = blockIdx.y;
    }
    const int r0 = ti * BM, c0 = tj * BN;
    const int split = blockIdx.z;

    double acc[RT][RT];
#pragma unroll
    for (int i = 0; i < RT; i++)
#pragma unroll
        for (int j = 0; j < RT; j++) acc[i][j] = 0.0;

    const int npairs = g.k2 > 0 ? 2 : 1;
    for (int p = 0; p < npairs; p++) {
        const double *A = p ? g.A2 : g.A;
        const double *B = p ? g.B2 : g.B;
        const long long lda = p ? g.lda2 : g.lda, ldb = p ? g.ldb2 : g.ldb;
        const int K = p ? g.k2 : g.k;
        // the split's part of this product (the reductions follow each other)
        const int k0 = p ? (g.k + BK - 1) / BK * BK : 0;
        const int kb = max(0, split * g.kchunk - k0);
        const int ke = min(K, (split + 1) * g.kchunk - k0);
        if (kb >= ke) continue;
        double va[2], vb[2];
        int ar[2], aq[2], bq[2], bc[2];
        load_a<MA, TS>(A, lda, g.m, ke, r0, kb, va, ar, aq);
        load_b<MB, TS>(B, ldb, g.n, ke, kb, c0, vb, bq, bc);
        __syncthreads();  // the previous pair's last reads of the buffers are done
#pragma unroll
        for (int t = 0; t < 2; t++) {
            As[0][aq[t]][ar[t]] = va[t];
            Bs[0][bq[t]][bc[t]] = vb[t];
        }
        __syncthreads();
        int buf = 0;
        for (int q0 = kb; q0 < ke; q0 += BK) {
            const bool more = q0 + BK < ke;
            if (more) {
                load_a<MA, TS>(A, lda, g.m, ke, r0, q0 + BK, va, ar, aq);
                load_b<MB, TS>(B, ldb, g.n, ke, q0 + BK, c0, vb, bq, bc);
            }
#pragma unroll
            for (int q = 0; q < BK; q++) {
                double a[RT], b[RT];
#pragma unroll
                for (int i = 0; i < RT; i++) a[i] = As[buf][q][tx + 16 * i];
#pragma unroll
                for (int j = 0; j < RT; j++) b[j] = Bs[buf][q][ty + 16 * j];
#pragma unroll
                for (int i = 0; i < RT; i++)
#pragma unroll
                    for (int j = 0; j < RT; j++) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
            if (more) {
#pragma unroll
                for (int t = 0; t < 2; t++) {
                    As[buf ^ 1][aq[t]][ar[t]] = va[t];
                    Bs[buf ^ 1][bq[t]][bc[t]] = vb[t];
                }
            }
            __syncthreads();
            buf ^= 1;
        }
    }

    const bool diag = g.lower && ti == tj;
    if (g.partial) {  // split-K: raw partial product
        double *P = g.partial + (long long)split * g.m * g.n;
#pragma unroll
        for (int i = 0; i < RT; i++)
#pragma unroll
            for (int j = 0; j < RT; j++) {
                const int r = r0 + tx + 16 * i, c = c0 + ty + 16 * j;
                if (r < g.m && c < g.n) P[(long long)c * g.m + r] = acc[i][j];
            }
        return;
    }
#pragma unroll
    for (int i = 0; i < RT; i++)
#pragma unroll
        for (int j = 0; j < RT; j++) {
            const int r = r0 + tx + 16 * i, c = c0 + ty + 16 * j;
            if (r < g.m && c < g.n && (!diag || r >= c)) {
                double *cp = g.C + (long long)c * g.ldc + r;
                *cp = (g.beta == 0.0) ? g.alpha * acc[i][j] : fma(g.alpha, acc[i][j], g.beta * *cp);
            }
        }
}

// C = alpha sum_s P[s] + beta C, the splits added in a fixed order.
__global__ void __launch_bounds__(128) splitk_reduce(int m, int n, int splits, const double *__restrict__ P,
                                                     double alpha, double beta, double *__restrict__ C,
                                                     long long ldc)
{
    const long long total = (long long)m * n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int z = 0; z < splits; z++) s += P[(long long)z * total + e];
        const long long c = e / m, r = e - c * m;
        double *cp = C + c * ldc + r;
        *cp = (beta == 0.0) ? alpha * s : fma(alpha, s, beta * *cp);
    }
}

int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 148;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
    return sms;
}

// Tile and splits: the cheapest of 64 x 64 and 32 x 32 tiles, the reduction in
// one piece or split so that the CTAs fill one to eight per SM (16 values of k
// a split at least, the partials within the workspace).  The cost of a shape
// is its fullest SM's FP64 issue, two FMAs a clock, with kEdge values of k for a
// CTA's start and end, and for splits the partials' way through memory; 32 x 32
// tiles issue 4 % slower, a CTA alone on its SM 6 %.  (Splitting to two CTAs an SM
// left its last wave half empty: 64 x 4096, k = 16384 8.24 ms in 512 CTAs, 7.2 in 1024.)
struct Shape {
    int ts, splits;
};

Shape choose_shape(const Gemm &g, size_t work_elems)
{
    constexpr int kEdge = 8;
    const long long sms = sm_count(), k = (long long)g.k + g.k2, out = (long long)g.m * g.n;
    const long long most = g.partial && !g.lower ? std::min({k / 16, 64LL, (long long)(work_elems / (size_t)out)}) : 1;
    Shape best{32, 1};
    double least = 0.0;
    for (int ts : {64, 32}) {
        if (ts == 64 && std::min(g.m, g.n) <= 32) continue;
        const long long tm = (g.m + ts - 1) / ts, tn = (g.n + ts - 1) / ts, bk = 512 / ts;
        const long long t = g.lower ? tm * (tm + 1) / 2 : tm * tn;
        long long sp = 1;
        for (int per = 0; per <= 8; per++) {   // CTAs per SM (0: no split)
            if (per) {
                const long long next = std::min(per * sms / t, most);
                if (next <= sp) {
                    if (sp >= most) break;
                    continue;
                }
                sp = next;
            }
            const long long kc = ((k + sp - 1) / sp + bk - 1) / bk * bk;
            const long long fullest = (t * sp + sms - 1) / sms;
            double clocks = (double)fullest * (ts * ts / 2) * (double)(kc + kEdge);
            if (ts == 32) clocks *= 1.04;
            if (fullest == 1) clocks *= 1.06;
            if (sp > 1) clocks += 3000.0 + (double)(sp * out) * 16.0 / 3300.0;   // a launch; 6.8 TB/s at 2.07 GHz
            if (least == 0.0 || clocks < least) {
                least = clocks;
                best = Shape{ts, (int)sp};
            }
        }
    }
    return best;
}

template <int MA, int MB, int TS>
cudaError_t launch_as(Gemm g, int splits, cudaStream_t st)
{
    constexpr int BK = 512 / TS;
    const int tm = (g.m + TS - 1) / TS, tn = (g.n + TS - 1) / TS;
    g.tiles_m = tm;
    const int k = (g.k + BK - 1) / BK * BK + g.k2;
    g.kchunk = ((k + splits - 1) / splits + BK - 1) / BK * BK;
    if (g.kchunk <= 0) g.kchunk = BK;
    splits = std::max(1, (k + g.kchunk - 1) / g.kchunk);
    g.partial = splits > 1 ? g.partial : nullptr;
    dim3 grid;
    if (g.lower) grid = dim3((unsigned)((long long)tm * (tm + 1) / 2), 1, (unsigned)splits);
    else grid = dim3((unsigned)tm, (unsigned)tn, (unsigned)splits);
    dfma_gemm_kernel<MA, MB, TS><<<grid, NT, 0, st>>>(g);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || splits == 1) return e;
    const long long total = (long long)g.m * g.n;
    splitk_reduce<<<(unsigned)std::min(1024LL, (total + 127) / 128), 128, 0, st>>>(g.m, g.n, splits, g.partial, g.alpha,
                                                                                   g.beta, g.C, g.ldc);
    return cudaGetLastError();
}

template <int MA, int MB>
cudaError_t launch(Gemm g, size_t work_elems, cudaStream_t st)
{
    if (g.m <= 0 || g.n <= 0) return cudaSuccess;
    const Shape s = choose_shape(g, work_elems);
    return s.ts == 64 ? launch_as<MA, MB, 64>(g, s.splits, st) : launch_as<MA, MB, 32>(g, s.splits, st);
}

Gemm base(int m, int n, int k, double alpha, const double *A, long long lda, const double *B, long long ldb,
          double beta, double *C, long long ldc, double *work)
{
    Gemm g{};
    g.m = m;
    g.n = n;
    g.k = k;
    g.k2 = 0;
    g.A = A;
    g.B = B;
    g.lda = lda;
    g.ldb = ldb;
    g.C = C;
    g.ldc = ldc;
    g.alpha = alpha;
    g.beta = beta;
    g.partial = work;
    g.lower = 0;
    return g;
}

}  // namespace

cudaError_t dfma_gemm(char transa, char transb, int m, int n, int k, double alpha, const double *A, long long lda,
                      const double *B, long long ldb, double beta, double *C, long long ldc, double *work,
                      size_t work_elems, cudaStream_t st)
{
    Gemm g = base(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, work);
    const bool ta = transa == 'T' || transa == 't', tb = transb == 'T' || transb == 't';
    if (!ta && !tb) return launch<MODE_N, MODE_N>(g, work_elems, st);
    if (ta && !tb) return launch<MODE_T, MODE_N>(g, work_elems, st);
    if (!ta && tb) return launch<MODE_N, MODE_T>(g, work_elems, st);
    return launch<MODE_T, MODE_T>(g, work_elems, st);
}

cudaError_t dfma_symm(char side, int m, int n, double alpha, const double *S, long long lds, const double *B,
                      long long ldb, double beta, double *C, long long ldc, double *work, size_t work_elems,
                      cudaStream_t st)
{
    if (side == 'L' || side == 'l') {
        Gemm g = base(m, n, m, alpha, S, lds, B, ldb, beta, C, ldc, work);
        return launch<MODE_SYM, MODE_N>(g, work_elems, st);
    }
    Gemm g = base(m, n, n, alpha, B, ldb, S, lds, beta, C, ldc, work);
    return launch<MODE_N, MODE_SYM>(g, work_elems, st);
}

cudaError_t dfma_syr2k_lower(int n, int k, double alpha, const double *A, long long lda, const double *B,
                             long long ldb, double beta, double *C, long long ldc, cudaStream_t st)
{
    // A B^T + B A^T as two products with op(A) = N, op(B) = T
    Gemm g = base(n, n, k, alpha, A, lda, B, ldb, beta, C, ldc, nullptr);
    g.A2 = B;
    g.lda2 = ldb;
    g.B2 = A;
    g.ldb2 = lda;
    g.k2 = k;
    g.lower = 1;
    return launch<MODE_N, MODE_T>(g, 0, st);
}

cudaError_t dfma_syrk_lower_t(int n, int k, double alpha, const double *A, long long lda, double beta, double *C,
                              long long ldc, cudaStream_t st)
{
    Gemm g = base(n, n, k, alpha, A, lda, A, lda, beta, C, ldc, nullptr);
    g.lower = 1;
    return launch<MODE_T, MODE_N>(g, 0, st);
}

}  // namespace gb

extern "C" {

size_t gb_dgemm_workspace_bytes(int m, int n)
{
    if (m < 0 || n < 0) return 0;
    return (size_t)512 * (size_t)(m > 0 ? m : 1) * (size_t)(n > 0 ? n : 1) * 8;
}

static bool bad_ptr(const void *p) { return !p || ((uintptr_t)p % 8) != 0; }

int gb_dgemm(char transa, char transb, int m, int n, int k, double alpha, const double *A, int lda,
             const double *B, int ldb, double beta, double *C, int ldc, void *workspace, size_t ws_bytes,
             void *stream)
{
    const bool ta = transa == 'T' || transa == 't', tb = transb == 'T' || transb == 't';
    if (!ta && transa != 'N' && transa != 'n') return -1;
    if (!tb && transb != 'N' && transb != 'n') return -2;
    if (m < 0) return -3;
    if (n < 0) return -4;
    if (k < 0) return -5;
    if (m == 0 || n == 0) return GB_OK;
    if (k > 0 && bad_ptr(A)) return -7;
    if (lda < (ta ? (k > 1 ? k : 1) : m)) return -8;
    if (k > 0 && bad_ptr(B)) return -9;
    if (ldb < (tb ? n : (k > 1 ? k : 1))) return -10;
    if (bad_ptr(C)) return -12;
    if (ldc < m) return -13;
    if (ws_bytes > 0 && bad_ptr(workspace)) return -14;
    cudaError_t e = gb::dfma_gemm(ta ? 'T' : 'N', tb ? 'T' : 'N', m, n, k, alpha, A, lda, B, ldb, beta, C, ldc,
                                  ws_bytes ? (double *)workspace : nullptr, ws_bytes / 8, (cudaStream_t)stream);
    return e == cudaSuccess ? GB_OK : GB_ERR_CUDA;
}

int gb_dsymm(char side, int m, int n, double alpha, const double *S, int lds, const double *B, int ldb,
             double beta, double *C, int ldc, void *workspace, size_t ws_bytes, void *stream)
{
    const bool left = side == 'L' || side == 'l';
    if (!left && side != 'R' && side != 'r') return -1;
    if (m < 0) return -2;
    if (n < 0) return -3;
    if (m == 0 || n == 0) return GB_OK;
    if (bad_ptr(S)) return -5;
    if (lds < (left ? m : n)) return -6;
    if (bad_ptr(B)) return -7;
    if (ldb < m) return -8;
    if (bad_ptr(C)) return -10;
    if (ldc < m) return -11;
    if (ws_bytes > 0 && bad_ptr(workspace)) return -12;
    cudaError_t e = gb::dfma_symm(left ? 'L' : 'R', m, n, alpha, S, lds, B, ldb, beta, C, ldc,
                                  ws_bytes ? (double *)workspace : nullptr, ws_bytes / 8, (cudaStream_t)stream);
    return e == cudaSuccess ? GB_OK : GB_ERR_CUDA;
}

int gb_dsyr2k(int n, int k, double alpha, const double *A, int lda, const double *B, int ldb, double beta,
              double *C, int ldc, void *stream)
{
    if (n < 0) return -1;
    if (k < 0) return -2;
    if (n == 0) return GB_OK;
    if (k > 0 && bad_ptr(A)) return -4;
    if (lda < n) return -5;
    if (k > 0 && bad_ptr(B)) return -6;
    if (ldb < n) return -7;
    if (bad_ptr(C)) return -9;
    if (ldc < n) return -10;
    cudaError_t e = gb::dfma_syr2k_lower(n, k, alpha, A, lda, B, ldb, beta, C, ldc, (cudaStream_t)stream);
    return e == cudaSuccess ? GB_OK : GB_ERR_CUDA;
}

int gb_dsyrk(int n, int k, double alpha, const double *A, int lda, double beta, double *C, int ldc, void *stream)
{
    if (n < 0) return -1;
    if (k < 0) return -2;
    if (n == 0) return GB_OK;
    if (k > 0 && bad_ptr(A)) return -4;
    if (lda < (k > 1 ? k : 1)) return -5;
    if (bad_ptr(C)) return -7;
    if (ldc < n) return -8;
    cudaError_t e = gb::dfma_syrk_lower_t(n, k, alpha, A, lda, beta, C, ldc, (cudaStream_t)stream);
    return e == cudaSuccess ? GB_OK : GB_ERR_CUDA;
}

}  // extern "C"
