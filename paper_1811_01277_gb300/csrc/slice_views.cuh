// Reading a slice-row matrix: element (r, k) of a view of a column-major
// source (the views are listed in dgemm_sliced.cuh), and a 32 x 32 tile of it
// staged in shared memory.
#pragma once
#include "dgemm_sliced.cuh"

namespace gb {

// entry (a, b) of the 2 x 2 real block [x -y; y x] of x + iy
__device__ __forceinline__ double zblock(double x, double y, int a, int b) { return a == b ? x : (a ? y : -y); }

// element (r, k) of the view (r < R, k < K)
__device__ __forceinline__ double view_at(int view, const double *__restrict__ src, long long ld, int r, int k)
{
    switch (view) {
    case kViewRow: return src[r + (long long)k * ld];
    case kViewCol: return src[k + (long long)r * ld];
    case kViewSym: return r >= k ? src[r + (long long)k * ld] : src[k + (long long)r * ld];
    case kViewZExpandN: {
        const double *p = src + 2 * ((r >> 1) + (long long)(k >> 1) * ld);
        return zblock(p[0], p[1], r & 1, k & 1);
    }
    case kViewZExpandC: {  // A^H(i, j) = conj(A(j, i))
        const double *p = src + 2 * ((k >> 1) + (long long)(r >> 1) * ld);
        return zblock(p[0], -p[1], r & 1, k & 1);
    }
    case kViewZHermExpand: {
        const int i = r >> 1, j = k >> 1;
        if (i > j) {
            const double *p = src + 2 * (i + (long long)j * ld);
            return zblock(p[0], p[1], r & 1, k & 1);
        }
        const double *p = src + 2 * (j + (long long)i * ld);
        return zblock(p[0], i == j ? 0.0 : -p[1], r & 1, k & 1);
    }
    default: {  // kViewZRowConj
        const double *p = src + 2 * (r + (long long)(k >> 1) * ld);
        return (k & 1) ? -p[1] : p[0];
    }
    }
}

// Loads the 32 x 32 tile at (r0, k0) into t[r][k] (zero outside R x K), with
// the thread index running along the source's contiguous index.
__device__ __forceinline__ void load_tile(int view, const double *__restrict__ src, long long ld, int R, int K,
                                          int r0, int k0, double (*t)[33])
{
    const int tx = threadIdx.x, ty = threadIdx.y;
    // which index is contiguous in memory for this tile
    bool along_r;
    if (view == kViewRow || view == kViewZExpandN || view == kViewZRowConj) along_r = true;
    else if (view == kViewCol || view == kViewZExpandC) along_r = false;
    else along_r = (r0 >= k0 + 31) || !(r0 + 31 < k0);  // lower or diagonal tiles: read src[r + k ld]
    for (int i = ty; i < 32; i += 8) {
        const int a = along_r ? i : tx, bb = along_r ? tx : i;  // a: k offset, bb: r offset
        const int r = r0 + bb, k = k0 + a;
        double v = 0.0;
        if (r < R && k < K) v = view_at(view, src, ld, r, k);
        t[bb][a] = v;
    }
}

}  // namespace gb
