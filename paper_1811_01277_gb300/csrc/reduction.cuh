// Building blocks shared by the reduction kernels (panel QR, bulge chase):
// arithmetic on real and complex entries behind one set of names, sums over
// neighbouring lanes in a fixed tree, the Householder reflector's scalars,
// and mbarrier arrivals and waits across the blocks of a cluster.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "tcgen05.cuh"

namespace gb {

struct Zc {
    double re, im;
};

__device__ __forceinline__ void zero_of(double &x) { x = 0.0; }
__device__ __forceinline__ void zero_of(Zc &x) { x.re = x.im = 0.0; }
__device__ __forceinline__ void one_of(double &x) { x = 1.0; }
__device__ __forceinline__ void one_of(Zc &x) { x = Zc{1.0, 0.0}; }
__device__ __forceinline__ double conj_of(double a) { return a; }
__device__ __forceinline__ Zc conj_of(Zc a) { return {a.re, -a.im}; }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ Zc mul(Zc a, Zc b) { return {fma(a.re, b.re, -a.im * b.im), fma(a.re, b.im, a.im * b.re)}; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ Zc add(Zc a, Zc b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ double scale(double a, double f) { return a * f; }
__device__ __forceinline__ Zc scale(Zc a, double f) { return {a.re * f, a.im * f}; }
__device__ __forceinline__ double re_of(double a) { return a; }
__device__ __forceinline__ double re_of(Zc a) { return a.re; }
__device__ __forceinline__ bool is_zero(double a) { return a == 0.0; }
__device__ __forceinline__ bool is_zero(Zc a) { return a.re == 0.0 && a.im == 0.0; }
// a b + c
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ Zc mad(Zc a, Zc b, Zc c)
{
    return {fma(-a.im, b.im, fma(a.re, b.re, c.re)), fma(a.im, b.re, fma(a.re, b.im, c.im))};
}
// conj(a) b + c
__device__ __forceinline__ double madc(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ Zc madc(Zc a, Zc b, Zc c)
{
    return {fma(a.im, b.im, fma(a.re, b.re, c.re)), fma(-a.im, b.re, fma(a.re, b.im, c.im))};
}
template <class T>
__device__ __forceinline__ T one_v()
{
    T x;
    one_of(x);
    return x;
}
// c - a b
__device__ __forceinline__ double nmad(double a, double b, double c) { return fma(-a, b, c); }
__device__ __forceinline__ Zc nmad(Zc a, Zc b, Zc c) { return mad(Zc{-a.re, -a.im}, b, c); }

// Sum over TP neighbouring lanes, each holding V / TP of V partial sums
// (partial `lane + TP w` in a[w]).  The tree over the V partials is the same
// for every TP, so that a problem's results do not depend on the cluster
// shape its chase ran on (alone or in a batch with wider bands).
__device__ __forceinline__ double xor_add(double x, int o) { return x + __shfl_xor_sync(0xffffffffu, x, o); }
__device__ __forceinline__ Zc xor_add(Zc x, int o) { return {xor_add(x.re, o), xor_add(x.im, o)}; }
template <int V, int TP, class T>
__device__ __forceinline__ T tree_sum(T (&a)[V / TP])
{
#pragma unroll
    for (int h = V / TP / 2; h >= 1; h /= 2)
#pragma unroll
        for (int i = 0; i < h; i++) a[i] = add(a[i], a[i + h]);
    T x = a[0];
#pragma unroll
    for (int o = TP / 2; o >= 1; o /= 2) x = xor_add(x, o);
    return x;
}

// x of lane `src`
__device__ __forceinline__ double lane_of(double x, int src) { return __shfl_sync(0xffffffffu, x, src); }
__device__ __forceinline__ Zc lane_of(Zc x, int src) { return {lane_of(x.re, src), lane_of(x.im, src)}; }

__device__ __forceinline__ double ld_cg(const double *p) { return __ldcg(p); }
__device__ __forceinline__ Zc ld_cg(const Zc *p)
{
    const double2 t = __ldcg(reinterpret_cast<const double2 *>(p));
    return {t.x, t.y};
}

// 1/x from the hardware's approximate FP64 reciprocal and two Newton-Raphson
// steps, to about one ulp, for 2^-1000 <= |x| < 2^1000.
__device__ __forceinline__ double newton_recip(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double t = fma(-x, r, 1.0);
    r = fma(r, t, r);
    t = fma(-x, r, 1.0);
    return fma(r, t, r);
}

// s in (2^-1000, 2^1000): *nrm = sqrt(s) and *inv = 1 / sqrt(s), from the
// approximate reciprocal square root: two Newton-Raphson steps for the
// inverse, and one for the root itself (within an ulp each).
__device__ __forceinline__ void newton_sqrt(double s, double *nrm, double *inv)
{
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s));
    double e = fma(-s * r, r, 1.0);
    r = fma(0.5 * r, e, r);
    e = fma(-s * r, r, 1.0);
    r = fma(0.5 * r, e, r);
    const double g = s * r;
    *nrm = fma(0.5 * r, fma(-g, g, s), g);
    *inv = r;
}

__device__ __forceinline__ bool mid_range(double x)   // 2^-1000 <= |x| < 2^1000
{
    return (((unsigned)__double2hiint(x) >> 20) & 0x7FFu) - 23u < 2000u;
}

// tau, scale and beta of the reflector (LAPACK form, v_0 = 1): alpha the
// first entry, ss the sum of |x_i|^2 below it; called by whole warps with the
// same arguments.  It sits on the chain of both reductions, and every dependent
// FP64 operation costs a warp about 64 clocks there: beta = -sgn(alpha) nrm
// gives tau = 1 + |alpha| / nrm without waiting for a division, and scale =
// sgn(alpha) / (|alpha| + nrm) takes one Newton reciprocal.
struct Refl {
    double tau, scal, beta;
};
struct ReflZ {
    Zc tau, scal;
    double beta;
};
__device__ __forceinline__ Refl reflector(double alpha, double ss)
{
    double tau = 0.0, scal = 0.0, beta = alpha;
    if (ss != 0.0) {
        const double s = fma(alpha, alpha, ss), a = fabs(alpha);
        if (mid_range(s)) {
            double nrm, inv;
            newton_sqrt(s, &nrm, &inv);
            tau = fma(a, inv, 1.0);
            scal = copysign(newton_recip(a + nrm), alpha);
            beta = -copysign(nrm, alpha);
        } else {
            const double nrm = sqrt(s);
            beta = -copysign(nrm, alpha);
            tau = (beta - alpha) / beta;
            scal = 1.0 / (alpha - beta);
        }
        if (alpha == 0.0) {   // sgn(0) = +1, also for a negative zero
            beta = -fabs(beta);
            scal = fabs(scal);
        }
    }
    return {tau, scal, beta};
}
__device__ __forceinline__ ReflZ reflector(Zc alpha, double ss)
{
    Zc tau{0.0, 0.0}, scal{0.0, 0.0};
    double beta = alpha.re;
    if (!(ss == 0.0 && alpha.im == 0.0)) {
        const double s = fma(alpha.re, alpha.re, fma(alpha.im, alpha.im, ss));
        const double sg = alpha.re >= 0.0 ? 1.0 : -1.0, a = fabs(alpha.re);
        double nrm, inv;
        if (mid_range(s)) newton_sqrt(s, &nrm, &inv);
        else inv = 1.0 / (nrm = sqrt(s));
        beta = -sg * nrm;
        // tau = (beta - alpha) / beta; 1 / (alpha - beta) with alpha - beta =
        // sg (a + nrm) + i im, |alpha - beta|^2 = (a + nrm)^2 + im^2
        tau = Zc{fma(a, inv, 1.0), sg * alpha.im * inv};
        const double dr = a + nrm, dd = fma(dr, dr, alpha.im * alpha.im);
        if (mid_range(dd)) {
            const double f = newton_recip(dd);
            scal = Zc{sg * dr * f, -alpha.im * f};
        } else {   // 1 / dd overflows from dd = 2^-1024 down, the quotients do not
            scal = Zc{sg * dr / dd, -alpha.im / dd};
        }
    }
    return {tau, scal, beta};
}

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// one arrival on the barrier at `bar`'s offset in block `rank` of the cluster
__device__ __forceinline__ void mbar_arrive_remote(void *bar, int rank)
{
    asm volatile(
        "{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %0, %1;\n"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [a];\n}\n" ::"r"(tc5::smem_addr(bar)),
        "r"(rank)
        : "memory");
}

// One value into block `rank`'s shared memory at `to`'s offset, counted in bytes
// on the mbarrier at `bar`'s offset there: data and signal in one message.
__device__ __forceinline__ void send(double *to, double x, void *bar, int rank)
{
    asm volatile(
        "{\n.reg .b32 a, b;\nmapa.shared::cluster.u32 a, %0, %3;\nmapa.shared::cluster.u32 b, %1, %3;\n"
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [a], %2, [b];\n}\n" ::"r"(tc5::smem_addr(to)),
        "r"(tc5::smem_addr(bar)), "l"(__double_as_longlong(x)), "r"(rank)
        : "memory");
}
__device__ __forceinline__ void send(Zc *to, Zc x, void *bar, int rank)
{
    asm volatile(
        "{\n.reg .b32 a, b;\nmapa.shared::cluster.u32 a, %0, %4;\nmapa.shared::cluster.u32 b, %1, %4;\n"
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [a], {%2, %3}, [b];\n}\n" ::"r"(
            tc5::smem_addr(to)),
        "r"(tc5::smem_addr(bar)), "l"(__double_as_longlong(x.re)), "l"(__double_as_longlong(x.im)), "r"(rank)
        : "memory");
}

// this block's arrival on its own barrier, which then waits for `bytes` too
__device__ __forceinline__ void mbar_expect(void *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc5::smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

}  // namespace gb
