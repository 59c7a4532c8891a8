// FP32 inner-solver BLAS-1 kernels on the paired layout of pair.cuh: one
// thread per (site, RHS pair), every update one packed f32x2 instruction for
// the two RHS, per-RHS scalars (alpha, omega, beta) held per lane.  Dot
// products are summed in FP32 over the 24 terms of a site, compensated over the
// sites one thread visits (an FP64 add per site would run on GB300's 1/64-rate
// FP64 pipe) and across threads and blocks on 64-bit integers per RHS; the reductions and the scalar
// recurrences (those the FP64 kernels share, and the shadow-form BiCGStab's
// own) are in reduce.cuh, so every decision stays per RHS.
//
// A pair is processed while either of its RHS is active; an inactive lane's
// solution x is never changed (lane blend), and its terms are excluded from
// every reduction.  Other vectors of an inactive lane are scratch.
#include <algorithm>
#include <cmath>

#include "cplx.cuh"
#include "dp_internal.h"
#include "pair.cuh"
#include "reduce.cuh"

namespace dp {
namespace {

// The passes stream whole fields, bound by HBM (L2 on small lattices).  What
// keeps the memory busy is loads in flight, and a thread that issues many
// before it uses one does better than more threads: the launch bounds ask for
// one block per SM, so up to 128 registers hold them, and the smaller grid
// also leaves the reduction fewer partials.  Components of a site loaded
// together in the s and the update pass, measured over 1 to 12:
// 48x24^3, 12 RHS: s 305 -> 275 us, update 557 -> 497 us (6.9 TB/s);
// 32x16^3, 48 RHS: 233 -> 178, 394 -> 310; 24x16x12^2, 12 RHS: 42 -> 29, 62 -> 45.
constexpr int kSBatch = 6, kUBatch = 2;

struct P12 {
    C2 c[12];
};

__device__ __forceinline__ P12 ldp(const void *base, long long cs, long long me)
{
    P12 v;
    load_pair(static_cast<const float4 *>(base) + me, cs, v.c);
    return v;
}
__device__ __forceinline__ void stp(void *base, long long cs, long long me, const P12 &v)
{
    store_pair(static_cast<float4 *>(base) + me, cs, v.c);
}

// component k of one pair
__device__ __forceinline__ C2 ld1(const void *base, long long cs, long long me, int k)
{
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(base) + me + k * cs);
    return {v.x, v.y};
}
__device__ __forceinline__ void st1(void *base, long long cs, long long me, int k, C2 v)
{
    reinterpret_cast<ulonglong2 *>(base)[me + k * cs] = make_ulonglong2(v.re, v.im);
}

// per-lane complex scalar from the two RHS states
__device__ __forceinline__ C2 lanes(float2 a0, float2 a1) { return {pk(a0.x, a1.x), pk(a0.y, a1.y)}; }
__device__ __forceinline__ C2 neg(C2 a) { return {fneg2(a.re), fneg2(a.im)}; }

// <a, b> per lane over one site, FP32
__device__ __forceinline__ C2 pdot(const P12 &a, const P12 &b)
{
    f2 re = 0ull, im = 0ull;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        re = ffma2(a.c[k].re, b.c[k].re, re);
        re = ffma2(a.c[k].im, b.c[k].im, re);
        im = ffma2(a.c[k].re, b.c[k].im, im);
        im = ffma2(fneg2(a.c[k].im), b.c[k].re, im);
    }
    return {re, im};
}
__device__ __forceinline__ f2 pnorm(const P12 &a)
{
    f2 s = 0ull;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        s = ffma2(a.c[k].re, a.c[k].re, s);
        s = ffma2(a.c[k].im, a.c[k].im, s);
    }
    return s;
}

// a thread's sum over its sites, compensated (Kahan): its error does not grow
// with the sites a thread visits, so the grid can be chosen for speed alone
struct KSum {
    f2 s = 0ull, c = 0ull;
    __device__ __forceinline__ void add(f2 x)
    {
        const f2 y = fadd2(x, fneg2(c)), t = fadd2(s, y);
        c = fadd2(fadd2(t, fneg2(s)), fneg2(y));
        s = t;
    }
};

// the two lanes of a thread's sum, zero for an inactive RHS
__device__ __forceinline__ void set_lanes(float &d0, float &d1, const KSum &v, bool a0, bool a1)
{
    float l0, l1;
    upk(v.s, l0, l1);
    d0 = a0 ? l0 : 0.f;
    d1 = a1 ? l1 : 0.f;
}

#define PAIR_VARS                                                              \
    const int P = nrhs / 2;                                                    \
    const int q = threadIdx.x % P, lane = threadIdx.x / P;                     \
    const long long cs = Vh * P;                                               \
    const bool a0 = st[2 * q].active != 0, a1 = st[2 * q + 1].active != 0
#define PAIR_FOR                                                               \
    for (long long s = (long long)blockIdx.x * c.lanes + lane; (a0 || a1) && s < Vh; \
         s += (long long)gridDim.x * c.lanes)
#define PAIR_LOOP                                                              \
    PAIR_VARS;                                                                 \
    PAIR_FOR

__global__ void __launch_bounds__(kMaxBlock, 1) k32_alpha(Cfg c, const void *rh, const void *vv, long long Vh, int nrhs,
                          RhsState *st, double *partials, unsigned int *counter, int *n_active)
{
    float acc[4];  // RHS 2q: re, im; 2q + 1: re, im
    {
        KSum sum0, sum1;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            const C2 d = pdot(ldp(rh, cs, me), ldp(vv, cs, me));
            sum0.add(d.re);
            sum1.add(d.im);
        }
        set_lanes(acc[0], acc[2], sum0, a0, a1);
        set_lanes(acc[1], acc[3], sum1, a0, a1);
    }
    double v[2];
    const int r = threadIdx.x;
    if (!reduce_last<2, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_alpha(st[r], v[0], v[1]);
    count_active(st, nrhs, n_active);
}

// keep the lanes of `old` whose RHS is inactive
__device__ __forceinline__ f2 blend(f2 nw, f2 old, f2 m) { return (nw & m) | (old & ~m); }

__global__ void __launch_bounds__(kMaxBlock, 1) k32_init(Cfg c, const void *bv, void *rv, void *rh, void *pv,
                                                      long long Vh, int nrhs, RhsState *st,
                                                      double *partials, unsigned int *counter, int *n_active)
{
    float acc[2];
    {
        KSum sum0;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            const P12 b = ldp(bv, cs, me);
            stp(rv, cs, me, b);
            stp(rh, cs, me, b);
            if (pv) stp(pv, cs, me, b);
            sum0.add(pnorm(b));
        }
        set_lanes(acc[0], acc[1], sum0, a0, a1);
    }
    double v[1];
    const int r = threadIdx.x;
    if (!reduce_last<1, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_init(st[r], v[0]);
    count_active(st, nrhs, n_active);
}

// ---- BiCGStab with the shadow image rhat' = Mhat^dag rhat ----
//
// <rhat, v> = <rhat', p> is formed where p is written (update_pa), <rhat, t>
// = <rhat', s> where s is written (s_dots), <t, s> and |t|^2 in the
// x - A^-1 D launch that forms t (per-site sums, totalled by omega_dots):
// 14 vector streams per iteration (s_dots: r, v, rhat, rhat' -> s; update:
// x, p, s, t, v, rhat' -> x, r, p) and no separate alpha or omega pass.

__global__ void __launch_bounds__(kMaxBlock, 1) k32_s_dots(Cfg c, const void *rv, const void *vv,
                                                        void *sv, const void *rh, const void *rh2,
                                                        long long Vh, int nrhs, RhsState *st,
                                                        double *partials, unsigned int *counter)
{
    float acc[8];
    {
        const int qq = threadIdx.x % (nrhs / 2);
        const C2 mal = neg(lanes(st[2 * qq].alpha_f, st[2 * qq + 1].alpha_f));
        KSum sum0, sum1, sum2, sum3;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            f2 rsr = 0ull, rsi = 0ull, rtr = 0ull, rti = 0ull;
#pragma unroll 1
            for (int k0 = 0; k0 < 12; k0 += kSBatch) {
                C2 r[kSBatch], v[kSBatch], h[kSBatch], h2[kSBatch];
#pragma unroll
                for (int i = 0; i < kSBatch; i++) {
                    r[i] = ld1(rv, cs, me, k0 + i);
                    v[i] = ld1(vv, cs, me, k0 + i);
                    h[i] = ld1(rh, cs, me, k0 + i);
                    h2[i] = ld1(rh2, cs, me, k0 + i);
                }
#pragma unroll
                for (int i = 0; i < kSBatch; i++) {
                    const C2 sx = c2_lanefma(mal, v[i], r[i]);
                    st1(sv, cs, me, k0 + i, sx);
                    rsr = ffma2(h[i].re, sx.re, rsr);
                    rsr = ffma2(h[i].im, sx.im, rsr);
                    rsi = ffma2(h[i].re, sx.im, rsi);
                    rsi = ffma2(fneg2(h[i].im), sx.re, rsi);
                    rtr = ffma2(h2[i].re, sx.re, rtr);
                    rtr = ffma2(h2[i].im, sx.im, rtr);
                    rti = ffma2(h2[i].re, sx.im, rti);
                    rti = ffma2(fneg2(h2[i].im), sx.re, rti);
                }
            }
            sum0.add(rsr);
            sum1.add(rsi);
            sum2.add(rtr);
            sum3.add(rti);
        }
        set_lanes(acc[0], acc[4], sum0, a0, a1);
        set_lanes(acc[1], acc[5], sum1, a0, a1);
        set_lanes(acc[2], acc[6], sum2, a0, a1);
        set_lanes(acc[3], acc[7], sum3, a0, a1);
    }
    double v[4];
    const int r = threadIdx.x;
    if (!reduce_last<4, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_s_dots(st[r], v[0], v[1], v[2], v[3]);
}

__global__ void __launch_bounds__(kMaxBlock, 1) k32_omega_dots(Cfg c, const void *dots, long long Vh,
                                                            int nrhs, RhsState *st,
                                                            double *partials, unsigned int *counter)
{
    float acc[6];
    {
        const f2 *d = static_cast<const f2 *>(dots);
        KSum sum0, sum1, sum2;
        PAIR_VARS;
        // three 8-byte loads an item: eight items' in flight, also at the end
        constexpr int kItems = 8;
        const long long step = (long long)gridDim.x * c.lanes;
        for (long long s0 = (long long)blockIdx.x * c.lanes + lane; (a0 || a1) && s0 < Vh; s0 += kItems * step) {
            f2 w[kItems][3];
#pragma unroll
            for (int i = 0; i < kItems; i++) {
                const long long s = s0 + i * step;
#pragma unroll
                for (int k = 0; k < 3; k++) w[i][k] = s < Vh ? __ldg(d + s * P + q + k * cs) : 0ull;
            }
#pragma unroll
            for (int i = 0; i < kItems; i++) {
                sum0.add(w[i][0]);
                sum1.add(w[i][1]);
                sum2.add(w[i][2]);
            }
        }
        set_lanes(acc[0], acc[3], sum0, a0, a1);
        set_lanes(acc[1], acc[4], sum1, a0, a1);
        set_lanes(acc[2], acc[5], sum2, a0, a1);
    }
    double v[3];
    const int r = threadIdx.x;
    if (!reduce_last<3, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_omega_shadow(st[r], v[0], v[1], v[2]);
}

__global__ void __launch_bounds__(kMaxBlock, 1)
k32_update_pa(Cfg c, void *xv, void *rv, void *pv, const void *sv, const void *tv, const void *vv,
              const void *rh2, long long Vh, int nrhs, RhsState *st, int max_iter,
              double *partials, unsigned int *counter, int *n_active)
{
    float acc[6];
    {
        const int qq = threadIdx.x % (nrhs / 2);
        const C2 al = lanes(st[2 * qq].alpha_f, st[2 * qq + 1].alpha_f);
        const C2 om = lanes(st[2 * qq].omega_f, st[2 * qq + 1].omega_f);
        const C2 be = lanes(st[2 * qq].beta_f, st[2 * qq + 1].beta_f);
        const C2 mom = neg(om);
        KSum sum0, sum1, sum2;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            const f2 m = (a0 ? 0x00000000ffffffffull : 0ull) | (a1 ? 0xffffffff00000000ull : 0ull);
            f2 nn = 0ull, rpr = 0ull, rpi = 0ull;
#pragma unroll 1
            for (int k0 = 0; k0 < 12; k0 += kUBatch) {
                C2 x[kUBatch], p[kUBatch], sx[kUBatch], t[kUBatch], v[kUBatch], h2[kUBatch];
#pragma unroll
                for (int i = 0; i < kUBatch; i++) {
                    x[i] = ld1(xv, cs, me, k0 + i);
                    p[i] = ld1(pv, cs, me, k0 + i);
                    sx[i] = ld1(sv, cs, me, k0 + i);
                    t[i] = ld1(tv, cs, me, k0 + i);
                    v[i] = ld1(vv, cs, me, k0 + i);
                    h2[i] = ld1(rh2, cs, me, k0 + i);
                }
#pragma unroll
                for (int i = 0; i < kUBatch; i++) {
                    C2 xn = c2_lanefma(om, sx[i], c2_lanefma(al, p[i], x[i]));
                    xn.re = blend(xn.re, x[i].re, m);
                    xn.im = blend(xn.im, x[i].im, m);
                    st1(xv, cs, me, k0 + i, xn);
                    const C2 r = c2_lanefma(mom, t[i], sx[i]);
                    st1(rv, cs, me, k0 + i, r);
                    const C2 pn = c2_lanefma(be, c2_lanefma(mom, v[i], p[i]), r);
                    st1(pv, cs, me, k0 + i, pn);
                    nn = ffma2(r.re, r.re, nn);
                    nn = ffma2(r.im, r.im, nn);
                    rpr = ffma2(h2[i].re, pn.re, rpr);
                    rpr = ffma2(h2[i].im, pn.im, rpr);
                    rpi = ffma2(h2[i].re, pn.im, rpi);
                    rpi = ffma2(fneg2(h2[i].im), pn.re, rpi);
                }
            }
            sum0.add(nn);
            sum1.add(rpr);
            sum2.add(rpi);
        }
        set_lanes(acc[0], acc[3], sum0, a0, a1);
        set_lanes(acc[1], acc[4], sum1, a0, a1);
        set_lanes(acc[2], acc[5], sum2, a0, a1);
    }
    double v[3];
    const int r = threadIdx.x;
    if (!reduce_last<3, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    // convergence on |r|^2, then the next alpha = rho' / <rhat', p> for the
    // RHS still iterating
    if (r < nrhs) {
        finish_update_rr(st[r], v[0], max_iter);
        finish_alpha(st[r], v[1], v[2]);
    }
    count_active(st, nrhs, n_active);
}

// ---- CGNE on the normal equations: real per-RHS scalars, per lane ----

__device__ __forceinline__ f2 lanes_re(float a0, float a1) { return pk(a0, a1); }

__global__ void __launch_bounds__(kMaxBlock, 1)
k32_cg_gamma(Cfg c, const void *zv, long long Vh, int nrhs, RhsState *st, int first,
             double *partials, unsigned int *counter)
{
    float acc[2];
    {
        KSum sum0;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            f2 nn = 0ull;
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const C2 z = ld1(zv, cs, me, k);
                nn = ffma2(z.re, z.re, nn);
                nn = ffma2(z.im, z.im, nn);
            }
            sum0.add(nn);
        }
        set_lanes(acc[0], acc[1], sum0, a0, a1);
    }
    double v[1];
    const int r = threadIdx.x;
    if (!reduce_last<1, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_cg_gamma(st[r], v[0], first);
}

// p = z + beta p
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_cg_p(Cfg c, const void *zv, void *pv, long long Vh, int nrhs, const RhsState *st)
{
    const int qq = threadIdx.x % (nrhs / 2);
    const f2 be = lanes_re(st[2 * qq].beta_f.x, st[2 * qq + 1].beta_f.x);
    PAIR_LOOP
    {
        const long long me = s * P + q;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            const C2 z = ld1(zv, cs, me, k);
            C2 p = ld1(pv, cs, me, k);
            p.re = ffma2(be, p.re, z.re);
            p.im = ffma2(be, p.im, z.im);
            st1(pv, cs, me, k, p);
        }
    }
}

// alpha = rho / |w|^2
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_cg_alpha(Cfg c, const void *wv, long long Vh, int nrhs, RhsState *st, double *partials,
             unsigned int *counter)
{
    float acc[2];
    {
        KSum sum0;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            f2 nn = 0ull;
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const C2 w = ld1(wv, cs, me, k);
                nn = ffma2(w.re, w.re, nn);
                nn = ffma2(w.im, w.im, nn);
            }
            sum0.add(nn);
        }
        set_lanes(acc[0], acc[1], sum0, a0, a1);
    }
    double v[1];
    const int r = threadIdx.x;
    if (!reduce_last<1, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_cg_alpha(st[r], v[0]);
}

// x += alpha p (active lanes only), r -= alpha w, |r|^2
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_cg_update(Cfg c, void *xv, void *rv, const void *pv, const void *wv, long long Vh, int nrhs,
              RhsState *st, int max_iter, double *partials, unsigned int *counter, int *n_active)
{
    float acc[2];
    {
        const int qq = threadIdx.x % (nrhs / 2);
        const f2 al = lanes_re(st[2 * qq].alpha_f.x, st[2 * qq + 1].alpha_f.x);
        const f2 mal = fneg2(al);
        KSum sum0;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            const f2 m = (a0 ? 0x00000000ffffffffull : 0ull) | (a1 ? 0xffffffff00000000ull : 0ull);
            f2 nn = 0ull;
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const C2 x = ld1(xv, cs, me, k), p = ld1(pv, cs, me, k);
                C2 xn = {ffma2(al, p.re, x.re), ffma2(al, p.im, x.im)};
                xn.re = blend(xn.re, x.re, m);
                xn.im = blend(xn.im, x.im, m);
                st1(xv, cs, me, k, xn);
                C2 r = ld1(rv, cs, me, k);
                const C2 w = ld1(wv, cs, me, k);
                r.re = ffma2(mal, w.re, r.re);
                r.im = ffma2(mal, w.im, r.im);
                st1(rv, cs, me, k, r);
                nn = ffma2(r.re, r.re, nn);
                nn = ffma2(r.im, r.im, nn);
            }
            sum0.add(nn);
        }
        set_lanes(acc[0], acc[1], sum0, a0, a1);
    }
    double v[1];
    const int r = threadIdx.x;
    if (!reduce_last<1, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_cg_update(st[r], v[0], max_iter);
    count_active(st, nrhs, n_active);
}

// ---- GCR (the Krylov part of SAP+GCR): per-RHS dot products into device
// arrays, and updates with per-RHS coefficients read from them ----

// out[r] = <a, b> = sum conj(a) b (complex) per RHS
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_dotv(Cfg c, const void *av, const void *bv, long long Vh, int nrhs, const RhsState *st,
         double2 *out, double *partials, unsigned int *counter)
{
    float acc[4];
    {
        KSum sum0, sum1;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            f2 re = 0ull, im = 0ull;
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const C2 x = ld1(av, cs, me, k), y = ld1(bv, cs, me, k);
                re = ffma2(x.re, y.re, re);
                re = ffma2(x.im, y.im, re);
                im = ffma2(x.re, y.im, im);
                im = ffma2(fneg2(x.im), y.re, im);
            }
            sum0.add(re);
            sum1.add(im);
        }
        set_lanes(acc[0], acc[2], sum0, a0, a1);
        set_lanes(acc[1], acc[3], sum1, a0, a1);
    }
    double v[2];
    const int r = threadIdx.x;
    if (!reduce_last<2, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) out[r] = make_double2(v[0], v[1]);
}

// out[r] = |a|^2 per RHS
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_norm2v(Cfg c, const void *av, long long Vh, int nrhs, const RhsState *st, double *out,
           double *partials, unsigned int *counter)
{
    float acc[2];
    {
        KSum sum0;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            f2 nn = 0ull;
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const C2 x = ld1(av, cs, me, k);
                nn = ffma2(x.re, x.re, nn);
                nn = ffma2(x.im, x.im, nn);
            }
            sum0.add(nn);
        }
        set_lanes(acc[0], acc[1], sum0, a0, a1);
    }
    double v[1];
    const int r = threadIdx.x;
    if (!reduce_last<1, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) out[r] = v[0];
}

__device__ __forceinline__ C2 coef_lanes(const double2 *cf, int q, double sign)
{
    const double2 c0 = cf[2 * q], c1 = cf[2 * q + 1];
    return {pk((float)(sign * c0.x), (float)(sign * c1.x)), pk((float)(sign * c0.y), (float)(sign * c1.y))};
}

// w -= c wi, z -= c zi (modified Gram-Schmidt step, c per RHS)
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_mgs(Cfg c, void *wv, void *zv, const void *wiv, const void *ziv, long long Vh, int nrhs,
        const RhsState *st, const double2 *cf)
{
    const int qq = threadIdx.x % (nrhs / 2);
    const C2 mc = coef_lanes(cf, qq, -1.0);
    PAIR_LOOP
    {
        const long long me = s * P + q;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            st1(wv, cs, me, k, c2_lanefma(mc, ld1(wiv, cs, me, k), ld1(wv, cs, me, k)));
            st1(zv, cs, me, k, c2_lanefma(mc, ld1(ziv, cs, me, k), ld1(zv, cs, me, k)));
        }
    }
}

// w /= |w|, z /= |w| (nrm = |w|^2 per RHS)
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_normalise(Cfg c, void *wv, void *zv, long long Vh, int nrhs, const RhsState *st,
              const double *nrm)
{
    const int qq = threadIdx.x % (nrhs / 2);
    const double n0 = nrm[2 * qq], n1 = nrm[2 * qq + 1];
    // a vanishing direction (|w|^2 below FP32 range) is dropped rather than
    // scaled to overflow
    const f2 sc = pk(n0 > 1e-60 ? (float)(1.0 / sqrt(n0)) : 0.f, n1 > 1e-60 ? (float)(1.0 / sqrt(n1)) : 0.f);
    PAIR_LOOP
    {
        const long long me = s * P + q;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            const C2 w = ld1(wv, cs, me, k), z = ld1(zv, cs, me, k);
            st1(wv, cs, me, k, {fmul2(sc, w.re), fmul2(sc, w.im)});
            st1(zv, cs, me, k, {fmul2(sc, z.re), fmul2(sc, z.im)});
        }
    }
}

// x += a z (active lanes), r -= a w, |r|^2 -> convergence (a = <w, r> per RHS)
__global__ void __launch_bounds__(kMaxBlock, 1)
k32_gcr_update(Cfg c, void *xv, void *rv, const void *zv, const void *wv, long long Vh, int nrhs,
               RhsState *st, const double2 *cf, int max_iter, double *partials,
               unsigned int *counter, int *n_active)
{
    float acc[2];
    {
        const int qq = threadIdx.x % (nrhs / 2);
        const C2 a = coef_lanes(cf, qq, 1.0), ma = coef_lanes(cf, qq, -1.0);
        KSum sum0;
        PAIR_LOOP
        {
            const long long me = s * P + q;
            const f2 m = (a0 ? 0x00000000ffffffffull : 0ull) | (a1 ? 0xffffffff00000000ull : 0ull);
            f2 nn = 0ull;
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const C2 x = ld1(xv, cs, me, k);
                C2 xn = c2_lanefma(a, ld1(zv, cs, me, k), x);
                xn.re = blend(xn.re, x.re, m);
                xn.im = blend(xn.im, x.im, m);
                st1(xv, cs, me, k, xn);
                const C2 r = c2_lanefma(ma, ld1(wv, cs, me, k), ld1(rv, cs, me, k));
                st1(rv, cs, me, k, r);
                nn = ffma2(r.re, r.re, nn);
                nn = ffma2(r.im, r.im, nn);
            }
            sum0.add(nn);
        }
        set_lanes(acc[0], acc[1], sum0, a0, a1);
    }
    double v[1];
    const int r = threadIdx.x;
    if (!reduce_last<1, 2>(acc, c, partials, counter, nrhs / 2, v)) return;
    if (r < nrhs) finish_cg_update(st[r], v[0], max_iter);
    count_active(st, nrhs, n_active);
}

// out = a - b (every pair)
__global__ void k32_xmy(const float4 *a, const float4 *b, float4 *out, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const ulonglong2 x = reinterpret_cast<const ulonglong2 *>(a)[i];
    const ulonglong2 y = reinterpret_cast<const ulonglong2 *>(b)[i];
    reinterpret_cast<ulonglong2 *>(out)[i] = make_ulonglong2(fsub2(x.x, y.x), fsub2(x.y, y.y));
}

// r32 (paired) = r64 / |r| per RHS (zero for inactive RHS)
__global__ void k32_from64(const double2 *r64, float4 *r32, long long Vh, int n, const RhsState *st)
{
    const int P = n / 2;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= Vh * P) return;
    const long long s = gid / P;
    const int q = (int)(gid - s * P);
    const double i0 = st[2 * q].active ? 1.0 / st[2 * q].scale : 0.0;
    const double i1 = st[2 * q + 1].active ? 1.0 / st[2 * q + 1].scale : 0.0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const long long b64 = ((long long)k * Vh + s) * n + 2 * q;
        const double2 u = r64[b64], v = r64[b64 + 1];
        r32[((long long)k * Vh + s) * P + q] =
            make_float4((float)(u.x * i0), (float)(v.x * i1), (float)(u.y * i0), (float)(v.y * i1));
    }
}

// x64 += |r| e32 per active RHS
__global__ void k32_acc64(double2 *x64, const float4 *e32, long long Vh, int n, const RhsState *st)
{
    const int P = n / 2;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= Vh * P) return;
    const long long s = gid / P;
    const int q = (int)(gid - s * P);
    // refined RHS take blas_acc_f32_ratio instead
    const bool a0 = st[2 * q].active != 0 && !st[2 * q].refine;
    const bool a1 = st[2 * q + 1].active != 0 && !st[2 * q + 1].refine;
    if (!a0 && !a1) return;
    const double s0 = st[2 * q].scale, s1 = st[2 * q + 1].scale;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const float4 e = e32[((long long)k * Vh + s) * P + q];
        const long long b64 = ((long long)k * Vh + s) * n + 2 * q;
        if (a0) {
            double2 x = x64[b64];
            x.x = fmx(s0, (double)e.x, x.x);
            x.y = fmx(s0, (double)e.z, x.y);
            x64[b64] = x;
        }
        if (a1) {
            double2 x = x64[b64 + 1];
            x.x = fmx(s1, (double)e.y, x.x);
            x.y = fmx(s1, (double)e.w, x.y);
            x64[b64 + 1] = x;
        }
    }
}

inline unsigned blocks_for(long long n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

cudaError_t blas32_init(BlasCtx &bc, const void *b, void *r, void *rh, long long Vh, int nrhs,
                        RhsState *st, cudaStream_t s, void *p)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_init, Vh, nrhs / 2);
    k32_init<<<c.grid, c.block, 0, s>>>(c, b, r, rh, p, Vh, nrhs, st, bc.partials, bc.counter, bc.n_active);
    return cudaGetLastError();
}

cudaError_t blas32_s_dots(BlasCtx &bc, const void *r, const void *v, void *sv, const void *rh,
                          const void *rh2, long long Vh, int nrhs, RhsState *st, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_s_dots, Vh, nrhs / 2);
    k32_s_dots<<<c.grid, c.block, 0, s>>>(c, r, v, sv, rh, rh2, Vh, nrhs, st, bc.partials, bc.counter);
    return cudaGetLastError();
}

cudaError_t blas32_omega_dots(BlasCtx &bc, const void *dots, long long Vh, int nrhs, RhsState *st,
                              cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    Cfg c = cfg_wave(bc, k32_omega_dots, Vh, nrhs / 2);
    // 24 bytes an item: what counts is the rounds of eight loads, Vh / (8 lanes
    // grid) in the blocks and 6 grid / (8 lanes) in the last one, fewest near
    // grid = sqrt(Vh) / 2 (32x16^3, 48 RHS: 304 blocks 41 us, 128 blocks 21)
    c.grid = std::min(c.grid, std::max(c.lanes, (int)std::sqrt((double)Vh) / 2));
    k32_omega_dots<<<c.grid, c.block, 0, s>>>(c, dots, Vh, nrhs, st, bc.partials, bc.counter);
    return cudaGetLastError();
}

cudaError_t blas32_update_pa(BlasCtx &bc, void *x, void *r, void *p, const void *sv, const void *t,
                             const void *v, const void *rh2, long long Vh, int nrhs, RhsState *st,
                             int max_iter, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_update_pa, Vh, nrhs / 2);
    k32_update_pa<<<c.grid, c.block, 0, s>>>(c, x, r, p, sv, t, v, rh2, Vh, nrhs, st, max_iter,
                                             bc.partials, bc.counter, bc.n_active);
    return cudaGetLastError();
}

cudaError_t blas32_alpha(BlasCtx &bc, const void *rh, const void *v, long long Vh, int nrhs,
                         RhsState *st, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_alpha, Vh, nrhs / 2);
    k32_alpha<<<c.grid, c.block, 0, s>>>(c, rh, v, Vh, nrhs, st, bc.partials, bc.counter, bc.n_active);
    return cudaGetLastError();
}

cudaError_t blas32_cg_gamma(BlasCtx &bc, const void *z, long long Vh, int nrhs, RhsState *st,
                            int first, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_cg_gamma, Vh, nrhs / 2);
    k32_cg_gamma<<<c.grid, c.block, 0, s>>>(c, z, Vh, nrhs, st, first, bc.partials, bc.counter);
    return cudaGetLastError();
}

cudaError_t blas32_cg_p(BlasCtx &bc, const void *z, void *p, long long Vh, int nrhs,
                        const RhsState *st, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_cg_p, Vh, nrhs / 2);
    k32_cg_p<<<c.grid, c.block, 0, s>>>(c, z, p, Vh, nrhs, st);
    return cudaGetLastError();
}

cudaError_t blas32_cg_alpha(BlasCtx &bc, const void *w, long long Vh, int nrhs, RhsState *st,
                            cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_cg_alpha, Vh, nrhs / 2);
    k32_cg_alpha<<<c.grid, c.block, 0, s>>>(c, w, Vh, nrhs, st, bc.partials, bc.counter);
    return cudaGetLastError();
}

cudaError_t blas32_cg_update(BlasCtx &bc, void *x, void *r, const void *p, const void *w,
                             long long Vh, int nrhs, RhsState *st, int max_iter, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_cg_update, Vh, nrhs / 2);
    k32_cg_update<<<c.grid, c.block, 0, s>>>(c, x, r, p, w, Vh, nrhs, st, max_iter, bc.partials,
                                             bc.counter, bc.n_active);
    return cudaGetLastError();
}

cudaError_t blas32_dotv(BlasCtx &bc, const void *a, const void *b, long long Vh, int nrhs,
                        const RhsState *st, double2 *out, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_dotv, Vh, nrhs / 2);
    k32_dotv<<<c.grid, c.block, 0, s>>>(c, a, b, Vh, nrhs, st, out, bc.partials, bc.counter);
    return cudaGetLastError();
}

cudaError_t blas32_norm2v(BlasCtx &bc, const void *a, long long Vh, int nrhs, const RhsState *st,
                          double *out, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_norm2v, Vh, nrhs / 2);
    k32_norm2v<<<c.grid, c.block, 0, s>>>(c, a, Vh, nrhs, st, out, bc.partials, bc.counter);
    return cudaGetLastError();
}

cudaError_t blas32_mgs(BlasCtx &bc, void *w, void *z, const void *wi, const void *zi, long long Vh,
                       int nrhs, const RhsState *st, const double2 *cf, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_mgs, Vh, nrhs / 2);
    k32_mgs<<<c.grid, c.block, 0, s>>>(c, w, z, wi, zi, Vh, nrhs, st, cf);
    return cudaGetLastError();
}

cudaError_t blas32_normalise(BlasCtx &bc, void *w, void *z, long long Vh, int nrhs,
                             const RhsState *st, const double *nrm, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_normalise, Vh, nrhs / 2);
    k32_normalise<<<c.grid, c.block, 0, s>>>(c, w, z, Vh, nrhs, st, nrm);
    return cudaGetLastError();
}

cudaError_t blas32_gcr_update(BlasCtx &bc, void *x, void *r, const void *z, const void *w,
                              long long Vh, int nrhs, RhsState *st, const double2 *cf, int max_iter,
                              cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    const Cfg c = cfg_wave(bc, k32_gcr_update, Vh, nrhs / 2);
    k32_gcr_update<<<c.grid, c.block, 0, s>>>(c, x, r, z, w, Vh, nrhs, st, cf, max_iter, bc.partials,
                                              bc.counter, bc.n_active);
    return cudaGetLastError();
}

cudaError_t blas32_xmy(const void *a, const void *b, void *out, long long Vh, int nrhs, cudaStream_t s)
{
    const long long n = Vh * 12 * (nrhs / 2);
    k32_xmy<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(static_cast<const float4 *>(a),
                                                         static_cast<const float4 *>(b),
                                                         static_cast<float4 *>(out), n);
    return cudaGetLastError();
}

cudaError_t blas_to_f32_scaled(const double2 *r64, float4 *r32, long long Vh, int nrhs,
                               const RhsState *st, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    k32_from64<<<blocks_for(Vh * (nrhs / 2), 256), 256, 0, s>>>(r64, r32, Vh, nrhs, st);
    return cudaGetLastError();
}

cudaError_t blas_acc_f32(double2 *x64, const float4 *e32, long long Vh, int nrhs,
                         const RhsState *st, cudaStream_t s)
{
    if (nrhs % 2) return cudaErrorInvalidValue;
    k32_acc64<<<blocks_for(Vh * (nrhs / 2), 256), 256, 0, s>>>(x64, e32, Vh, nrhs, st);
    return cudaGetLastError();
}

}  // namespace dp
