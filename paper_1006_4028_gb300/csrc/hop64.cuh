// The FP64 hopping term at one (output site, RHS) in scalar FP64 arithmetic:
// spin projection, link product, accumulation and the epilogues of the FP64
// kernels.  Chiral gamma basis and layouts as in dp_internal.h.
#pragma once

#include "cplx.cuh"
#include "dp_internal.h"
#include "sites.cuh"

namespace dp {

// h = upper two spins of (1 + SG*gamma_mu) psi, SG = -1 forward, +1 backward
template <int MU, int SG, typename R>
__device__ __forceinline__ void project(const Cx<R> ps[12], Cx<R> h[6])
{
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const Cx<R> p0 = ps[a], p1 = ps[3 + a], p2 = ps[6 + a], p3 = ps[9 + a];
        if (MU == 0) {
            h[a] = SG < 0 ? p0 + p2 : p0 - p2;
            h[3 + a] = SG < 0 ? p1 + p3 : p1 - p3;
        } else if (MU == 1) {
            h[a] = SG < 0 ? p0 + mul_i(p3) : p0 - mul_i(p3);
            h[3 + a] = SG < 0 ? p1 + mul_i(p2) : p1 - mul_i(p2);
        } else if (MU == 2) {
            h[a] = SG < 0 ? p0 + p3 : p0 - p3;
            h[3 + a] = SG < 0 ? p1 - p2 : p1 + p2;
        } else {
            h[a] = SG < 0 ? p0 + mul_i(p2) : p0 - mul_i(p2);
            h[3 + a] = SG < 0 ? p1 - mul_i(p3) : p1 + mul_i(p3);
        }
    }
}

template <typename R>
__device__ __forceinline__ void axpy(R c, Cx<R> v, Cx<R> &acc)
{
    acc.re = fmx(c, v.re, acc.re);
    acc.im = fmx(c, v.im, acc.im);
}

// acc += c * (1 + SG*gamma_mu) psi given uh = U h (the upper spins); the lower
// spins are -SG e_mu^dag uh, written out per direction
template <int MU, int SG, typename R>
__device__ __forceinline__ void accumulate(Cx<R> acc[12], const Cx<R> uh[6], R c)
{
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const Cx<R> h0 = uh[a], h1 = uh[3 + a];
        axpy(c, h0, acc[a]);
        axpy(c, h1, acc[3 + a]);
        Cx<R> l2, l3;
        if (MU == 0) {
            l2 = SG < 0 ? h0 : -h0;
            l3 = SG < 0 ? h1 : -h1;
        } else if (MU == 1) {
            l2 = SG < 0 ? mul_mi(h1) : mul_i(h1);
            l3 = SG < 0 ? mul_mi(h0) : mul_i(h0);
        } else if (MU == 2) {
            l2 = SG < 0 ? -h1 : h1;
            l3 = SG < 0 ? h0 : -h0;
        } else {
            l2 = SG < 0 ? mul_mi(h0) : mul_i(h0);
            l3 = SG < 0 ? mul_i(h1) : mul_mi(h1);
        }
        axpy(c, l2, acc[6 + a]);
        axpy(c, l3, acc[9 + a]);
    }
}

// exponents of fx spinors (dslash_fx.cu: a spinor is W 2^(e - 1023 - 59), W
// int64) that stand for all components zero and for raw doubles in place of W
constexpr int kFxZero = -1, kFxRaw = -2;

// W 2^k as FP64; the exponents of fx spinors keep every non-zero result normal
__device__ __forceinline__ double fx_value(long long w, int k)
{
    const double d = (double)w;
    return w ? __hiloint2double(__double2hiint(d) + k * (1 << 20), __double2loint(d)) : 0.0;
}

// one fx spinor as FP64
__device__ __forceinline__ void load_fx(const longlong2 *b, long long cs, int e, Cx<double> s[12])
{
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const longlong2 w = b[k * cs];
        if (e == kFxRaw)
            s[k] = {__longlong_as_double(w.x), __longlong_as_double(w.y)};
        else
            s[k] = {fx_value(w.x, e - 1023 - 59), fx_value(w.y, e - 1023 - 59)};
    }
}

// one hop (SG = -1: forward with U, SG = +1: backward with U^dag); FX: the
// neighbour is an fx spinor of exponent e
template <int MU, int SG, bool FX>
__device__ __forceinline__ void hop64(Cx<double> acc[12], const double2 *nb, long long cs,
                                      const void *lk, long long Vh, long long lsite, double c, int e)
{
    Cx<double> u[9];
    load_link<LINK_F64_18, double>(lk, Vh, lsite, MU, u);
    Cx<double> ps[12];
    if (FX)
        load_fx(reinterpret_cast<const longlong2 *>(nb), cs, e, ps);
    else
        load_spinor(nb, cs, ps);
    Cx<double> h[6];
    project<MU, SG>(ps, h);
    Cx<double> uh[6];
#pragma unroll
    for (int sp = 0; sp < 2; sp++)
#pragma unroll
        for (int a = 0; a < 3; a++) {
            Cx<double> t;
            if (SG < 0) {
                t = cmul(u[3 * a], h[3 * sp]);
                t = cfma(u[3 * a + 1], h[3 * sp + 1], t);
                t = cfma(u[3 * a + 2], h[3 * sp + 2], t);
            } else {
                t = cjmul(u[a], h[3 * sp]);
                t = cjfma(u[3 + a], h[3 * sp + 1], t);
                t = cjfma(u[6 + a], h[3 * sp + 2], t);
            }
            uh[3 * sp + a] = t;
        }
    accumulate<MU, SG>(acc, uh, c);
}

// one output spinor: hopping term of site s, RHS r, with the epilogue
template <int EPI, bool FX>
__device__ __forceinline__ void hop_site64_body(const DslashParams &p, long long s, int r)
{
    const Geom &g = p.g;
    const int n = p.nrhs;
    const Nbr nb = neighbours(g, s, p.parity);
    const long long cs = g.Vh * n;
    const double2 *in = static_cast<const double2 *>(p.in) + r;
    const int grp = p.grp_of[r];
    const double *ht = static_cast<const double *>(p.hop) + (long long)grp * 8 * g.Lmax;
    const void *lown = p.links[p.parity], *loth = p.links[1 - p.parity];
    const long long Vh = g.Vh;
    auto ex = [&](int site) { return FX ? p.in_exp[(long long)site * n + r] : 0; };
    Cx<double> acc[12];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = {0.0, 0.0};
    hop64<0, -1, FX>(acc, in + nb.f[0] * n, cs, lown, Vh, s, ht[0 * g.Lmax + nb.t], ex(nb.f[0]));
    hop64<0, +1, FX>(acc, in + nb.b[0] * n, cs, loth, Vh, nb.b[0], ht[1 * g.Lmax + nb.t], ex(nb.b[0]));
    hop64<1, -1, FX>(acc, in + nb.f[1] * n, cs, lown, Vh, s, ht[2 * g.Lmax + nb.x], ex(nb.f[1]));
    hop64<1, +1, FX>(acc, in + nb.b[1] * n, cs, loth, Vh, nb.b[1], ht[3 * g.Lmax + nb.x], ex(nb.b[1]));
    hop64<2, -1, FX>(acc, in + nb.f[2] * n, cs, lown, Vh, s, ht[4 * g.Lmax + nb.y], ex(nb.f[2]));
    hop64<2, +1, FX>(acc, in + nb.b[2] * n, cs, loth, Vh, nb.b[2], ht[5 * g.Lmax + nb.y], ex(nb.b[2]));
    hop64<3, -1, FX>(acc, in + nb.f[3] * n, cs, lown, Vh, s, ht[6 * g.Lmax + nb.z], ex(nb.f[3]));
    hop64<3, +1, FX>(acc, in + nb.b[3] * n, cs, loth, Vh, nb.b[3], ht[7 * g.Lmax + nb.z], ex(nb.b[3]));

    const long long me = s * n + r;
    double2 *out = static_cast<double2 *>(p.out) + me;
    const double2 *xin = static_cast<const double2 *>(p.x) + me;
    Cx<double> v[12];
    if (EPI == EPI_HOP || EPI == EPI_XPY || EPI == EPI_XMY_G5) {
        if (EPI == EPI_XPY) {
            load_spinor(xin, cs, v);
#pragma unroll
            for (int j = 0; j < 12; j++) acc[j] = v[j] + acc[j];
        }
        if (EPI == EPI_XMY_G5) {  // gamma5 = +1 on spins 0, 1 and -1 on spins 2, 3
            load_spinor(xin, cs, v);
#pragma unroll
            for (int j = 0; j < 12; j++) acc[j] = j < 6 ? v[j] - acc[j] : v[j] + acc[j];
        }
        store_spinor(out, cs, acc);
        return;
    }
    if (EPI == EPI_AINV_XMY) {
        load_spinor(xin, cs, v);
#pragma unroll
        for (int j = 0; j < 12; j++) acc[j] = v[j] - acc[j];
    }
    const double2 *cl = static_cast<const double2 *>(p.clov[grp]);
    Cx<double> w[12];
#pragma unroll
    for (int blk = 0; blk < 2; blk++) {
        double m[36];
        load_clover_block(cl, Vh, s, blk, m);
        herm6_apply(m, acc + 6 * blk, w + 6 * blk);
    }
    if (EPI == EPI_XMY_AINV) {
        load_spinor(xin, cs, v);
#pragma unroll
        for (int j = 0; j < 12; j++) w[j] = v[j] - w[j];
    }
    store_spinor(out, cs, w);
}

}  // namespace dp
