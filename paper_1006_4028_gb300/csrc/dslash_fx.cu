// The FP64 hopping term in integer arithmetic: the operator of dslash.cu's
// k_dslash64 (same arguments, same epilogues, FP64 in and out) with its
// products on the integer multiplier.
//
// Why: GB300 issues one FP64 FMA per warp and SM quarter every 64 cycles (67
// measured) but one 32 x 32 + 64 bit integer multiply-add (mad.wide.s32) every
// 2 (2.2 measured).  k_dslash64 needs 1128 FP64 instructions per output spinor
// and sat on that pipe: 7.4 ms for 12 right-hand sides on 48x24^3 whose bytes
// take 0.31 ms.
//
// Numbers: block floating point ("fx" spinors: the layout of an FP64 spinor
// field with each double replaced by an int64 W, and one exponent per (site,
// RHS)).  The 24 reals of a spinor are W 2^(e - 1023 - 59), e the biased
// exponent of the largest, whose leading bit is bit 59.  A neighbour is
// projected in these integers, and the projected h held as two limbs, h = hi
// 2^32 + lo 2, lo in [0, 2^31).  Links (unitary: the field's flag) are U 2^60 =
// hi 2^31 + lo, lo in [-2^30, 2^30).  A product is three mad.wide (hi hi, hi lo
// + lo hi; lo lo lies below 2^-57 and has no preferred sign, since a link's lo
// has none, and is left out).  Sums of products stay exact 64-bit integers;
// each direction adds round(U h) in units of 2^-56 into 24 int64 accumulators,
// whose exponent R is the largest seen so far (a larger one shifts the
// accumulators down).  The clover inverse is applied the same way on the
// renormalised accumulators; the result is rounded to FP64 once, or written as
// an fx spinor for the next launch.  So a component's error is about 2^-55 of
// the largest one around where a chain of FP64 operations leaves about 2^-53.
// Bounds (rows and columns of U of norm 1, six products a sum): hi hi below 2^59.3, hi lo +
// lo hi below 2^62.5, eight directions below 2^62.3; clover (twelve products of
// anything below 2^59): hi hi below 2^58.6, hi lo + lo hi below 2^62.9.
//
// Small components: what FP64 leaves of a component is about 2^-53 of the sum T
// of its terms' magnitudes.  Where T is near the largest neighbour's size R, as
// on links that mix the colours, 2^-55 R is less than that; where it is not
// (links near the unit matrix, one colour much smaller than another) it could
// be all of a component.  A result with a complex component below 2^-10 R is
// therefore looked at again (mixes): if some neighbour's projected h is
// nowhere below 2^-10 R, T is at least that (a row or column of U has norm 1,
// so its entries' magnitudes add up to 1 or more) and the component is small by
// cancellation, else the FP64 arithmetic answers.  A spinor with a non-zero
// component below 2^-16 of its largest is not converted.  So a component is
// off by at most 2^-41 T (worst case of all truncations: 2^-51 R; 2^-36 T where
// the inverse clover block has a diagonal entry near a thirty-second of its
// largest), and a result by 2^-55 of its norm.  On rough links one thread in
// some 10^5 looks again and the first neighbour answers.  Cost: A^-1 D 540 ->
// 549 us for 12 RHS on 32x16^3, the FP64 solve there 0.2 % (5 % without the
// second look).
//
// On links that hardly mix the colours a point-source solve falls back often,
// and a thread alone on the FP64 pipe is slow: 16x8^3, FP64 solve, links exp(i
// eps H), eps = 0.05 / 0.02 / 0.01 / 0.006: 8.5 / 10.7 / 21 / 23 ms against
// 7.8 without the guard and 16.7 with k_dslash64.  A field with an entry below
// 2^-12 in more than one link of 500 (eps below about 0.015; diagonal links)
// has k_dslash64 throughout (Field::fx).
//
// What the integers cannot hold is handed to the FP64 arithmetic, per thread
// (hop_site64, the code of k_dslash64): a spinor with an infinity or NaN or
// whose largest component is below 2^-942 or near the overflow threshold, or
// with a small one as above, is kept as raw doubles (exponent kFxRaw), and its
// neighbours take that path, as do sites with such entries in the clover block
// or a result out of range.
//
// Why a converted copy: converting in the thread that loads a neighbour (each
// spinor eight times) cost 13 integer instructions or one 68-cycle cvt per
// real and 48 registers for the raw spinor: 0.61 ms for 12 RHS on 32x16^3.
// Converting once (k_to_fx, a pass at copy rate: 0.04 ms) leaves the hop kernel
// with adds and products.  A^-1 D with the conversion, all RHS active: 12 RHS on
// 32x16^3 0.55 ms where k_dslash64 takes 1.49, on 48x24^3 2.72 against 7.40
// (x - A^-1 D 0.1 more: its 24 subtractions are on the FP64 pipe), one RHS on
// 32x16^3 0.117 against 0.150.  What holds it now is latency: 10.5 thousand
// instructions a warp, four warps a quarter (128 registers: 24 int64
// accumulators alone are 48), 0.41 of the issue slots, fixed-latency waits
// first; at 96 registers for five warps it spills and took a half more.
//
// Layout of the work: a block holds whole sites, all right-hand sides of each,
// one thread per (site, RHS).  The limbs of a direction's links (and of a
// clover block) are made once per site by all threads of the block, in shared
// memory; U^dag is transposed and conjugated there, so both hops of a
// direction multiply alike.
#include <type_traits>

#include "cplx.cuh"
#include "dp_internal.h"
#include "hop64.cuh"
#include "sites.cuh"

namespace dp {
namespace {

typedef long long i64;

struct L2w {  // limbs of a real
    int hi, lo;
};

__device__ __forceinline__ i64 madw(int a, int b, i64 c)
{
    i64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// logical right shift; amounts of 64 and above give 0
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, int n)
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}

// v as an integer with the leading bit of numbers of biased exponent `base`
// (>= 64, at least v's) at bit 59.  (In integer instructions: cvt.s64.f64
// occupies the FP64 pipe for 68 cycles a warp.)
__device__ __forceinline__ i64 w59(double v, int base)
{
    const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
    const unsigned m = (h & 0xfffffu) | 0x100000u;
    const i64 w = (i64)shr64(((unsigned long long)__funnelshift_l(l, m, 7) << 32) | (l << 7),
                             base - (int)((h >> 20) & 0x7ffu));
    const i64 s = (i64)((int)h >> 31);
    return (w ^ s) - s;
}

// W = hi 2^32 + lo 2 (the last bit dropped)
__device__ __forceinline__ L2w cut32(i64 w)
{
    return {(int)(w >> 32), (int)((unsigned)w >> 1)};
}
// W = hi 2^31 + lo, lo in [-2^30, 2^30)
__device__ __forceinline__ L2w cut31(i64 w)
{
    return {(int)((w + (1ll << 30)) >> 31), (int)((unsigned)w << 1) >> 1};
}

__device__ __forceinline__ unsigned mag_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// v 2^e rounded to FP64; ok = false outside the normal range
__device__ __forceinline__ double to_double(i64 v, int e, bool &ok)
{
    const double d = __ll2double_rn(v);
    const int h = __double2hiint(d);
    const int x = ((h >> 20) & 0x7ff) + e;
    if (v == 0) return 0.0;
    if (x < 1 || x > 2046) ok = false;
    return __hiloint2double(h + (int)((unsigned)e << 20), __double2loint(d));
}

// position of the leading bit of the largest |v| whose high words are or-ed in
__device__ __forceinline__ unsigned top_or(i64 v)
{
    const int a = (int)(v >> 32);
    return (unsigned)(a ^ (a >> 31));
}

// the smallest of N complex integers, by the high word of its larger part
template <int N>
__device__ __forceinline__ unsigned least(const i64 *re, const i64 *im)
{
    unsigned m = ~0u;
#pragma unroll
    for (int k = 0; k < N; k++) m = min(m, top_or(re[k]) | top_or(im[k]));
    return m;
}

constexpr int kSmall = 10;  // results with a component below 2^-kSmall R are looked at again
constexpr int kKeep = 16;   // spinors with one below 2^-kKeep of the largest are not converted
constexpr int kMinExp = 81, kMaxExp = 2040;  // biased exponents of the blocks the integers take
constexpr int kHalf = 1023 + 59;             // value = W 2^(e - kHalf)

// how a launch divides its work
struct FxLaunch {
    int sites;             // sites per block
    int ngrp;              // distinct groups among the RHS
    int8_t grp[kMaxGroups];
    int8_t of[kMaxRhs];    // RHS -> index into grp
};

constexpr int kNoExp = -(1 << 20);   // R before the first contribution

struct Acc {
    i64 re[12], im[12];
    int R;  // value = acc 2^(R - 1023 - 56)
};

__device__ __forceinline__ void raise(Acc &a, int R)
{
    if (a.R == kNoExp) a.R = R;
    const int n = min(R - a.R, 63);
    if (n > 0) {
#pragma unroll
        for (int k = 0; k < 12; k++) {
            a.re[k] >>= n;
            a.im[k] >>= n;
        }
        a.R = R;
    }
}

// acc -= c (1 + SG gamma_mu) U psi for one fx neighbour of exponent e, with the upper spins of
// the projection h_0 = p_0 + f_0 q_0, h_1 = p_1 + f_1 q_1 (q_0, q_1 the lower
// spins of psi in the order this mu pairs them with the upper ones), f = +-1
// (IMAG = false: mu = 0, 2) or +-i (IMAG: mu = 1, 3), minus where flip_0,
// flip_1 are -1 (else 0); acc's lower spins are held in the order of q, with
// that sign taken out, and get conj(|f|) (U h).  sl: the limbs of U (or U^dag)
// of this site, row-major: (re hi, re lo, im hi, im lo), then (-im hi, -im lo)
template <bool IMAG>
__device__ __forceinline__ void hop_fx(Acc &acc, const longlong2 *up, const longlong2 *q0, const longlong2 *q1,
                                       i64 cs, int e, i64 flip0, i64 flip1, const int4 *sl, double c, bool &bad)
{
    const unsigned chi = (unsigned)__double2hiint(c), clo = (unsigned)__double2loint(c);
    const int ecb = (int)((chi >> 20) & 0x7ffu);
    if (e == kFxRaw) bad = true;
    // a zero neighbour adds nothing, nor is there a hop across a Dirichlet boundary
    if (e < 0 || ((chi & 0x7fffffffu) | clo) == 0) return;
    if (ecb < 64 || ecb > 1983) {
        bad = true;
        return;
    }
    // -c = 2^k: only the exponent; else -c = +-cm 2^(k + 1), cm in [1/2, 1), which multiplies h
    const bool pow2 = (chi & 0x800fffffu) == 0x80000000u && clo == 0;
    const int eff = e + ecb - 1023 + (pow2 ? 0 : 1);
    raise(acc, eff);
    const int down = min(acc.R - eff, 63);
    L2w hr[6], hm[6];
#pragma unroll
    for (int s = 0; s < 2; s++) {
        const i64 m = s ? flip1 : flip0;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int k = 3 * s + a;
            const longlong2 p = __ldg(up + k * cs), q = __ldg((s ? q1 : q0) + a * cs);
            const i64 qr = q.x ^ m, qi = q.y ^ m;  // (-q - 1: one unit of 2^-59)
            hr[k] = cut32((IMAG ? p.x - qi : p.x + qr) >> down);
            hm[k] = cut32((IMAG ? p.y + qr : p.y + qi) >> down);
        }
    }
    if (!pow2) {  // h times cm, in the units of h
        const double m = __hiloint2double((int)((chi & 0x800fffffu) | (1022u << 20)), (int)clo);
        const L2w cm = cut31(w59(-m, 1022));  // cm 2^60
        auto mul = [&](L2w &x) {
            const i64 hh = madw(cm.hi, x.hi, 0);
            const i64 xx = madw(cm.lo, x.hi, madw(cm.hi, x.lo, 1ll << 27));
            x = cut32((hh << 3) + (xx >> 28));
        };
#pragma unroll
        for (int k = 0; k < 6; k++) {
            mul(hr[k]);
            mul(hm[k]);
        }
    }
    const int2 *neg = reinterpret_cast<const int2 *>(sl + 9);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int4 u[3] = {sl[3 * a], sl[3 * a + 1], sl[3 * a + 2]};
        const int2 v[3] = {neg[3 * a], neg[3 * a + 1], neg[3 * a + 2]};
#pragma unroll
        for (int s = 0; s < 2; s++) {
            i64 ph = 0, px = 1ll << 30, mh = 0, mx2 = 1ll << 30;
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const L2w x = hr[3 * s + b], y = hm[3 * s + b];
                ph = madw(v[b].x, y.hi, madw(u[b].x, x.hi, ph));
                px = madw(u[b].y, x.hi, madw(u[b].x, x.lo, px));
                px = madw(v[b].y, y.hi, madw(v[b].x, y.lo, px));
                mh = madw(u[b].z, x.hi, madw(u[b].x, y.hi, mh));
                mx2 = madw(u[b].y, y.hi, madw(u[b].x, y.lo, mx2));
                mx2 = madw(u[b].w, x.hi, madw(u[b].z, x.lo, mx2));
            }
            const i64 tr = ph + (px >> 31), ti = mh + (mx2 >> 31);
            const int k = 3 * s + a;
            acc.re[k] += tr;
            acc.im[k] += ti;
            if (IMAG) {  // -i t
                acc.re[6 + k] += ti;
                acc.im[6 + k] -= tr;
            } else {
                acc.re[6 + k] += tr;
                acc.im[6 + k] += ti;
            }
        }
    }
}

// change the sign under which acc holds its lower spin s
__device__ __forceinline__ void flip_lower(Acc &acc, int s)
{
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int k = 6 + 3 * s + a;
        acc.re[k] = -acc.re[k];
        acc.im[k] = -acc.im[k];
    }
}

// shared memory of a block: neighbour indices and coordinates per site, then
// the limbs of a direction's links ([site][kLinkSlot]: 9 int4, then 9 int2)
// or of a clover block ([group of the launch][site][18 int4], 36 reals)
struct SiteIx {
    int nb[8];
    int t, x, y, z;
};
constexpr int kLinkSlot = 14;  // int4
constexpr int kFxBlock = 128;  // threads of a block at most; 128 registers each

// links of one direction -> limbs, U forward, U^dag backward; this thread
// makes the entries e0, e0 + es, ... of the block's site j0
__device__ __forceinline__ void stage_links(int4 *buf, const double2 *lk, i64 Vh, const SiteIx *ix,
                                            i64 s0, int j0, int e0, int es, int mu, bool back)
{
    const i64 site = back ? (i64)ix[j0].nb[2 * mu + 1] : s0 + j0;
    int4 *slot = buf + j0 * kLinkSlot;
    for (int e = e0; e < 9; e += es) {
        const double2 v = __ldg(lk + ((i64)mu * 9 + e) * Vh + site);
        const i64 w = w59(back ? -v.y : v.y, 1023) << 1;
        const L2w r = cut31(w59(v.x, 1023) << 1), i = cut31(w), m = cut31(-w);
        const int o = back ? 3 * (e % 3) + e / 3 : e;
        slot[o] = make_int4(r.hi, r.lo, i.hi, i.lo);
        reinterpret_cast<int2 *>(slot + 9)[o] = make_int2(m.hi, m.lo);
    }
}

// the same output spinor in FP64 arithmetic, out of line (rare)
template <int EPI>
__device__ __noinline__ void hop_site64(const DslashParams &p, i64 s, int r)
{
    hop_site64_body<EPI, true>(p, s, r);
}

// whether some neighbour's projected h (times its hop factor) has no complex
// component below 2^-kSmall of the largest neighbour's size, of exponent R
// (out of line, rare)
__device__ __noinline__ bool mixes(const DslashParams &p, i64 s, int r, int R)
{
    const Geom &g = p.g;
    const Nbr nb = neighbours(g, s, p.parity);
    const i64 cs = g.Vh * p.nrhs;
    const double *ht = static_cast<const double *>(p.hop) + (i64)p.grp_of[r] * 8 * g.Lmax;
    const int x[4] = {nb.t, nb.x, nb.y, nb.z};
    bool yes = false;
#pragma unroll
    for (int d = 0; d < 8; d++) {
        if (yes) break;  // (on rough links the first neighbour answers)
        const int mu = d >> 1;
        const i64 at = (i64)(d & 1 ? nb.b[mu] : nb.f[mu]) * p.nrhs + r;
        const unsigned chi = (unsigned)__double2hiint(__ldg(ht + d * g.Lmax + x[mu]));
        const int e = __ldg(p.in_exp + at) + (int)((chi >> 20) & 0x7ffu) - 1023;
        const longlong2 *v = static_cast<const longlong2 *>(p.in) + at;
        const i64 f0 = d & 1 ? -1 : 0, f1 = mu >= 2 ? ~f0 : f0;
        const int l0 = mu == 1 || mu == 2 ? 9 : 6;  // the lower spin that goes with upper spin 0
        unsigned m = ~0u;
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const longlong2 a = __ldg(v + k * cs), q = __ldg(v + (k < 3 ? l0 + k : 15 - l0 + k - 3) * cs);
            const i64 qr = q.x ^ (k < 3 ? f0 : f1), qi = q.y ^ (k < 3 ? f0 : f1);
            m = min(m, mu & 1 ? top_or(a.x - qi) | top_or(a.y + qr) : top_or(a.x + qr) | top_or(a.y + qi));
        }
        // leading bit of the smallest against bit 59
        yes = m != 0 && e + (63 - __clz((int)m)) - 59 >= R - kSmall;
    }
    return yes;
}

template <int EPI>
__global__ void __launch_bounds__(kFxBlock, 512 / kFxBlock)
    k_dslash_fx(const __grid_constant__ DslashParams p, const __grid_constant__ FxLaunch fl)
{
    extern __shared__ int4 smem[];
    const Geom &g = p.g;
    const i64 Vh = g.Vh;
    const int n = p.nrhs, spb = fl.sites;
    SiteIx *ix = reinterpret_cast<SiteIx *>(smem);
    int4 *buf = smem + spb * (int)(sizeof(SiteIx) / sizeof(int4));
    __shared__ int cmax[kFxBlock];  // largest magnitude (high word) per (group of the launch, site)
    // the groups with a live RHS: an idle group's clover pointer may be that of
    // an inverse freed since its job ended
    __shared__ unsigned groups;
    if (threadIdx.x == 0) groups = 0;
    const i64 s0 = (i64)blockIdx.x * spb;
    const int ns = (int)min((i64)spb, Vh - s0);
    const int j = threadIdx.x / n, r = threadIdx.x - j * n;
    const i64 s = s0 + j;
    const bool live = j < ns && (!p.active || p.active[r * p.active_stride]);
    if (!__syncthreads_or(live)) return;  // (converged RHS fill the block)
    if (live) atomicOr(&groups, 1u << fl.of[r]);  // (barriers before its first use)
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
        const Nbr nb = neighbours(g, s0 + k, p.parity);
        SiteIx q;
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            q.nb[2 * mu] = nb.f[mu];
            q.nb[2 * mu + 1] = nb.b[mu];
        }
        q.t = nb.t;
        q.x = nb.x;
        q.y = nb.y;
        q.z = nb.z;
        ix[k] = q;
    }
    const i64 cs = Vh * n;
    const longlong2 *in = static_cast<const longlong2 *>(p.in) + r;
    const int grp = live ? p.grp_of[r] : 0;
    const double *ht = static_cast<const double *>(p.hop) + (i64)grp * 8 * g.Lmax;
    const double2 *lown = static_cast<const double2 *>(p.links[p.parity]);
    const double2 *loth = static_cast<const double2 *>(p.links[1 - p.parity]);
    Acc acc;
#pragma unroll
    for (int k = 0; k < 12; k++) acc.re[k] = acc.im[k] = 0;
    acc.R = kNoExp;
    bool bad = false;
    // this thread's share of the staging: entries e0, e0 + es, ... of site j0
    const int j0 = threadIdx.x % ns, es = blockDim.x / ns;
    const int e0 = (int)threadIdx.x / ns < es ? threadIdx.x / ns : 18;  // (the rest of the block: none)
    // (loading the next direction's neighbour, exponent and link ahead, into L1,
    // registers and a second buffer, changed nothing: 0.51 ms against 0.50)
    auto direction = [&](int mu, bool back, bool swapped, auto imag) {
        __syncthreads();
        stage_links(buf, back ? loth : lown, Vh, ix, s0, j0, e0, es, mu, back);
        __syncthreads();
        if (!live) return;
        const SiteIx &q = ix[j];
        const i64 at = (i64)q.nb[2 * mu + back] * n;
        const longlong2 *nb = in + at;
        const int x = mu == 0 ? q.t : mu == 1 ? q.x : mu == 2 ? q.y : q.z;
        // backward hops turn both signs of the projection, mu = 2, 3 pair a + with a -
        const i64 f0 = back ? -1 : 0, f1 = mu >= 2 ? ~f0 : f0;
        hop_fx<decltype(imag)::value>(acc, nb, nb + (swapped ? 9 : 6) * cs, nb + (swapped ? 6 : 9) * cs, cs,
                                      __ldg(p.in_exp + at + r), f0, f1, buf + kLinkSlot * j,
                                      __ldg(ht + (2 * mu + back) * g.Lmax + x), bad);
    };
    // One body for the directions with real factors (mu = 0, then 2), one for
    // the imaginary ones (3, then 1): with eight straight-line bodies (190 KB of
    // instructions) warps waited for instructions more than for anything else.
    // mu = 2 and 1 pair the lower spins the other way round, so acc's are
    // exchanged half way; the signs of (f_0, f_1) go ++ +- -- -+ and, after
    // the exchange, +- ++ -+ --, one change from each to the next.
#pragma unroll 1
    for (int half = 0; half < 2; half++) {
#pragma unroll 1
        for (int back = 0; back < 2; back++) {
            direction(half ? 2 : 0, back, half, std::false_type{});
            flip_lower(acc, 1);
            direction(half ? 1 : 3, back, half, std::true_type{});
            if (!back) flip_lower(acc, 0);
        }
#pragma unroll
        for (int k = 6; k < 9; k++) {
            const i64 a = acc.re[k], b = acc.im[k];
            acc.re[k] = acc.re[k + 3];
            acc.im[k] = acc.im[k + 3];
            acc.re[k + 3] = a;
            acc.im[k + 3] = b;
        }
    }
    flip_lower(acc, 0);
    flip_lower(acc, 1);
    const i64 me = s * n + r;
    double2 *out = static_cast<double2 *>(p.out) + me;
    const double2 *xin = static_cast<const double2 *>(p.x) + me;
    if (EPI == EPI_HOP || EPI == EPI_XPY || EPI == EPI_XMY_G5) {
        if (live) {
            bool ok = !bad;
            // (a component of the largest neighbour's size has its leading bit at 56)
            if (ok && acc.R != kNoExp && !(least<12>(acc.re, acc.im) >> (56 - 32 - kSmall))) ok = mixes(p, s, r, acc.R);
            double2 w[12];
#pragma unroll
            for (int k = 0; k < 12; k++)  // acc holds -D
                w[k] = make_double2(to_double(-acc.re[k], acc.R - 1023 - 56, ok),
                                    to_double(-acc.im[k], acc.R - 1023 - 56, ok));
            if (ok) {
#pragma unroll
                for (int k = 0; k < 12; k++) {
                    if (EPI != EPI_HOP) {
                        const double2 v = __ldg(xin + k * cs);
                        const bool minus = EPI == EPI_XMY_G5 && k < 6;
                        w[k].x = minus ? v.x - w[k].x : v.x + w[k].x;
                        w[k].y = minus ? v.y - w[k].y : v.y + w[k].y;
                    }
                    out[k * cs] = w[k];
                }
            } else {
                hop_site64<EPI>(p, s, r);
            }
        }
        return;
    }
    if (EPI == EPI_AINV_XMY && live) {  // acc <- x - D: x joins in the units of acc
        double2 v[12];
        unsigned mx = 0, any = 0;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            v[k] = __ldg(xin + k * cs);
            mx = max(mx, max(mag_hi(v[k].x), mag_hi(v[k].y)));
            any |= (unsigned)__double2loint(v[k].x) | (unsigned)__double2loint(v[k].y);
        }
        const int em = (int)(mx >> 20);
        if (em > kMaxExp || (em < kMinExp && (mx | any))) bad = true;
        if (em >= kMinExp && em <= kMaxExp) {
            raise(acc, em);
#pragma unroll
            for (int k = 0; k < 12; k++) {
                acc.re[k] += (w59(v[k].x, acc.R) + 4) >> 3;
                acc.im[k] += (w59(v[k].y, acc.R) + 4) >> 3;
            }
        }
    }
    bool ok = !bad, small = false, hard = false;
    int wexp[2] = {0, 0};
#pragma unroll
    for (int blk = 0; blk < 2; blk++) {
        // the inverse block of every (group of the launch, site): its largest
        // exponent, then its limbs (leading bit at 58); bit 0 of cmax: a diagonal
        // entry is below 2^-kSmall/2 of the largest, so that its row may add little
        // of x to the result
        __syncthreads();
        for (int k = threadIdx.x; k < fl.ngrp * ns; k += blockDim.x) cmax[k] = 0;
        __syncthreads();
        for (int gi = 0; gi < fl.ngrp; gi++) {
            if (!(groups >> gi & 1)) continue;
            const double2 *cl = static_cast<const double2 *>(p.clov[fl.grp[gi]]) + (i64)18 * blk * Vh + s0 + j0;
            unsigned mx = 0;
            for (int e = e0; e < 18; e += es) {
                const double2 v = __ldg(cl + (i64)e * Vh);
                mx = max(mx, max(mag_hi(v.x), mag_hi(v.y)));
            }
            if (mx) atomicMax(&cmax[gi * ns + j0], (int)(mx & ~1u));
        }
        __syncthreads();
        for (int gi = 0; gi < fl.ngrp; gi++) {
            if (!(groups >> gi & 1)) continue;
            const double2 *cl = static_cast<const double2 *>(p.clov[fl.grp[gi]]) + (i64)18 * blk * Vh + s0 + j0;
            const int base = max((cmax[gi * ns + j0] >> 20) + 1, 64);
            for (int e = e0; e < 18; e += es) {
                const double2 v = __ldg(cl + (i64)e * Vh);
                const L2w a = cut31(w59(v.x, base)), b = cut31(w59(v.y, base));
                buf[(gi * ns + j0) * 18 + e] = make_int4(a.hi, a.lo, b.hi, b.lo);
                if (e < 3 && min(a.hi < 0 ? -a.hi : a.hi, b.hi < 0 ? -b.hi : b.hi) < 1 << (27 - kSmall / 2))
                    atomicOr(&cmax[gi * ns + j0], 1);
            }
        }
        __syncthreads();
        if (!live) continue;
        const int gs = fl.of[r] * ns + j;
        const int eb = cmax[gs] >> 20;
        if (eb < kMinExp || eb > kMaxExp) ok = false;
        // renormalise the 12 reals of this chiral block: leading bit to 62, then 58
        unsigned top = 0;
#pragma unroll
        for (int k = 0; k < 6; k++) top |= top_or(acc.re[6 * blk + k]) | top_or(acc.im[6 * blk + k]);
        const int sh = top ? __clz((int)top) - 1 : 31;
        L2w xr[6], xi[6];
#pragma unroll
        for (int k = 0; k < 6; k++) {
            xr[k] = cut32((acc.re[6 * blk + k] << sh) >> 4);
            xi[k] = cut32((acc.im[6 * blk + k] << sh) >> 4);
        }
        const int we = eb + acc.R - sh - 2 * 1023 - 51;
        const int4 *m = buf + gs * 18;
        const int2 *m2 = reinterpret_cast<const int2 *>(m);
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const int2 d = m2[i];
            i64 ph = madw(d.x, xr[i].hi, 0), px = madw(d.y, xr[i].hi, madw(d.x, xr[i].lo, 1ll << 26));
            i64 mh = madw(d.x, xi[i].hi, 0), mx = madw(d.y, xi[i].hi, madw(d.x, xi[i].lo, 1ll << 26));
            i64 qh = 0, qx = 0, rh = 0, rx = 0;  // subtracted parts
#pragma unroll
            for (int k = 0; k < 6; k++) {
                if (k == i) continue;
                const int lo = i < k ? i : k, hi = i < k ? k : i;
                // packed upper triangle, row-major: entry (lo, hi) is the complex number 3 + index
                const int4 u = m[3 + lo * 5 - lo * (lo - 1) / 2 + hi - lo - 1];
                ph = madw(u.x, xr[k].hi, ph);
                px = madw(u.y, xr[k].hi, madw(u.x, xr[k].lo, px));
                mh = madw(u.x, xi[k].hi, mh);
                mx = madw(u.y, xi[k].hi, madw(u.x, xi[k].lo, mx));
                if (i < k) {  // a x: re -= im im, im += im re
                    qh = madw(u.z, xi[k].hi, qh);
                    qx = madw(u.w, xi[k].hi, madw(u.z, xi[k].lo, qx));
                    mh = madw(u.z, xr[k].hi, mh);
                    mx = madw(u.w, xr[k].hi, madw(u.z, xr[k].lo, mx));
                } else {  // conj(a) x: re += im im, im -= im re
                    ph = madw(u.z, xi[k].hi, ph);
                    px = madw(u.w, xi[k].hi, madw(u.z, xi[k].lo, px));
                    rh = madw(u.z, xr[k].hi, rh);
                    rx = madw(u.w, xr[k].hi, madw(u.z, xr[k].lo, rx));
                }
            }
            const i64 vr = ((ph - qh) << 4) + ((px - qx) >> 27), vi = ((mh - rh) << 4) + ((mx - rx) >> 27);
            // acc was -D (x - D for A^-1 (x - D))
            acc.re[6 * blk + i] = EPI != EPI_AINV_XMY ? -vr : vr;
            acc.im[6 * blk + i] = EPI != EPI_AINV_XMY ? -vi : vi;
        }
        wexp[blk] = we;
        // (the largest neighbour's size times the block's largest entry: bit 51 + sh)
        const int low = 51 - 32 - kSmall + sh;
        if (low > 30 || !(least<6>(acc.re + 6 * blk, acc.im + 6 * blk) >> low)) {
            small = true;
            hard = hard || (cmax[gs] & 1);
        }
        if (EPI == EPI_AINV && p.out_exp) continue;
#pragma unroll
        for (int k = 6 * blk; k < 6 * blk + 6; k++) {
            double2 w = make_double2(to_double(acc.re[k], we, ok), to_double(acc.im[k], we, ok));
            if (EPI == EPI_XMY_AINV) {
                const double2 v = __ldg(xin + k * cs);
                w = make_double2(v.x - w.x, v.y - w.y);
            }
            out[k * cs] = w;
        }
    }
    if (!live) return;
    if (ok && small && acc.R != kNoExp) ok = !hard && mixes(p, s, r, acc.R);
    if (EPI == EPI_AINV && p.out_exp) {
        // an fx spinor: the largest leading bit of the two chiral blocks to bit 59
        int lead = kNoExp;
#pragma unroll
        for (int blk = 0; blk < 2; blk++) {
            i64 any = 0;
            unsigned top = 0;
#pragma unroll
            for (int k = 6 * blk; k < 6 * blk + 6; k++) {
                top |= top_or(acc.re[k]) | top_or(acc.im[k]);
                any |= acc.re[k] | acc.im[k];
            }
            if (any) lead = max(lead, wexp[blk] + (top ? 63 - __clz((int)top) : 31));
        }
        const int e = lead == kNoExp ? kFxZero : lead + 1023;
        if (ok && (lead == kNoExp || (e >= kMinExp && e <= kMaxExp))) {
            longlong2 *wo = reinterpret_cast<longlong2 *>(out);
#pragma unroll
            for (int k = 0; k < 12; k++) {
                const int sh = wexp[k / 6] - lead + 59;
                const i64 a = acc.re[k], b = acc.im[k];
                const int dn = min(-sh, 63);
                wo[k * cs] = sh >= 0 ? make_longlong2(a << min(sh, 63), b << min(sh, 63))
                                     : make_longlong2(a >> dn, b >> dn);
            }
            p.out_exp[me] = e;
            return;
        }
        ok = false;
        p.out_exp[me] = kFxRaw;
    }
    if (!ok) hop_site64<EPI>(p, s, r);
}

// ---- conversions ----

// FP64 spinors -> fx spinors (in place: in == w), the RHS with mask[r * stride] != 0
__global__ void __launch_bounds__(128) k_to_fx(const double2 *in, longlong2 *w, int *ex, i64 Vh, int n,
                                               const int *mask, int stride)
{
    const i64 gid = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= Vh * n) return;
    if (mask && !mask[(int)(gid % n) * stride]) return;
    const i64 cs = Vh * n;
    double2 v[12];
    unsigned mx = 0, mn = ~0u;  // largest and smallest non-zero complex component
#pragma unroll
    for (int k = 0; k < 12; k++) {
        v[k] = in[k * cs + gid];
        const unsigned m = max(mag_hi(v[k].x), mag_hi(v[k].y));
        mx = max(mx, m);
        if (m | (unsigned)__double2loint(v[k].x) | (unsigned)__double2loint(v[k].y)) mn = min(mn, m);
    }
    const int em = (int)(mx >> 20);
    int e = em;
    if (mn == ~0u) e = kFxZero;
    else if (em > kMaxExp || em < kMinExp || (int)(mn >> 20) < em - kKeep) e = kFxRaw;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        longlong2 o;
        if (e == kFxRaw)
            o = make_longlong2(__double_as_longlong(v[k].x), __double_as_longlong(v[k].y));
        else if (e == kFxZero)
            o = make_longlong2(0, 0);
        else
            o = make_longlong2(w59(v[k].x, em), w59(v[k].y, em));
        w[k * cs + gid] = o;
    }
    ex[gid] = e;
}

// out = a - t for fx spinors t, the RHS with mask[r] != 0
__global__ void __launch_bounds__(128) k_sub_fx(const double2 *a, const longlong2 *t, const int *ex, double2 *out,
                                                i64 Vh, int n, const int *mask)
{
    const i64 gid = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= Vh * n || !mask[gid % n]) return;
    const i64 cs = Vh * n;
    Cx<double> v[12];
    load_fx(t + gid, cs, ex[gid], v);
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const double2 x = a[k * cs + gid];
        out[k * cs + gid] = make_double2(x.x - v[k].re, x.y - v[k].im);
    }
}

}  // namespace

cudaError_t launch_to_fx(const double2 *in, void *w, int *ex, long long Vh, int n, const int *mask, int stride,
                         cudaStream_t st)
{
    k_to_fx<<<(unsigned)((Vh * n + 127) / 128), 128, 0, st>>>(in, static_cast<longlong2 *>(w), ex, Vh, n, mask,
                                                              stride);
    return cudaGetLastError();
}

cudaError_t launch_sub_fx(const double2 *a, const void *t, const int *ex, double2 *out, long long Vh, int n,
                          const int *mask, cudaStream_t st)
{
    k_sub_fx<<<(unsigned)((Vh * n + 127) / 128), 128, 0, st>>>(a, static_cast<const longlong2 *>(t), ex, out, Vh, n,
                                                               mask);
    return cudaGetLastError();
}

// Sites per block: as many as keep the block within kFxBlock threads, fewer
// where that leaves fewer idle threads in its last warp (12 RHS: 8 sites = 96
// threads; 48: 2).  A small lattice is cut finer, to two blocks an SM, and the
// threads left over help with the links: one RHS on 16x8^3 took 0.054 ms in 32
// full blocks (k_dslash64 0.039), 0.031 in 256.
cudaError_t launch_dslash_fx(const DslashParams &p, int epi, cudaStream_t st)
{
    if (p.nrhs < 1 || p.nrhs > kMaxRhs || !p.in_exp) return cudaErrorInvalidValue;
    FxLaunch fl{};
    const int n = p.nrhs;
    int best = 1;
    double use = 0;
    for (int k = 1; k * n <= kFxBlock; k++) {
        const int thr = (k * n + 31) / 32 * 32;
        const double u = (double)(k * n) / thr;
        if (u >= use && thr >= (use > 0 ? 64 : 0)) {
            use = u;
            best = k;
        }
    }
    constexpr long long kFill = 2 * kSms;
    const long long fine = (p.g.Vh + kFill - 1) / kFill;
    fl.sites = (int)(fine < best ? fine : best);
    // the distinct groups of the launch
    int slot[kMaxGroups];
    for (int k = 0; k < kMaxGroups; k++) slot[k] = -1;
    for (int r = 0; r < n; r++) {
        const int gr = p.grp_of[r];
        if (slot[gr] < 0) {
            slot[gr] = fl.ngrp;
            fl.grp[fl.ngrp++] = (int8_t)gr;
        }
        fl.of[r] = (int8_t)slot[gr];
    }
    int threads = (fl.sites * n + 31) / 32 * 32;
    if (fl.sites < best) {
        const int help = (fl.sites * 18 + 31) / 32 * 32;  // a clover block's entries
        threads = threads > help ? threads : help < kFxBlock ? help : kFxBlock;
    }
    const bool clover = epi == EPI_AINV || epi == EPI_XMY_AINV || epi == EPI_AINV_XMY;
    const size_t per = clover ? (size_t)fl.ngrp * 18 : kLinkSlot;  // (a clover block is the larger)
    const size_t smem = (size_t)fl.sites * (sizeof(SiteIx) + per * sizeof(int4));
    const long long blocks = (p.g.Vh + fl.sites - 1) / fl.sites;
    const unsigned grid = (unsigned)blocks;
    switch (epi) {
    case EPI_HOP: k_dslash_fx<EPI_HOP><<<grid, threads, smem, st>>>(p, fl); break;
    case EPI_AINV: k_dslash_fx<EPI_AINV><<<grid, threads, smem, st>>>(p, fl); break;
    case EPI_XMY_AINV: k_dslash_fx<EPI_XMY_AINV><<<grid, threads, smem, st>>>(p, fl); break;
    case EPI_AINV_XMY: k_dslash_fx<EPI_AINV_XMY><<<grid, threads, smem, st>>>(p, fl); break;
    case EPI_XPY: k_dslash_fx<EPI_XPY><<<grid, threads, smem, st>>>(p, fl); break;
    case EPI_XMY_G5: k_dslash_fx<EPI_XMY_G5><<<grid, threads, smem, st>>>(p, fl); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dp
