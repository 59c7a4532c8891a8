// Deterministic per-RHS grid reductions shared by the BLAS-1 kernels.
//
// A block is `lanes` sites x `units` threads, thread t = lane*units + unit;
// a unit is one RHS (FP64) or one RHS pair (FP32 paired layout, LANES = 2).
// Each thread passes per-RHS partial sums; the block sums them over its
// lanes in a fixed order, writes one partial per RHS to global scratch, and
// the last block to finish (atomic ticket) sums the block partials in a fixed
// order.  The result for an RHS never depends on the other RHS.
//
// The sums across threads run on 64-bit integers with an exponent (Sum): an
// FP64 add holds GB300's FP64 pipe for 64 cycles a warp, so the trees of a
// 384-thread block with 8 values a thread, the last block's pass over 300
// partials and the FP64 conversions around them took most of a reduction
// kernel on a small lattice (16x8^3, 12 RHS: the three of a BiCGStab iteration
// 20, 17 and 16 us, with integers 16, 13 and 10).  An integer add with
// alignment is about 10 instructions.  A block's terms have their leading bit at
// lead_for(lanes) (53 at 256 lanes, 60 at 2) and are aligned to the largest one,
// each addition rounding down by a unit at most: off by lanes 2^-lead_for(lanes)
// of the largest term.  The block's total keeps lead_for(grid) bits (50 at 1216
// blocks, 53 at 152), and the last block's sum is off by 2 grid 2^-lead_for(grid)
// of the largest total, half of that expected.  (FP64 adds: N 2^-53 of the sum.)
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "dp_internal.h"

namespace dp {

constexpr int kMaxBlock = 512;

struct Cfg {
    int lanes, block, grid;
};

inline Cfg cfg_for(long long Vh, int units, int max_grid)
{
    Cfg c;
    c.lanes = 256;
    while (c.lanes * units > kMaxBlock && c.lanes > 1) c.lanes >>= 1;
    c.block = c.lanes * units;
    long long g = (Vh + c.lanes - 1) / c.lanes;
    if (g > max_grid) g = max_grid;
    if (g < 1) g = 1;
    c.grid = (int)g;
    return c;
}

// Grid of a grid-stride reduction: one full wave (resident blocks per SM x
// SMs, from the occupancy calculator), so no partial second wave idles the
// machine at the end; never more blocks than the scratch holds.
template <typename K>
inline int one_wave(K kernel, int block, int cap)
{
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, int> cache;
    std::lock_guard<std::mutex> lk(mu);
    auto key = std::make_pair((const void *)kernel, block);
    auto it = cache.find(key);
    if (it != cache.end()) return std::min(it->second, cap);
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, block, 0) != cudaSuccess || per < 1)
        per = 1;
    cudaGetLastError();
    const int w = std::max(1, per * std::max(1, sms));
    cache[key] = w;
    return std::min(w, cap);
}

template <typename K>
inline Cfg cfg_wave(const BlasCtx &bc, K kernel, long long Vh, int units)
{
    Cfg c = cfg_for(Vh, units, bc.blocks);
    c.grid = std::min(c.grid, one_wave(kernel, c.block, bc.blocks));
    return c;
}

__device__ __forceinline__ double2 zdiv(double2 a, double2 b)
{
    const double d = b.x * b.x + b.y * b.y;
    return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 zmul(double2 a, double2 b)
{
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ bool zfinite(double2 a) { return isfinite(a.x) && isfinite(a.y); }

// ---- sums of floats or doubles on integers ------------------------------------

// m 2^e; e = kSumBad: an infinity or NaN went in
struct Sum {
    long long m;
    int e;
};
constexpr int kSumZero = -(1 << 20), kSumBad = 1 << 20;

// x with its leading bit at 2^lead
__device__ __forceinline__ Sum sum_of(float x, int lead)
{
    const int b = __float_as_int(x), be = (b >> 23) & 0xff;
    const int f = b & 0x7fffff;
    const long long m = (long long)(be ? f | 0x800000 : f) << (lead - 23);
    const int e = (be ? be : 1) - 127 - lead;
    return {b < 0 ? -m : m, be == 0xff ? kSumBad : m ? e : kSumZero};
}
__device__ __forceinline__ Sum sum_of(double x, int lead)
{
    const long long b = __double_as_longlong(x);
    const int be = (int)(b >> 52) & 0x7ff;
    long long m = b & 0xfffffffffffffll;
    if (be) m |= 1ll << 52;
    const int e = (be ? be : 1) - 1023 - lead;
    m = lead >= 52 ? m << (lead - 52) : m >> (52 - lead);
    return {b < 0 ? -m : m, be == 0x7ff ? kSumBad : m ? e : kSumZero};
}
__device__ __forceinline__ Sum add(Sum a, Sum b)
{
    const int e = max(a.e, b.e);
    return {(a.m >> min(e - a.e, 63)) + (b.m >> min(e - b.e, 63)), e};
}
// leading bit brought down to 2^lead or below (no bit is lost upwards)
__device__ __forceinline__ Sum cap(Sum a, int lead)
{
    const int top = 63 - __clzll(a.m < 0 ? ~a.m : a.m);
    const int n = top > lead ? top - lead : 0;
    return {a.m >> n, a.e >= kSumBad ? a.e : a.e + n};
}
__device__ __forceinline__ double value(Sum a)
{
    if (a.e >= kSumBad) return __longlong_as_double(0x7ff8000000000000ll);
    if (!a.m) return 0.0;
    const double d = (double)a.m;
    const int x = ((__double2hiint(d) >> 20) & 0x7ff) + a.e;
    if (x < 1 || x > 2046) return scalbn(d, a.e);  // subnormal or infinite
    return __hiloint2double(__double2hiint(d) + a.e * (1 << 20), __double2loint(d));
}

// bit for the leading term that leaves room for n additions in 63 bits
__device__ __forceinline__ int lead_for(int n) { return 61 - (32 - __clz(n - 1 > 0 ? n - 1 : 1)); }

// ---- per-RHS BiCGStab scalar recurrences, applied by the last block ----------

// alpha = rho / <rhat, v>
__device__ __forceinline__ void finish_alpha(RhsState &S, double re, double im)
{
    if (!S.active) return;
    const double2 rv = make_double2(re, im);
    if (!zfinite(rv)) {
        S.status = 3;
        S.active = 0;
    } else if (rv.x == 0.0 && rv.y == 0.0) {
        S.status = 2;
        S.active = 0;
    } else {
        S.alpha = zdiv(S.rho, rv);
        S.alpha_f = make_float2((float)S.alpha.x, (float)S.alpha.y);
    }
}

// omega = <t, s> / <t, t>
__device__ __forceinline__ void finish_omega(RhsState &S, double re, double im, double tt)
{
    if (!S.active) return;
    if (!(isfinite(re) && isfinite(im) && isfinite(tt))) {
        S.status = 3;
        S.active = 0;
        return;
    }
    S.omega = tt > 0 ? make_double2(re / tt, im / tt) : make_double2(0.0, 0.0);
}

// FP32 BiCGStab with the shadow image rhat' = Mhat^dag rhat: the s pass keeps
// <rhat, s> and <rhat', s> (= <rhat, t>) for the omega step
__device__ __forceinline__ void finish_s_dots(RhsState &S, double rs_re, double rs_im, double rt_re,
                                              double rt_im)
{
    if (!S.active) return;
    S.rs = make_double2(rs_re, rs_im);
    S.rt = make_double2(rt_re, rt_im);
    if (!(zfinite(S.rs) && zfinite(S.rt))) {
        S.status = 3;
        S.active = 0;
    }
}

// omega = <t, s>/|t|^2 from the x - A^-1 D epilogue's sums, rho' = <rhat, s> -
// omega <rhat', s>, beta = (rho'/rho)(alpha/omega); a breakdown is flagged
// for the update pass (finish_update_rr)
__device__ __forceinline__ void finish_omega_shadow(RhsState &S, double ts_re, double ts_im, double tt)
{
    if (!S.active) return;
    if (!(isfinite(ts_re) && isfinite(ts_im) && isfinite(tt))) {
        S.status = 3;
        S.active = 0;
        return;
    }
    S.omega = tt > 0 ? make_double2(ts_re / tt, ts_im / tt) : make_double2(0.0, 0.0);
    S.omega_f = make_float2((float)S.omega.x, (float)S.omega.y);
    const double2 wrt = zmul(S.omega, S.rt);
    const double2 rho_new = make_double2(S.rs.x - wrt.x, S.rs.y - wrt.y);
    if ((S.omega.x == 0.0 && S.omega.y == 0.0) || (rho_new.x == 0.0 && rho_new.y == 0.0)) {
        S.brk = 1;
        S.beta = make_double2(0.0, 0.0);
    } else {
        // one division (each is some 20 FP64 instructions of 64 cycles)
        S.beta = zdiv(zmul(rho_new, S.alpha), zmul(S.rho, S.omega));
        S.rho = rho_new;
    }
    S.beta_f = make_float2((float)S.beta.x, (float)S.beta.y);
}

// iteration count, convergence, cap, breakdown; beta = (rho'/rho)(alpha/omega)
__device__ __forceinline__ void finish_update(RhsState &S, double re, double im, double rr,
                                              int max_iter)
{
    if (!S.active) return;
    S.iters++;
    const double2 rho_new = make_double2(re, im);
    S.rr = rr;
    if (!(zfinite(rho_new) && isfinite(rr))) {
        S.status = 3;
        S.active = 0;
    } else if (S.rr <= S.tol2) {
        S.status = 1;
        S.active = 0;
    } else if (S.iters >= max_iter) {
        S.status = 4;
        S.active = 0;
    } else if ((S.omega.x == 0.0 && S.omega.y == 0.0) || (rho_new.x == 0.0 && rho_new.y == 0.0)) {
        S.status = 2;
        S.active = 0;
    } else {
        S.beta = zmul(zdiv(rho_new, S.rho), zdiv(S.alpha, S.omega));
        S.rho = rho_new;
    }
}

// iteration count, convergence, cap, and a breakdown flagged by
// finish_omega_shadow
__device__ __forceinline__ void finish_update_rr(RhsState &S, double rr, int max_iter)
{
    if (!S.active) return;
    S.iters++;
    S.rr = rr;
    if (!isfinite(rr)) {
        S.status = 3;
        S.active = 0;
    } else if (S.rr <= S.tol2) {
        S.status = 1;
        S.active = 0;
    } else if (S.iters >= max_iter) {
        S.status = 4;
        S.active = 0;
    } else if (S.brk) {
        S.status = 2;
        S.active = 0;
    }
}

// start of an inner solve: rho = |r|^2, tol2 (tol^2 on entry) *= |r|^2
__device__ __forceinline__ void finish_init(RhsState &S, double bb)
{
    if (!S.active) return;
    S.rr = bb;
    S.bb = bb;
    S.tol2 = S.tol2 * bb;
    S.rho = make_double2(bb, 0.0);
    S.alpha = make_double2(1.0, 0.0);
    S.omega = make_double2(1.0, 0.0);
    S.beta = make_double2(0.0, 0.0);
    S.alpha_f = S.omega_f = make_float2(1.f, 0.f);
    S.beta_f = make_float2(0.f, 0.f);
    S.iters = 0;
    S.brk = 0;
    if (!isfinite(bb)) {
        S.status = 3;
        S.active = 0;
    } else if (bb <= S.tol2) {
        S.status = 1;
        S.active = 0;
    }
}

// ---- per-RHS CGNE scalar recurrences (real, in the .x parts) ----------------

// rho' = |Mhat^dag r|^2; beta = rho'/rho (first iteration: 0)
__device__ __forceinline__ void finish_cg_gamma(RhsState &S, double zz, int first)
{
    if (!S.active) return;
    if (!isfinite(zz)) {
        S.status = 3;
        S.active = 0;
    } else if (zz == 0.0) {  // Mhat^dag r = 0 with r != 0: singular operator
        S.status = 2;
        S.active = 0;
    } else {
        S.beta = make_double2(first ? 0.0 : zz / S.rho.x, 0.0);
        S.beta_f = make_float2((float)S.beta.x, 0.f);
        S.rho = make_double2(zz, 0.0);
    }
}

// alpha = rho / |Mhat p|^2
__device__ __forceinline__ void finish_cg_alpha(RhsState &S, double ww)
{
    if (!S.active) return;
    if (!isfinite(ww)) {
        S.status = 3;
        S.active = 0;
    } else if (ww == 0.0) {
        S.status = 2;
        S.active = 0;
    } else {
        S.alpha = make_double2(S.rho.x / ww, 0.0);
        S.alpha_f = make_float2((float)S.alpha.x, 0.f);
    }
}

// iteration count and the stop rules on |r|^2 (the Mhat residual)
__device__ __forceinline__ void finish_cg_update(RhsState &S, double rr, int max_iter)
{
    if (!S.active) return;
    S.iters++;
    S.rr = rr;
    if (!isfinite(rr)) {
        S.status = 3;
        S.active = 0;
    } else if (rr <= S.tol2) {
        S.status = 1;
        S.active = 0;
    } else if (S.iters >= max_iter) {
        S.status = 4;
        S.active = 0;
    }
}

// Block + grid reduction of NV values per RHS for LANES RHS per thread
// (v[L*NV + k] belongs to RHS LANES*unit + L; floats or doubles).  Returns
// true in the threads of the last block; its thread r (r < the RHS count) then
// has the totals of RHS r in `tot`, so the scalar recurrences of all RHS run
// side by side in one or two warps.
//
// In both passes thread g*n + j sums value j of the n = W*units values over
// every G-th lane (or block) from g, and thread j then the G results: the
// W*lanes additions spread over all threads, two barriers a pass.  A tree over
// the lanes leaves its threads W additions a level, six levels at 12 RHS, and
// six barriers: the three reductions of an iteration at 16x8^3, 12 RHS, took
// 16, 13 and 10 us with it and take 11, 7 and 7.
// n <= the block: cfg_for leaves lanes >= W for every RHS count.

struct __align__(16) Partial {
    long long m;
    int e, pad;
};
static_assert(sizeof(Partial) == 16, "two doubles of the scratch each");

// the G sums of each value, left by thread g*n + j at [g*n + j]: thread j's total
struct GroupSums {
    long long m[kMaxBlock];
    int e[kMaxBlock];
    __device__ __forceinline__ void put(int t, Sum s)
    {
        m[t] = s.m;
        e[t] = s.e;
    }
    __device__ __forceinline__ Sum total(int j, int n, int groups) const
    {
        Sum s{m[j], e[j]};
        for (int g = 1; g < groups; g++) s = add(s, Sum{m[g * n + j], e[g * n + j]});
        return s;
    }
};

template <int NV, int LANES, typename T>
__device__ __forceinline__ bool reduce_last(const T (&in)[LANES * NV], const Cfg c, double *partials,
                                            unsigned int *counter, int units, double (&tot)[NV])
{
    static_assert(2 * NV <= kRedWidth, "per-RHS partials hold kRedWidth doubles");
    constexpr int W = LANES * NV;
    __shared__ T raw[W * (kMaxBlock + kMaxRhs / LANES)];
    __shared__ GroupSums gs;
    __shared__ double val[W * (kMaxRhs / LANES)];
    __shared__ bool last;
    const int t = threadIdx.x;
    const int n = W * units, grp = t / n, j = t - grp * n, groups = c.block / n;
    Partial *part = reinterpret_cast<Partial *>(partials);
    constexpr int kStride = kMaxRhs * kRedWidth / 2;  // per block
    // value j = k*units + u of lane l at j + l*units + k*block: no bank conflicts
    const int ld = c.block + units;
#pragma unroll
    for (int k = 0; k < W; k++) raw[k * ld + t] = in[k];
    __syncthreads();
    if (grp < groups) {
        const int lead = lead_for(c.lanes), k = j / units;
        const T *mine = raw + j + k * c.block;
        Sum s{0, kSumZero};
#pragma unroll 4
        for (int l = grp; l < c.lanes; l += groups) s = add(s, sum_of(mine[l * units], lead));
        gs.put(t, s);
    }
    __syncthreads();
    if (t < n) {
        const Sum s = cap(gs.total(t, n, groups), lead_for((int)gridDim.x));
        part[(long long)blockIdx.x * kStride + t] = Partial{s.m, s.e, 0};
        __threadfence();
    }
    __syncthreads();
    if (t == 0) {
        __threadfence();
        last = (atomicAdd(counter, 1u) == (unsigned)(gridDim.x - 1));
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    if (grp < groups) {
        Sum s{0, kSumZero};
        // eight loads ahead, also at the end (each round waits for L2, about 1 us)
        constexpr int kAhead = 8;
        for (int b0 = grp; b0 < (int)gridDim.x; b0 += kAhead * groups) {
            longlong2 w[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; i++) {
                const int b = b0 + i * groups;
                w[i] = make_longlong2(0, kSumZero);
                if (b < (int)gridDim.x)
                    w[i] = __ldcg(reinterpret_cast<const longlong2 *>(part + (long long)b * kStride + j));
            }
#pragma unroll
            for (int i = 0; i < kAhead; i++) s = add(s, Sum{w[i].x, (int)w[i].y});
        }
        gs.put(t, s);
    }
    if (t == 0) *counter = 0u;
    __syncthreads();
    if (t < n) val[t] = value(gs.total(t, n, groups));
    __syncthreads();
    if (t < LANES * units)
#pragma unroll
        for (int k = 0; k < NV; k++) tot[k] = val[(t % LANES * NV + k) * units + t / LANES];
    return true;
}

// in the last block, after thread r has finished RHS r: how many still iterate
__device__ __forceinline__ void count_active(const RhsState *st, int nrhs, int *n_active)
{
    const int t = threadIdx.x;
    const int k = __syncthreads_count(t < nrhs && st[t].active != 0);
    if (t == 0) *n_active = k;
}

}  // namespace dp
