// Sums over the sites of a time slice of |psi|^2 / alpha_B^2, per group: the
// common part of the contraction (field.cu) and of the per-slice norms
// (slices.cu).
//
// A block takes a share of one slice for a contiguous range of RHS; thread t
// = lane * nr + (RHS - r0) keeps its RHS and walks the sites.  What bounds
// it is meant to be the read of the spinors, so the FP64 pipe (64 cycles a
// warp instruction) is kept out: |psi|^2 is formed on integers (norm2_int),
// and 1/alpha_B^2 is a product of per-coordinate inverse squares that the
// block makes once, the time direction's applied to the block's sum.  FP64
// instructions per spinor: 4, where scaling each component by 1/alpha_B and
// squaring took 48 and a division.
#pragma once

#include "cplx.cuh"
#include "dp_internal.h"
#include "reduce.cuh"

namespace dp {

// sum of the squares of 24 doubles, to be multiplied by the weight w >= 0 and
// added up over the slice.  With the leading bit of the largest at bit 59, |v|
// = hi 2^32 + lo 2: hi hi and hi lo summed in 64 bits, lo lo to 2^34 (all of
// them below 2^-57 of the sum).  false (general arithmetic, which scales each
// component by 1/alpha first): an infinity or a NaN, a largest component or a
// weight outside 2^+-400 (squares stay below 2^805), or a product outside
// 2^+-900: with 1/alpha_t^2 still to come it could leave the normal range
// although the scaled sum does not (alpha_t = 2^520 and 2^-50 in each space
// direction: 2^740 times 2^300).  2^900 leaves room for 2^120 terms.
__device__ __forceinline__ bool norm2_int(const double2 (&v)[12], double w, double &s)
{
    unsigned mx = 0;
#pragma unroll
    for (int k = 0; k < 12; k++)
        mx = max(mx, max((unsigned)__double2hiint(v[k].x) & 0x7fffffffu, (unsigned)__double2hiint(v[k].y) & 0x7fffffffu));
    const int em = (int)(mx >> 20), ew = __double2hiint(w) >> 20;
    if (em < 623 || em > 1423 || ew < 623 || ew > 1423) return false;
    if (abs(2 * em + ew - 3 * 1023) > 900) return false;
    unsigned long long hh = 0, hl = 0;
    auto sq = [&](double x) {
        const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
        const unsigned m = (h & 0xfffffu) | 0x100000u;
        unsigned long long w = ((unsigned long long)__funnelshift_l(l, m, 7) << 32) | (l << 7);
        const int d = em - (int)((h >> 20) & 0x7ffu);
        asm("shr.u64 %0, %0, %1;" : "+l"(w) : "r"(d));  // (amounts above 63 give 0: zeros, subnormals)
        const unsigned hi = (unsigned)(w >> 32), lo = (unsigned)w >> 1;
        hh += (unsigned long long)hi * hi;
        hl += (unsigned long long)hi * lo + __umulhi(lo, lo);
    };
#pragma unroll
    for (int k = 0; k < 12; k++) {
        sq(v[k].x);
        sq(v[k].y);
    }
    const double d = (double)((hh << 3) + (hl >> 27));
    s = __hiloint2double(__double2hiint(d) + (2 * (em - 1023 - 59) + 61) * (1 << 20), __double2loint(d));
    return true;
}

// the block's share of a slice
struct SliceShare {
    int j0, j1, lanes, lane, r;  // half-sites of the slice, this thread's lane and RHS
    bool on;                     // the thread takes part
};

// lanes of a block for nr RHS: a power of two, up to kSliceThreads threads
constexpr int kSliceThreads = 256;
inline int slice_lanes(int nr)
{
    int l = 1;
    while (2 * l * nr <= kSliceThreads) l *= 2;
    return l;
}
// shared memory for the inverse squares of ng groups
inline size_t slice_smem(const Geom &g, int ng) { return (size_t)ng * 3 * g.Lmax * sizeof(double); }

__device__ __forceinline__ SliceShare slice_share(const Geom &g, int r0, int nr)
{
    const int P = gridDim.x, p = blockIdx.x;
    const int Vs = (int)(g.Vh / g.T), chunk = (Vs + P - 1) / P;
    SliceShare h;
    h.j0 = min(Vs, p * chunk);
    h.j1 = min(Vs, h.j0 + chunk);
    h.lanes = blockDim.x / nr;
    h.lane = threadIdx.x / nr;
    h.r = r0 + threadIdx.x % nr;
    h.on = h.lane < h.lanes;
    return h;
}

// iw[(m*3 + {0: x, 1: y, 2: z})*Lmax + coordinate] = 1/alpha^2 of group m; 0
// (a weight that norm2_int refuses) where alpha is outside 2^+-170, so that no
// product of three, nor of two, rounds among the subnormals
__device__ __forceinline__ void slice_weights(double *iw, const Geom &g, const double *alpha, int ng)
{
    for (int k = threadIdx.x; k < ng * 3 * g.Lmax; k += blockDim.x) {
        const int m = k / (3 * g.Lmax), rest = k - m * 3 * g.Lmax;
        const double a = alpha[(long long)m * 4 * g.Lmax + g.Lmax + rest];
        const double w = 1.0 / (a * a);
        iw[k] = w > 0x1p-340 && w < 0x1p+340 ? w : 0.0;
    }
    __syncthreads();
}

// totals per group over the block: each thread's NV sums are added over the
// lanes, then over the RHS of a group (grp[r], shared memory) in order; the
// result is in thread m < ng
template <int NV>
__device__ __forceinline__ void slice_totals(const double (&in)[NV], int lanes, int nr, int r0, const int *grp, int ng,
                                             double (&tot)[NV])
{
    __shared__ long long shm[kSliceThreads * NV];
    __shared__ int she[kSliceThreads * NV];
    const int t = threadIdx.x, lane = t / nr;
    const int lead = lead_for(lanes);
    Sum v[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = sum_of(in[k], lead);
    for (int w = lanes / 2; w > 0; w >>= 1) {
        if (lane >= w && lane < 2 * w)
#pragma unroll
            for (int k = 0; k < NV; k++) {
                shm[k * kSliceThreads + t] = v[k].m;
                she[k * kSliceThreads + t] = v[k].e;
            }
        __syncthreads();
        if (lane < w)
#pragma unroll
            for (int k = 0; k < NV; k++)
                v[k] = add(v[k], Sum{shm[k * kSliceThreads + t + w * nr], she[k * kSliceThreads + t + w * nr]});
    }
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; k++) {
            const Sum c = cap(v[k], 57);  // room for the 12 RHS of a group
            shm[k * kSliceThreads + t] = c.m;
            she[k * kSliceThreads + t] = c.e;
        }
    __syncthreads();
    if (t < ng)
#pragma unroll
        for (int k = 0; k < NV; k++) {
            Sum s = {0, kSumZero};
            for (int q = 0; q < nr; q++)
                if (grp[r0 + q] == t) s = add(s, Sum{shm[k * kSliceThreads + q], she[k * kSliceThreads + q]});
            tot[k] = value(s);
        }
}

// (x / a) / a, 0 for x = 0 (a group without RHS has no profile)
__device__ __forceinline__ double over_square(double x, double a) { return x != 0.0 ? (x / a) / a : 0.0; }

}  // namespace dp
