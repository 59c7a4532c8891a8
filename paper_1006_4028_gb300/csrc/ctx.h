// Host-side state of a dpre context: device memory, resident gauge fields
// with their clover terms and clover inverses, reduction scratch, the launch
// tuner, per-kernel timing and the request scheduler.
#pragma once

#include <atomic>
#include <condition_variable>
#include <cstdint>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "../../include/dpre.h"
#include "dp_internal.h"

namespace dp {

void set_error(const char *fmt, ...);

struct Ctx;

// clover inverse for one mass; device memory is returned to the context when
// the last holder (field cache or running batch) lets go
struct CloverInv {
    Ctx *owner = nullptr;
    double M = 0;
    double2 *inv64[2] = {nullptr, nullptr};
    float4 *inv32[2] = {nullptr, nullptr};
    float4 *invdf[2] = {nullptr, nullptr};  // double-float copy, on first use
    ~CloverInv();
};

struct Field {
    Geom g;
    int bc_t;
    // FP64 products in integer arithmetic (dslash_fx.cu): every link's rows
    // and columns have norm 1 (to 1e-3), and at most one link of 500 has an entry below
    // 2^-12
    bool fx = false;
    double2 *l64[2] = {nullptr, nullptr};
    float2 *l32f[2] = {nullptr, nullptr};
    float4 *l32c[2] = {nullptr, nullptr};
    void *l16[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};  // [FP16, BF16][parity], lazily
    float4 *ldf[2] = {nullptr, nullptr};  // double-float links, lazily
    double2 *clov[2] = {nullptr, nullptr};  // clover term, FP64 (no mass)
    float4 *clov32[2] = {nullptr, nullptr}; // clover term, FP32 copy
    bool has_clover = false;
    double csw = 0;
    std::vector<std::shared_ptr<CloverInv>> invs;  // per mass, least recently used first
    std::mutex inv_mu;
    std::atomic<int> users{0};    // requests in flight on this field
};

// one point-source group = 12 RHS sharing (mass, profile, source)
struct Group {
    double M;
    dp_profile prof;
    std::vector<double> table[4];  // copies of TABLE profiles
    int src[4];
};

struct TimingRec {
    std::string name;
    cudaEvent_t a, b;
};

struct Stat {
    long launches = 0;
    double ms = 0;
};

struct TuneKey {
    long long Vh;
    int prec, link_fmt, nrhs;
    bool operator<(const TuneKey &o) const
    {
        if (Vh != o.Vh) return Vh < o.Vh;
        if (prec != o.prec) return prec < o.prec;
        if (link_fmt != o.link_fmt) return link_fmt < o.link_fmt;
        return nrhs < o.nrhs;
    }
};

struct Scheduler;
struct SchedDeleter {
    void operator()(Scheduler *s) const;  // defined with the scheduler (serve.cu)
};

struct Ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    dp_alloc_hooks hooks{};
    bool has_hooks = false;
    cudaMemPool_t pool = nullptr;  // without hooks: stream-ordered pool that keeps freed memory

    std::mutex mu;  // fields, allocations, tuner
    std::map<uint64_t, std::shared_ptr<Field>> fields;
    uint64_t next_field = 1;
    std::map<void *, size_t> allocs;
    size_t bytes = 0;

    BlasCtx bc{};
    int *h_nactive = nullptr;  // pinned

    bool timing = false;
    std::vector<TimingRec> pending;
    std::vector<cudaEvent_t> event_pool;
    std::map<std::string, Stat> stats;
    std::atomic<long> launches{0};

    std::map<TuneKey, Shape> tuned;

    std::unique_ptr<Scheduler, SchedDeleter> sched;

    void *alloc(size_t n);
    void release(void *p);
    cudaEvent_t get_event();
    // record a timed launch region: call before(name) / after(); only work on
    // the context stream is timed (st: the launching stream, NULL = it)
    void time_begin(const char *name, cudaEvent_t *a, cudaStream_t st = nullptr);
    void time_end(const char *name, cudaEvent_t a, cudaStream_t st = nullptr);
    void collect_timing();
    // dslash launch shape for the Schur launches: tuned, else a default
    Shape launch_shape(long long Vh, int prec, int link_fmt, int nrhs);
};

std::shared_ptr<Field> find_field(Ctx *c, dp_field f);
// device links of one parity in a storage format (16-bit ones built on first use)
dp_status field_links(Ctx *c, Field &f, int link_fmt, int parity, const void **out);
// link format of the inner solver for a precision and compress12 choice
int inner_link_format(int prec, int compress12);
// clover inverse of (4+M) + clover for both parities, cached per mass
dp_status get_clover_inv(Ctx *c, Field &f, double M, std::shared_ptr<CloverInv> *out);
// its double-float copy (made on first use)
dp_status clover_inv_df(Ctx *c, Field &f, CloverInv &ci);
// FP64 alpha_B tables [4][Lmax] and hop tables [4][2][Lmax] (with the -1/2)
dp_status profile_tables(const dp_profile &p, const Geom &g, int bc_t, const int src[4],
                         double *alpha, double *hop);

struct SolveResult {
    int iters_inner = 0, iters_outer = 0;
    double true_rel_residue = 0;
    int status = 0;
    double slice_residue = 0;  // max over time slices of the restored per-slice residual
    int refine_rounds = 0;     // outer rounds spent on per-slice refinement
};

// per-slice target of a solve at residue r: opts_tol > 0 as given, < 0 off,
// 0 the default: kSliceFactor * r, but never below kSliceFloor (a restored
// per-slice residual of 1e-8 already holds C_PP(y0) far inside 1e-6 on every
// workload tested; tighter per-slice work buys the correlator nothing)
constexpr double kSliceFactor = 10.0;
constexpr double kSliceFloor = 1e-8;
inline double slice_target(double opts_tol, double r)
{
    if (opts_tol > 0) return opts_tol;
    if (opts_tol < 0) return 0.0;
    const double t = kSliceFactor * r;
    return t > kSliceFloor ? t : kSliceFloor;
}

// the method for a set of point-source groups on one field (solver.cu)
// cap_dev (optional, device [n_groups][T]): also C_AP(y0)
dp_status solve_groups(Ctx *c, std::shared_ptr<Field> f, const std::vector<Group> &groups, double r_target,
                       const dp_solve_opts &opts, double *cpp_dev, double *prop_host,
                       std::vector<SolveResult> &res, double *cap_dev = nullptr,
                       double *hl_dev = nullptr);

dp_status check_opts(const dp_solve_opts *in, dp_solve_opts *out);

// forget the looked-up device address of the allocation-free entry point's
// scratch array on `device` (field.cu)
void noalloc_forget_address(int device);

}  // namespace dp

struct dp_ctx {
    dp::Ctx c;
};
