"""Performance cases of the library: what its users have it do, at the sizes
of its workloads.

A case is a dict of plain values.  Its ``kind`` says which entry points a pass
calls:

* ``solve``     one point-source solve (one or several masses) on a resident
                field: the call the library is for;
* ``config``    the per-configuration workflow of an ensemble: load the gauge
                field, build the clover term, solve once, free the field;
* ``serve``     a burst of requests to the running scheduler on two resident
                fields, waited for in order;
* ``schur``     the Schur operator and its adjoint on device spinors (the
                building block a caller's own Krylov solver uses);
* ``apply``     the full operator on host spinors;
* ``contract``  restore and contract of device propagators.

``dims`` are T, Lx, Ly, Lz; links are U = exp(i eps H) with Gaussian H (the
recipe of ``lattice_inputs``, drawn on the GPU).  ``tuned``: whether the
program called dp_autotune for the volume beforehand.  Sources sit at a site
drawn from the seed.
"""
import math

import numpy as np
import torch

import paper_1006_4028_gb300 as dp

MASSES4 = "0.01,0.1,0.5,0.8"


def _solve(name, dims, eps, csw, M, profile, r, **more):
    c = {"name": name, "kind": "solve", "dims": "%d,%d,%d,%d" % tuple(dims), "eps": eps, "csw": csw, "M": M,
         "profile": profile, "r": r, "prec": "mixed_fp32", "solver": "bicgstab", "batched": True, "graph": True,
         "tuned": True, "bc_t": -1, "out": "cpp"}
    c.update(more)
    return c


def listed():
    return [
        # the benchmark workload: heavy quark, residue 1e-11, 12 right-hand sides
        _solve("heavy_48x24", (48, 24, 24, 24), 0.3, 1.7, "0.5", "cosh_t:0.4", 1e-11),
        # the largest workload: light quark with FP16 links, per-slice refinement
        _solve("light_64x32_fp16", (64, 32, 32, 32), 0.5, 1.9, "0.005", "cosh_4d:0.2", 1e-10, prec="mixed_fp16"),
        # four masses from one source in one 48-column batch, launch shapes as the library picks them
        _solve("multimass_32x16", (32, 16, 16, 16), 0.4, 1.7, MASSES4, "auto", 1e-10, tuned=False),
        # the smallest solve of the workloads: launches and latency count
        _solve("small_16x8", (16, 8, 8, 8), 0.3, 1.7, "0.5", "exp_t:0.4", 1e-11, tuned=False),
        # the FP64 reference solve of the precision comparisons
        _solve("fp64_32x16", (32, 16, 16, 16), 0.3, 1.7, "0.8", "cosh_t:0.4", 1e-11, prec="fp64", graph=False),
        # the paper's own solver (SAP+GCR)
        _solve("sap_gcr_32x16", (32, 16, 16, 16), 0.5, 1.9, "0.05", "cosh_4d:0.2", 1e-10, solver="sap_gcr",
               tuned=False),
        # a propagator handed back to the host, ragged extents, Dirichlet time boundary
        _solve("propagator_20x12x10x14", (20, 12, 10, 14), 0.35, 1.7, "0.3", "exp_t:0.3", 1e-11, bc_t=0, out="prop",
               tuned=False),
        # a new gauge configuration of an ensemble: load, clover term, one solve
        dict(_solve("config_24x16x12x12", (24, 16, 12, 12), 0.4, 1.7, "0.2", "cosh_t:0.4", 1e-10, tuned=False),
             kind="config"),
        # a burst of the serving mix: two volumes, masses and sources at random
        {"name": "serve_16x8_32x16", "kind": "serve", "dims": "16,8,8,8", "dims2": "32,16,16,16", "eps": 0.3,
         "eps2": 0.4, "csw": 1.7, "requests": 8, "r": 1e-10},
        # the operators alone: benchmark size in FP32 ...
        {"name": "schur_fp32_48x24", "kind": "schur", "dims": "48,24,24,24", "eps": 0.3, "csw": 1.7, "M": "0.5",
         "profile": "cosh_t:0.4", "prec": "mixed_fp32", "compress12": 1, "nrhs": 12, "bc_t": -1},
        # ... and a few right-hand sides on a small ragged lattice in FP64, where the call itself counts
        {"name": "schur_fp64_8x4x6x4", "kind": "schur", "dims": "8,4,6,4", "eps": 0.5, "csw": 1.7, "M": "0.15",
         "profile": "cosh_4d:0.3", "prec": "fp64", "compress12": 1, "nrhs": 5, "bc_t": -1},
        # several propagators restored and contracted at once
        {"name": "contract_32x16_g3", "kind": "contract", "dims": "32,16,16,16", "groups": 3},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, vmin, vmax):
    """Even extents with a volume spread over its logarithm, T the longest."""
    v = _log(rng, vmin, vmax)
    ls = max(4.0, (v / 2.0) ** 0.25)
    L = [max(4, min(32, 2 * round(ls * rng.uniform(0.75, 1.3) / 2))) for _ in range(3)]
    T = max(6, min(64, 2 * round(v / (L[0] * L[1] * L[2]) / 2)))
    while T * L[0] * L[1] * L[2] > vmax and T > 6:
        T -= 2
    return (T, L[0], L[1], L[2])


def draw(rng):
    """One more case: mostly solves over the volumes, masses, profiles and
    precisions of the workloads, some operators and contractions."""
    def heavy_light():
        M = round(rng.uniform(0.3, 0.8) if rng.random() < 0.6 else _log(rng, 0.02, 0.3), 3)
        return M, ("cosh_t:0.4" if M >= 0.3 else "cosh_4d:0.2")

    eps = round(rng.uniform(0.25, 0.5), 3)
    csw = rng.choice([1.7, 1.9])
    pick = rng.random()
    if pick < 0.5:
        M, prof = heavy_light()
        prec = rng.choice(["mixed_fp32", "mixed_fp32", "mixed_fp16", "mixed_bf16", "fp64"])
        dims = _dims(rng, 4096, 262144 if prec == "fp64" else 663552)
        more = {"prec": prec, "tuned": rng.random() < 0.5, "out": rng.choice(["cpp", "corr"])}
        if prec == "fp64":
            more["graph"] = False
        if prec == "mixed_fp32" and rng.random() < 0.5:
            more["solver"] = rng.choice(["cgne", "sap_gcr"])
            more["compress12"] = rng.choice([0, 1])
        if more.get("solver") is None and rng.random() < 0.3:
            V = dims[0] * dims[1] * dims[2] * dims[3]
            if V <= 200000:
                Ms = MASSES4 if rng.random() < 0.5 else "%g,%g" % (M, M + 0.2)
                c = _solve("", dims, eps, csw, Ms, "auto", 1e-10, prec=prec, tuned=False, graph=prec != "fp64")
                return {k: v for k, v in c.items() if k != "name"}
        c = _solve("", dims, eps, csw, "%g" % M, prof, rng.choice([1e-10, 1e-11]), **more)
        return {k: v for k, v in c.items() if k != "name"}
    if pick < 0.6:
        M, prof = heavy_light()
        c = dict(_solve("", _dims(rng, 4096, 131072), eps, csw, "%g" % M, prof, 1e-10, tuned=False), kind="config")
        return {k: v for k, v in c.items() if k != "name"}
    if pick < 0.85:
        prec = rng.choice(["mixed_fp32", "mixed_fp32", "mixed_fp16", "fp64"])
        n = rng.choice([2, 4, 6, 12, 24, 48]) if prec != "fp64" else rng.choice([1, 3, 5, 12, 24])
        d = _dims(rng, 512, 663552 * 12 // max(n, 12))
        return {"kind": "schur", "dims": "%d,%d,%d,%d" % d, "eps": eps, "csw": csw, "M": "%g" % heavy_light()[0],
                "profile": rng.choice(["none:0", "cosh_t:0.4", "cosh_4d:0.2", "exp_t:0.2"]), "prec": prec,
                "compress12": rng.choice([0, 1]), "nrhs": n, "bc_t": rng.choice([-1, 1, 0])}
    if pick < 0.92:
        n = rng.choice([1, 2, 5])
        return {"kind": "apply", "dims": "%d,%d,%d,%d" % _dims(rng, 2048, 131072), "eps": eps, "csw": csw,
                "M": "0.1", "profile": "cosh_4d:0.2", "prec": rng.choice(["fp64", "mixed_fp32"]), "nrhs": n,
                "bc_t": -1}
    g = rng.choice([1, 2, 3, 4])
    return {"kind": "contract", "dims": "%d,%d,%d,%d" % _dims(rng, 2048, 663552 // g), "groups": g}


# ---- inputs -------------------------------------------------------------------

_CTX = {}


def _ctx(tuned):
    """One library context for the programs that tune their launches, one for
    those that do not; a program keeps it for as long as it runs."""
    if tuned not in _CTX:
        _CTX[tuned] = (dp.dp_create(0), set())
    return _CTX[tuned]


class _Field:
    def __init__(self, ctx, links, dims, bc_t, csw):
        self.ctx, self.dims = ctx, dims
        self.id = dp.dp_field_load(ctx, links, dims, bc_t)
        dp.dp_field_set_csw(ctx, self.id, csw)

    def __del__(self):
        dp.dp_field_free(self.ctx, self.id)


class _Serving:
    """A context of its own with its scheduler running."""

    def __init__(self):
        self.ctx = dp.dp_create(0)
        self.fields = []

    def __del__(self):
        dp.dp_serve_stop(self.ctx)
        self.fields.clear()
        dp.dp_destroy(self.ctx)


def _ints(text):
    return tuple(int(v) for v in text.split(","))


def _gell_mann():
    lam = np.zeros((8, 3, 3), np.complex128)
    lam[0][0, 1] = lam[0][1, 0] = 1
    lam[1][0, 1], lam[1][1, 0] = -1j, 1j
    lam[2][0, 0], lam[2][1, 1] = 1, -1
    lam[3][0, 2] = lam[3][2, 0] = 1
    lam[4][0, 2], lam[4][2, 0] = -1j, 1j
    lam[5][1, 2] = lam[5][2, 1] = 1
    lam[6][1, 2], lam[6][2, 1] = -1j, 1j
    lam[7] = np.diag([1, 1, -2]) / np.sqrt(3)
    return torch.from_numpy(lam).cuda()


def _links(dims, eps, seed):
    """SU(3) links U = exp(i eps H), H = sum c_a lambda_a / 2, c_a ~ N(0, 1):
    complex128 (T, Lz, Ly, Lx, 4, 3, 3) on the GPU."""
    T, Lx, Ly, Lz = dims
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    lam = (_gell_mann() / 2).reshape(8, 9)
    out = torch.empty((T, Lz, Ly, Lx, 4, 3, 3), dtype=torch.complex128, device="cuda")
    one = torch.eye(3, dtype=torch.complex128, device="cuda")

    def mul(A, B):  # 3x3 products (as broadcasts: batched library calls are slow at this size)
        return (A[:, :, :, None] * B[:, None]).sum(2)
    for t in range(T):
        c = torch.randn((Lz * Ly * Lx * 4, 8), dtype=torch.float64, device="cuda", generator=g)
        X = (c[:, :, None] * lam).sum(1).reshape(-1, 3, 3) * (1j * eps / 4)
        E = one + X / 10
        for k in range(9, 0, -1):  # Taylor series of exp(X), |X| below 1
            E = one + mul(X, E) / k
        for _ in range(2):
            E = mul(E, E)
        r0 = E[:, 0] / torch.linalg.vector_norm(E[:, 0], dim=-1, keepdim=True)
        r1 = E[:, 1] - (r0.conj() * E[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
        r2 = torch.linalg.cross(r0, r1).conj()
        out[t] = torch.stack([r0, r1, r2], -2).reshape(Lz, Ly, Lx, 4, 3, 3)
    return out


def _host_links(dims, eps, seed):
    return _links(dims, eps, seed).cpu().numpy()


def _source(dims, seed):
    rng = np.random.default_rng(seed + 77)
    return tuple(int(rng.integers(0, d)) for d in dims)


def _masses(case):
    return [float(m) for m in case["M"].split(",")]


def _profiles(case):
    """Per mass; "auto" is the heavy or light profile by the mass."""
    if case["profile"] == "auto":
        return [("cosh_t", 0.4) if m >= 0.3 else ("cosh_4d", 0.2) for m in _masses(case)]
    kind, a0 = case["profile"].split(":")
    return [(kind, float(a0))] * len(_masses(case))


def _opts(case):
    return {"prec": case["prec"], "solver": case["solver"], "batched": int(case["batched"]),
            "use_graph": int(case["graph"]), "compress12": case.get("compress12", 1)}


def _spinor(dims, nrhs, prec, seed):
    """Gaussian spinors of one parity in the library's device layout."""
    Vh = dims[0] * dims[1] * dims[2] * dims[3] // 2
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
    if prec == "fp64":
        return torch.randn((12, Vh, nrhs, 2), dtype=torch.float64, device="cuda", generator=g)
    return torch.randn((12, Vh, nrhs // 2, 4), dtype=torch.float32, device="cuda", generator=g)


def _requests(case, seed):
    rng = np.random.default_rng(seed + 99)
    got = []
    for k in range(case["requests"]):
        dims = _ints(case["dims"] if k % 2 == 0 else case["dims2"])
        M = float(rng.uniform(0.01, 0.8))
        prof = ("cosh_t", 0.4) if M >= 0.3 else ("cosh_4d", 0.2)
        got.append((k % 2, dims, M, prof, tuple(int(rng.integers(0, d)) for d in dims)))
    return got


def _groups(case, seed):
    dims = _ints(case["dims"])
    kinds = [("cosh_t", 0.4), ("cosh_4d", 0.2), ("exp_t", 0.3), ("none", 0.0)][: case["groups"]]
    return kinds, [_source(dims, seed + 1000 * k) for k in range(case["groups"])]


def prepare(case, seed):
    dims = _ints(case["dims"])
    s = {"case": case, "dims": dims}
    if case["kind"] == "serve":
        sv = _Serving()
        for k, (d, e) in enumerate((("dims", "eps"), ("dims2", "eps2"))):
            dd = _ints(case[d])
            f = dp.dp_field_load(sv.ctx, _host_links(dd, case[e], 2 * seed + k), dd, -1)
            dp.dp_field_set_csw(sv.ctx, f, case["csw"])
            sv.fields.append(f)
        dp.dp_serve_start(sv.ctx)
        s["serving"], s["requests"] = sv, _requests(case, seed)
        return s
    ctx, seen = _ctx(bool(case.get("tuned", False)))
    s["ctx"] = ctx
    if case["kind"] == "contract":
        s["profiles"], s["src"] = _groups(case, seed)
        # contracting needs the field's geometry alone
        s["field"] = _Field(ctx, _host_links(dims, 0.3, seed), dims, -1, 1.0)
        s["x"] = [_spinor(dims, 12 * case["groups"], "fp64", seed + p) for p in (0, 1)]
        s["cpp"] = torch.zeros((case["groups"], dims[0]), dtype=torch.float64, device="cuda")
        return s
    links = _host_links(dims, case["eps"], seed)
    s["src"] = _source(dims, seed)
    if case["kind"] == "config":
        s["links"] = links
        return s
    s["field"] = f = _Field(ctx, links, dims, case["bc_t"], case["csw"])
    if case["kind"] == "schur":
        s["in"] = _spinor(dims, case["nrhs"], case["prec"], seed)
        s["out"] = [torch.zeros_like(s["in"]) for _ in (0, 1)]
    elif case["kind"] == "apply":
        rng = np.random.default_rng(seed + 5)
        shape = (case["nrhs"], dims[0], dims[3], dims[2], dims[1], 4, 3)
        s["psi"] = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    elif case["tuned"]:  # a program tunes its launches once per volume
        n = 12 * len(_masses(case))
        key = (dims, case["prec"], case.get("compress12", 1), n)
        if key not in seen:
            dp.dp_autotune(ctx, f.id, case["prec"], case.get("compress12", 1), n)
            seen.add(key)
    return s


# ---- one pass ---------------------------------------------------------------------

def _one_solve(case, ctx, f, dims, src):
    Ms, profs, T, o = _masses(case), _profiles(case), dims[0], _opts(case)
    if len(Ms) > 1:
        return [dp.dp_solve_point_multi(ctx, f, Ms, profs, src, case["r"], o, T=T, allow=())[0]]
    if case["out"] == "corr":
        return list(dp.dp_solve_point_corr(ctx, f, Ms[0], profs[0], src, case["r"], o, T=T, allow=())[:2])
    V = dims[0] * dims[1] * dims[2] * dims[3]
    cpp, prop, _ = dp.dp_solve_point(ctx, f, Ms[0], profs[0], src, case["r"], o, T=T, V=V,
                                     want_prop=case["out"] == "prop", allow=())
    return [cpp] if prop is None else [cpp, prop]


def run(s):
    case, dims = s["case"], s["dims"]
    kind = case["kind"]
    if kind == "solve":
        return _one_solve(case, s["ctx"], s["field"].id, dims, s["src"])
    if kind == "config":
        f = dp.dp_field_load(s["ctx"], s["links"], dims, case["bc_t"])
        dp.dp_field_set_csw(s["ctx"], f, case["csw"])
        out = _one_solve(case, s["ctx"], f, dims, s["src"])
        dp.dp_field_free(s["ctx"], f)
        return out
    if kind == "serve":
        sv = s["serving"]
        ts = [dp.dp_submit(sv.ctx, sv.fields[k], M, prof, src, case["r"]) for k, _, M, prof, src in s["requests"]]
        return [dp.dp_wait(sv.ctx, t, q[1][0], allow=())[0] for t, q in zip(ts, s["requests"])]
    if kind == "schur":
        for dagger in (0, 1):
            dp.dp_schur_dev(s["ctx"], s["field"].id, _masses(case)[0], _profiles(case)[0], s["src"], case["prec"],
                            case["compress12"], 0, dagger, s["in"].data_ptr(), s["out"][dagger].data_ptr(),
                            case["nrhs"])
        return s["out"]
    if kind == "apply":
        return [dp.dp_apply(s["ctx"], s["field"].id, "full", _masses(case)[0], _profiles(case)[0], s["src"],
                            case["prec"], s["psi"])]
    dp.dp_restore_contract_dev(s["ctx"], s["field"].id, s["profiles"], s["src"], s["x"][0].data_ptr(),
                               s["x"][1].data_ptr(), s["cpp"].data_ptr())
    return [s["cpp"]]


def _iterations(M):
    """Nominal BiCGStab iterations of a solve to 1e-10 .. 1e-11."""
    return round(51 * math.exp(-0.95 * M))


def work(case):
    """Solves: the hopping applications of the nominal number of Krylov
    iterations, each reading its spinors, links and clover blocks once and
    writing its result, in the precision of the solver.  Operators and
    contractions: their inputs and outputs."""
    V = math.prod(_ints(case["dims"]))
    Vh = V // 2

    def hops(vh, n, prec):
        w = 8 if prec == "fp64" else 4
        link = {"fp64": 18 * 8, "mixed_fp32": 48, "mixed_fp16": 28, "mixed_bf16": 28}[prec]
        return vh * (n * 48 * w + 8 * link + 72 * w), vh * n * 1920
    if case["kind"] == "contract":
        return {"bytes": V * 12 * case["groups"] * 12 * 16, "flops": V * 12 * case["groups"] * 60}
    if case["kind"] == "schur":
        b, f = hops(Vh, case["nrhs"], case["prec"])
        return {"bytes": 4 * b, "flops": 4 * f}
    if case["kind"] == "apply":
        return {"bytes": V * case["nrhs"] * 24 * 16, "flops": V * case["nrhs"] * 1920}
    if case["kind"] == "serve":
        b = f = 0
        for k in range(case["requests"]):
            bb, ff = hops(math.prod(_ints(case["dims"] if k % 2 == 0 else case["dims2"])) // 2, 12, "mixed_fp32")
            b, f = b + 4 * _iterations(0.4) * bb, f + 4 * _iterations(0.4) * ff
        return {"bytes": b, "flops": f}
    Ms = _masses(case)
    b = f = 0
    for M in Ms:
        bb, ff = hops(Vh, 12, case["prec"])
        b, f = b + 4 * _iterations(M) * bb, f + 4 * _iterations(M) * ff
    if case["kind"] == "config":
        b += V * 4 * 18 * 8
    if case["out"] == "prop":
        b += V * 12 * 24 * 8
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits with plain torch ---------------------------------------------

_AXIS = (0, 3, 2, 1)  # direction -> axis of (T, Lz, Ly, Lx, ...)


def _gammas():
    s = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]], complex), np.array([[1, 0], [0, -1]], complex)]
    e = [-np.eye(2, dtype=complex)] + [-1j * k for k in s]
    g = np.zeros((4, 4, 4), complex)
    for mu in range(4):
        g[mu, :2, 2:] = e[mu]
        g[mu, 2:, :2] = e[mu].conj().T
    return g


def _alphas(prof, dims, src):
    out = []
    for mu in range(4):
        rel = (np.arange(dims[mu]) - src[mu]) % dims[mu]
        h = rel - 0.5 * dims[mu]
        a = np.ones(dims[mu])
        if prof[0] == "exp_t" and mu == 0:
            a = np.exp(prof[1] * rel)
        if prof[0] == "cosh_t" and mu == 0:
            a = 1 / np.cosh(prof[1] * h)
        if prof[0] == "cosh_4d":
            a = np.cosh(prof[1] * h)
        out.append(a)
    return out


class _Operator:
    """The preconditioned Wilson-clover operator on (T, Lz, Ly, Lx, 3, n, 4)
    complex128 spinors."""

    def __init__(self, U, dims, bc_t, csw, M, prof, src):
        self.U, self.dims = U, dims
        g = _gammas()
        self.al = _alphas(prof, dims, src)
        self.P = [[torch.from_numpy((np.eye(4) + sg * g[mu]).T.copy()).cuda() for sg in (-1, 1)] for mu in range(4)]
        self.coef = []
        for mu in range(4):
            a, L = self.al[mu], dims[mu]
            f, b = -0.5 * a / np.roll(a, -1), -0.5 * a / np.roll(a, 1)
            if mu == 0:
                f[L - 1] *= bc_t
                b[0] *= bc_t
            shape = [1] * 7
            shape[_AXIS[mu]] = L
            self.coef.append([torch.from_numpy(v).cuda().reshape(shape) for v in (f, b)])
        self.A = self._diagonal(csw, M, g)
        self.Ainv = torch.linalg.inv(self.A)

    def _diagonal(self, csw, M, g):
        U = [self.U[..., mu, :, :] for mu in range(4)]
        V = math.prod(self.dims)

        def at(X, mu, k):
            return torch.roll(X, -k, _AXIS[mu])
        A = (4 + M) * torch.eye(12, dtype=torch.complex128, device="cuda").expand(V, 12, 12).clone()
        for mu in range(4):
            for nu in range(mu + 1, 4):
                P = U[mu] @ at(U[nu], mu, 1) @ at(U[mu], nu, 1).mH @ U[nu].mH  # x -> mu -> nu
                Q = P.clone()
                C = U[nu] @ at(at(U[mu], nu, 1), mu, -1).mH @ at(U[nu], mu, -1).mH @ at(U[mu], mu, -1)
                Q += C
                lo = at(at(U[mu], mu, -1), nu, -1)
                Q += at(U[mu], mu, -1).mH @ at(at(U[nu], mu, -1), nu, -1).mH @ lo @ at(U[nu], nu, -1)
                Q += at(U[nu], nu, -1).mH @ at(U[mu], nu, -1) @ at(at(U[nu], mu, 1), nu, -1) @ U[mu].mH
                F = ((Q - Q.mH) / 8).reshape(V, 3, 3)
                sig = torch.from_numpy(0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])).cuda()
                A += 0.5j * csw * torch.einsum("st,vab->vsatb", sig, F).reshape(V, 12, 12)
        return A

    def site(self, mats, psi):
        """mats (V, 12, 12), index 3 * spin + colour, on every site."""
        n = psi.shape[5]
        v = psi.reshape(-1, 3, n, 4).permute(0, 3, 1, 2).reshape(-1, 12, n)
        return (mats @ v).reshape(-1, 4, 3, n).permute(0, 2, 3, 1).reshape(psi.shape)

    def hop(self, psi, reciprocal=False):
        out = torch.zeros_like(psi)
        n = psi.shape[5]
        flat = psi.shape[:5] + (4 * n,)
        for mu in range(4):
            Um = self.U[..., mu, :, :]
            f, b = self.coef[mu]
            if reciprocal:
                f, b = (torch.where(c != 0, 0.25 / torch.where(c != 0, c, torch.ones_like(c)), c) for c in (f, b))
            h = (Um @ torch.roll(psi, -1, _AXIS[mu]).reshape(flat)).reshape(psi.shape)
            out += f * (h @ self.P[mu][0])
            h = torch.roll((Um.mH @ psi.reshape(flat)).reshape(psi.shape), 1, _AXIS[mu])
            out += b * (h @ self.P[mu][1])
        return out

    def alpha(self):
        a = torch.ones((1,) * 7, dtype=torch.float64, device="cuda")
        for mu in range(4):
            shape = [1] * 7
            shape[_AXIS[mu]] = self.dims[mu]
            a = a * torch.from_numpy(self.al[mu]).cuda().reshape(shape)
        return a


def _parity(dims):
    T, Lx, Ly, Lz = dims
    ix = [torch.arange(n, device="cuda") for n in (T, Lz, Ly, Lx)]
    return (ix[0].view(-1, 1, 1, 1) + ix[1].view(-1, 1, 1) + ix[2].view(-1, 1) + ix[3]) & 1


def _halves(t, dims, prec):
    """Packed spinors of parity 0 -> (T, Lz, Ly, Lx, 3, n, 4)."""
    if prec != "fp64":
        t = t.double()
        t = torch.stack([torch.complex(t[..., 0], t[..., 2]), torch.complex(t[..., 1], t[..., 3])], -1).flatten(2)
    else:
        t = torch.view_as_complex(t)
    n = t.shape[2]
    T, Lx, Ly, Lz = dims
    out = torch.zeros((T, Lz, Ly, Lx, 3, n, 4), dtype=torch.complex128, device="cuda")
    out[_parity(dims) == 0] = t.reshape(4, 3, -1, n).permute(2, 1, 3, 0)
    return out


def _packed(psi, dims, prec):
    t = psi[_parity(dims) == 0].permute(3, 1, 0, 2).reshape(12, -1, psi.shape[5])
    if prec == "fp64":
        return torch.view_as_real(t.contiguous())
    t = t.reshape(12, t.shape[1], -1, 2)
    return torch.stack([t[..., 0].real, t[..., 1].real, t[..., 0].imag, t[..., 1].imag], -1)


def _propagator(op, src, tol=1e-14):
    """The 12 columns of (D' + M)^-1 on the scaled point source, restored."""
    T, Lx, Ly, Lz = op.dims
    b = torch.zeros((T, Lz, Ly, Lx, 3, 12, 4), dtype=torch.complex128, device="cuda")
    t, x, y, z = src
    for k in range(12):
        b[t, z, y, x, k % 3, k, k // 3] = 1
    a = op.alpha()
    b = op.site(op.Ainv, b * a)

    def dot(u, v):
        return (u.conj() * v).sum((0, 1, 2, 3, 4, 6)).reshape(1, 1, 1, 1, 1, -1, 1)

    def K(v):  # A^-1 (D' + M)
        return v + op.site(op.Ainv, op.hop(v))
    X, r, rh = torch.zeros_like(b), b.clone(), b.clone()
    p, rho, bb = r.clone(), dot(b, b), dot(b, b).real
    for _ in range(2000):
        v = K(p)
        al = rho / dot(rh, v)
        s = r - al * v
        q = K(s)
        om = dot(q, s) / dot(q, q)
        X = X + al * p + om * s
        r = s - om * q
        if bool((dot(r, r).real <= tol * tol * bb).all()):
            break
        new = dot(rh, r)
        p = r + (new / rho) * (al / om) * (p - om * v)
        rho = new
    return X / a


def exact(case, seed):
    dims = _ints(case["dims"])
    T, V, kind = dims[0], math.prod(_ints(case["dims"])), case["kind"]
    if kind == "contract":
        kinds, srcs = _groups(case, seed)
        xs = [_spinor(dims, 12 * case["groups"], "fp64", seed + p) for p in (0, 1)]
        par = _parity(dims)
        out = torch.zeros((case["groups"], T), dtype=torch.float64, device="cuda")
        for g in range(case["groups"]):
            full = torch.zeros(par.shape, dtype=torch.float64, device="cuda")
            for p in (0, 1):
                full[par == p] = xs[p][:, :, 12 * g: 12 * g + 12].square().sum((0, 2, 3))
            for mu, a in enumerate(_alphas(kinds[g], dims, srcs[g])):
                shape = [1] * 4
                shape[_AXIS[mu]] = dims[mu]
                full = full / torch.from_numpy(a).cuda().reshape(shape) ** 2
            out[g] = -torch.roll(full.sum((1, 2, 3)), -srcs[g][0])
        return [out]
    if kind == "serve":
        return None
    Ms, profs = _masses(case), _profiles(case)
    src = _source(dims, seed)
    if kind in ("solve", "config"):
        if V * len(Ms) > 150000:
            return None
        op = _Operator(_links(dims, case["eps"], seed), dims, case["bc_t"], case["csw"], Ms[0], profs[0], src)
        cpps, last = [], None
        for M, prof in zip(Ms, profs):
            if last is not None:
                op = _Operator(op.U, dims, case["bc_t"], case["csw"], M, prof, src)
            last = S = _propagator(op, src)
            cpps.append(-torch.roll(S.abs().square().sum((1, 2, 3, 4, 5, 6)), -src[0]))
        if len(Ms) > 1:
            return [torch.stack(cpps).cpu().numpy()]
        if case["out"] == "corr":
            g0 = torch.from_numpy(_gammas()[0]).cuda()
            ap = torch.einsum("tzyxcns,rs,tzyxcnr->t", S, g0, S.conj()).real
            return [cpps[0].cpu().numpy(), torch.roll(ap, -src[0]).cpu().numpy()]
        if case["out"] == "prop":
            return [cpps[0].cpu().numpy(), S.permute(5, 0, 1, 2, 3, 6, 4).reshape(12, V, 4, 3).cpu().numpy()]
        return [cpps[0].cpu().numpy()]
    if kind == "schur" and (V * case["nrhs"] > 9000000 or case["prec"] in ("mixed_fp16", "mixed_bf16")):
        return None  # (16-bit links are not the links of the field)
    op = _Operator(_links(dims, case["eps"], seed), dims, case["bc_t"], case["csw"], Ms[0], profs[0], src)
    if kind == "apply":
        rng = np.random.default_rng(seed + 5)
        shape = (case["nrhs"], dims[0], dims[3], dims[2], dims[1], 4, 3)
        psi = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
        x = torch.from_numpy(psi).cuda().permute(1, 2, 3, 4, 6, 0, 5).contiguous()
        return [(op.site(op.A, x) + op.hop(x)).permute(5, 0, 1, 2, 3, 6, 4).cpu().numpy()]
    x = _halves(_spinor(dims, case["nrhs"], case["prec"], seed), dims, case["prec"])
    even = (_parity(dims) == 0).reshape(_parity(dims).shape + (1, 1, 1))
    y = x - even * op.site(op.Ainv, op.hop(op.site(op.Ainv, op.hop(x))))
    sg = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda")
    u = op.hop(op.site(op.Ainv, op.hop(sg * op.site(op.Ainv, x), True)), True)
    z = x - even * (sg * u)
    return [_packed(y, dims, case["prec"]), _packed(z, dims, case["prec"])]
