"""The calls whose speed this repository answers for.

Each case is one call of the C ABI as a program makes it: angular power
spectra of one cosmology or of a batch (FP64, FP32, tensor cores; device or
host arrays; direct or as a replayed graph; split or symmetrised R form),
of a non-separable spectrum, with the non-linear correction, or the basis
integrals of a grid.

A program builds a plan once and evaluates many cosmologies on it, so plans
are kept between states.  Their basis tables are given with
``blast_basis_set``: the k quadrature of Chebyshev polynomials times two
spherical Bessel functions, with a few hundred k nodes and the Debye form of
j_l (oscillating past its turning point, exponentially small before it), so
that ranges, decay and cancellation are those of the real integrals and a
table takes a second instead of minutes.  Tracer kernels, growth and P(k) have
the shapes of ``synth`` (Gaussian bins, lensing efficiencies, wiggles).
"""
import collections
import ctypes
import math
import types

import numpy as np
import torch

from paper_2410_03632_gb300 import blast as bl
from paper_2410_03632_gb300 import synth

PREC = {"fp64": bl.BLAST_FP64, "fp32": bl.BLAST_FP32, "mixed": bl.BLAST_BF16S}
MASK = {"fp64": bl.BLAST_BASIS_FP64, "fp32": bl.BLAST_BASIS_FP32, "mixed": bl.BLAST_BASIS_BF16S}
K_MIN, K_MAX, CHI_MIN, CHI_MAX = 1e-4, 10.0, 26.0, 4100.0
N_TAB = 256    # points of the tabulated P(k)
N_KSUM = 512   # k nodes of the given basis tables
F64 = torch.float64


def _case(name, kind, prec, n, grid, bins, **more):
    n_ell, ell_hi, X, R, N = grid
    c = {"name": name, "kind": kind, "prec": prec, "n": n, "n_ell": n_ell, "ell_hi": ell_hi, "n_chi": X, "n_R": R,
         "n_cheb": N, "clust": bins[0], "lens": bins[1], "r_form": 0, "ragged": False, "host": False, "graph": False}
    c.update(more)
    return c


ONE_BIN = (16, 200, 64, 64, 32)          # 1+1 bins, 16 ells: synth's "c0"
TOMO = (64, 1000, 128, 128, 64)          # 5+5 bins, 64 ells: synth's "c1"
WIDE = (32, 2000, 256, 192, 96)          # 10+10 bins: synth's "c2" on every third of its ells


def listed():
    return [
        # the smallest call: one cosmology, one bin of each kind, as a 3x2pt script's first test does
        _case("fp64_one_small", "cl", "fp64", 1, ONE_BIN, (1, 1)),
        # one step of a sampler that asks for FP64, one cosmology at a time
        _case("fp64_one", "cl", "fp64", 1, TOMO, (5, 5)),
        # an ensemble of walkers or a training set in FP64
        _case("fp64_batch", "cl", "fp64", 24, TOMO, (5, 5)),
        # the precision grid with the non-linear correction, as a final best fit is evaluated
        _case("nonlinear_one_wide", "nonlinear", "fp64", 1, WIDE, (10, 10)),
        # the single-precision option on an ensemble
        _case("fp32_batch", "cl", "fp32", 48, TOMO, (5, 5)),
        # a serving request on its own: the tensor-core path at its smallest
        _case("mixed_one", "cl", "mixed", 1, TOMO, (5, 5)),
        # the headline: a large batch on the tensor cores
        _case("mixed_batch", "cl", "mixed", 256, TOMO, (5, 5)),
        # ragged requests (own bin counts, own ell sets) on the wide grid
        _case("mixed_wide_ragged", "cl", "mixed", 150, WIDE, (10, 10), ragged=True),
        # a user with NumPy arrays: pinned host inputs and outputs, an odd batch
        _case("mixed_host", "cl", "mixed", 37, TOMO, (5, 5), host=True),
        # an ensemble sampler's inner loop: the symmetrised form in a replayed graph
        _case("mixed_graph_sym", "cl", "mixed", 64, (40, 1000, 128, 96, 64), (5, 5), r_form=1, graph=True),
        # a spectrum with scale-dependent growth, sampled at every chi-R node
        _case("nonsep_one", "nonsep", "fp64", 1, TOMO, (5, 5)),
        # what a user pays once per grid: the basis integrals (part of the 1+1-bin grid, full k range)
        _case("basis_build", "basis", "fp64", 1, (16, 200, 38, 64, 32), (1, 1)),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["cl"] * 8 + ["nonlinear", "nonsep", "basis"])
    prec = rng.choice(["fp64", "fp64", "fp32", "mixed", "mixed", "mixed"]) if kind == "cl" else "fp64"
    mixed = prec == "mixed"
    n_ell, X = rng.randint(6, 64), rng.randint(9, 140)
    R = 32 * rng.randint(1, 6) if mixed else 2 * rng.randint(5, 96)
    N = rng.randint(12, 96)
    ng, ns = rng.randint(1, 10), rng.randint(1, 10)
    most = 256 if mixed else 48
    if kind == "basis":
        n_ell, X, R, N = rng.randint(6, 16), rng.randint(5, 38), 2 * rng.randint(4, 32), rng.randint(12, 32)
    while n_ell * X * R * N > 64 * 128 * 128 * 64:   # no grid above the 5+5-bin one
        X = X // 2 + 1
    # work of the batch within that of the largest listed ones
    cap = 64 * 128 * 128 * 64 * most // (n_ell * X * R * N)
    n = log_int(1, min(most, max(1, cap))) if kind == "cl" else 1
    c = _case("", kind, prec, n, (n_ell, 200 if kind == "basis" else rng.choice([200, 1000, 2000]), X, R, N), (ng, ns),
                 r_form=int(kind == "cl" and rng.random() < 0.3), ragged=n > 1 and rng.random() < 0.4,
                 host=rng.random() < 0.3 and kind == "cl")
    del c["name"]
    return c


# ------------------------------------------------------------------ grids
def _ells(case):
    return synth.ell_list(case["n_ell"], 2, case["ell_hi"]).astype(np.float64)


def _fejer1(n):
    th = np.pi * (2.0 * np.arange(n - 1, -1, -1) + 1.0) / (2.0 * n)
    j = np.arange(1, n // 2 + 1)
    w = 2.0 / n * (1.0 - 2.0 * np.sum(np.cos(2.0 * j * th[:, None]) / (4.0 * j * j - 1.0), axis=1))
    return np.cos(th), w


def _nodes(case):
    """chi, its weights, R, its weights and the Chebyshev k nodes of the case's grid."""
    X, n_R, N = case["n_chi"], case["n_R"], case["n_cheb"]
    chi = np.linspace(CHI_MIN, CHI_MAX, X)
    h, w = chi[1] - chi[0], np.zeros(X)
    end = X - 1 if X % 2 else X - 4
    for a in range(end + 1):
        w[a] += h / 3.0 * (1.0 if a in (0, end) else 4.0 if a % 2 else 2.0)
    if X % 2 == 0:
        w[X - 4:] += np.array([1.0, 3.0, 3.0, 1.0]) * 3.0 * h / 8.0
    if case["r_form"]:
        x, f = _fejer1(2 * n_R + 1)
        R, wR = x[n_R + 1:], f[n_R + 1:]
    else:
        x, f = _fejer1(n_R // 2)
        R = np.concatenate([0.6 + 0.4 * x, 1.4 + 0.4 * x])
        wR = np.concatenate([0.4 * f, 0.4 * f])
    t = np.cos(np.pi * (2.0 * np.arange(N) + 1.0) / (2.0 * N))
    return chi, w, R, wR, np.exp(math.log(K_MIN) + 0.5 * math.log(K_MAX / K_MIN) * (t + 1.0))


def _debye(l, x):
    """j_l(x) away from its turning point, smooth across it."""
    nu = l + 0.5
    s = nu / x
    d = torch.sqrt(torch.abs(x * x - nu * nu))
    amp = torch.rsqrt(x * torch.sqrt(d * d + nu ** (4.0 / 3.0)))
    over = amp * torch.cos(d - nu * torch.arccos(s.clamp(max=1.0)) - 0.25 * math.pi)
    under = 0.5 ** 0.5 * amp * torch.exp(d - nu * torch.arccosh(s.clamp(min=1.0)))
    return torch.where(s < 1.0, over, under)


def _table(case):
    """The given basis table [3][n_ell][n_cheb][n_chi n_R] in FP64 on the GPU."""
    chi, _, R, _, _ = _nodes(case)
    X, n_R, N = case["n_chi"], case["n_R"], case["n_cheb"]
    u = torch.linspace(-1.0, 1.0, N_KSUM, dtype=F64, device="cuda")
    k = torch.exp(math.log(K_MIN) + 0.5 * math.log(K_MAX / K_MIN) * (u + 1.0))
    w = k * (0.5 * math.log(K_MAX / K_MIN) * 2.0 / (N_KSUM - 1))
    w[0] *= 0.5
    w[-1] *= 0.5
    cheb = torch.cos(torch.arange(N, dtype=F64, device="cuda")[:, None] * torch.arccos(u))
    A = torch.cat([cheb * (w * k ** p) for p in (2, 0, -2)])            # [3 N][k]
    c = torch.tensor(chi, device="cuda")
    cR = (c[:, None] * torch.tensor(R, device="cuda")).reshape(-1)
    T = torch.empty(3, case["n_ell"], N, X * n_R, dtype=F64, device="cuda")
    for e, l in enumerate(_ells(case)):
        near = _debye(l, k[:, None] * c).repeat_interleave(n_R, dim=1)
        T[:, e] = (A @ (near * _debye(l, k[:, None] * cR))).view(3, N, X * n_R)
    return T


_PLANS = collections.OrderedDict()


def _plan(case):
    key = tuple(case[f] for f in ("n_ell", "ell_hi", "n_chi", "n_R", "n_cheb", "clust", "lens", "r_form", "prec")) + (
        case["kind"] == "basis",)
    if key not in _PLANS:
        spec = synth.PlanSpec(_ells(case).astype(np.int32), case["n_chi"], CHI_MIN, CHI_MAX, case["n_R"], 0.2, 1.8,
                              case["n_cheb"], K_MIN, K_MAX, 1, synth.kquad_points(K_MIN, K_MAX, CHI_MAX, 1.8),
                              case["clust"], case["lens"], case["r_form"])
        plan = bl.Plan(spec, device=torch.cuda.current_device())
        if case["kind"] != "basis":
            T = _table(case)
            torch.cuda.synchronize()
            bl._check(bl.lib().blast_basis_set(plan.h, T.data_ptr(), 1, MASK[case["prec"]], None), "blast_basis_set")
            del T
        _PLANS[key] = plan
        while len(_PLANS) > 6:
            _PLANS.popitem(last=False)
    return _PLANS[key]


# ------------------------------------------------------------------ cosmologies
def _growth(chi, om):
    return 1.0 / (1.0 + (0.55 + 0.5 * (om - 0.3)) * chi / 3000.0)


def _kernels(chi, ng, ns, om):
    """[ng + ns][...] clustering kernels, and lensing efficiencies over chi^2, at the distances chi."""
    far = 3200.0 * (1.0 - 0.5 * (om - 0.3))           # chi of the deepest bin

    def place(i, n):
        return 600.0 + (far - 600.0) * (i + 0.5) / n

    rows = []
    for i in range(ng):
        s = 120.0 + 18.0 * i
        rows.append(torch.exp(-0.5 * ((chi - place(i, ng)) / s) ** 2) / (s * math.sqrt(2.0 * math.pi)))
    for i in range(ns):
        eff = sum(wt * torch.clamp(1.0 - chi / (place(i, ns) + dx), min=0.0)
                  for dx, wt in ((-250.0, 0.1), (-120.0, 0.25), (0.0, 0.3), (120.0, 0.25), (250.0, 0.1)))
        rows.append(1.5 * om / 2997.92458 ** 2 * (1.0 + chi / 2600.0) * eff / chi)
    return torch.stack(rows)


def _pk(k, c):
    x = k / 0.02
    wig = 1.0 + c["wiggle"] * torch.sin(105.0 * k + c["phase"]) * torch.exp(-(k / 0.3) ** 2)
    return 5e4 * (c["s8"] / 0.8) ** 2 * x / (1.0 + x ** (1.0 - c["slope"])) * wig


def _cosmologies(case, seed):
    """Seeded parameters of the case's cosmologies, with their tracer counts and ell sets."""
    rng = np.random.default_rng([2410, seed])
    shapes = np.random.default_rng([2410, case["n"], case["n_ell"]])   # counts belong to the case
    out = []
    for _ in range(case["n"]):
        c = {"om": rng.uniform(0.25, 0.35), "slope": rng.uniform(-2.5, -1.5), "wiggle": rng.uniform(0.03, 0.08),
             "phase": rng.uniform(0.0, 2.0 * np.pi), "s8": rng.uniform(0.7, 0.9), "ng": case["clust"],
             "ns": case["lens"], "sel": None}
        if case["ragged"]:
            c["ng"] = int(shapes.integers(min(2, case["clust"]), case["clust"] + 1))
            c["ns"] = int(shapes.integers(min(2, case["lens"]), case["lens"] + 1))
            some = int(shapes.integers((case["n_ell"] + 3) // 4, case["n_ell"] + 1))
            c["sel"] = sorted(int(e) for e in shapes.choice(case["n_ell"], size=some, replace=False))
        out.append(c)
    return out


def _arrays(case, c):
    """One cosmology's request arrays, on the GPU."""
    chi, _, R, _, _ = _nodes(case)
    ch = torch.tensor(chi, device="cuda")
    cR = (ch[:, None] * torch.tensor(R, device="cuda")).reshape(-1)
    k = torch.logspace(math.log10(K_MIN), math.log10(K_MAX), N_TAB, dtype=F64, device="cuda")
    k[0], k[-1] = K_MIN * (1.0 - 1e-12), K_MAX * (1.0 + 1e-12)
    return {"kern_chi": _kernels(ch, c["ng"], c["ns"], c["om"]), "kern_Rchi": _kernels(cR, c["ng"], c["ns"], c["om"]),
            "growth_chi": _growth(ch, c["om"]), "growth_Rchi": _growth(cR, c["om"]), "k_tab": k, "p_tab": _pk(k, c)}


def _node_samples(case, c):
    """P(k_j, chi_a, R_r chi_a) with a scale-dependent growth, [n_chi n_R][n_cheb]."""
    chi, _, R, _, kc = _nodes(case)
    ch = torch.tensor(chi, device="cuda")
    near, far = ch[:, None].expand(-1, len(R)).reshape(-1, 1), (ch[:, None] * torch.tensor(R, device="cuda")).reshape(-1, 1)
    k = torch.tensor(kc, device="cuda")
    damp = 1.0 - 0.04 * (near + far) / 8000.0 * torch.tanh(k / 0.1)
    return (_pk(k, c) * damp).contiguous()


def _limber_samples(case, c):
    """A non-linear P(k) at the Limber points, [n_ell][n_chi]."""
    chi = torch.tensor(_nodes(case)[0], device="cuda")
    k = (torch.tensor(_ells(case), device="cuda")[:, None] + 0.5) / chi
    return (_pk(k, c) * _growth(chi, c["om"]) ** 2 * (1.0 + 0.6 * k / (0.2 + k))).contiguous()


def _pairs(c):
    return bl.blast_npairs(c["ng"], c["ns"])


def _n_sel(case, c):
    return case["n_ell"] if c["sel"] is None else len(c["sel"])


def prepare(case, seed):
    plan = _plan(case)
    st = types.SimpleNamespace(case=case, plan=plan, prec=PREC[case["prec"]])
    if case["kind"] == "basis":
        # the integrals depend on the grid alone: a seed moves the k range and with it every integral
        rng = np.random.default_rng([2410, seed])
        spec = types.SimpleNamespace(**vars(plan.spec))
        spec.k_min, spec.k_max = _basis_range(rng)
        st.plan = bl.Plan(spec, device=torch.cuda.current_device())
        st.out = torch.empty(3, plan.L, plan.N, plan.Q, dtype=F64, device="cuda")
        return st
    st.cosmo = _cosmologies(case, seed)
    st.arrays = [_arrays(case, c) for c in st.cosmo]
    if case["host"]:
        st.arrays = [{f: t.cpu().pin_memory().numpy() for f, t in a.items()} for a in st.arrays]
    st.reqs = []
    for c, a in zip(st.cosmo, st.arrays):
        rq = types.SimpleNamespace(n_clust=c["ng"], n_lens=c["ns"], **(
            a if case["host"] else {"k_tab": np.empty(N_TAB)}))
        st.reqs.append(plan.request(rq, ell_sel=c["sel"], device_arrays=None if case["host"] else a))
    sizes = [_pairs(c) * _n_sel(case, c) for c in st.cosmo]
    st.out = torch.zeros(sum(sizes), dtype=F64, device="cpu" if case["host"] else "cuda")
    if case["host"]:
        st.out = st.out.pin_memory()
    at = np.concatenate([[0], np.cumsum(sizes)])
    st.ptrs = [st.out.data_ptr() + 8 * int(o) for o in at[:-1]]
    if case["kind"] == "nonsep":
        st.extra = _node_samples(case, st.cosmo[0])
    elif case["kind"] == "nonlinear":
        st.extra = _limber_samples(case, st.cosmo[0])
    torch.cuda.synchronize()
    if case["graph"]:
        st.graph = _Graph(bl.blast_graph_create(plan.h, st.reqs, st.prec, st.ptrs), plan)
    return st


class _Graph:
    """A captured batch, freed with its last user."""

    def __init__(self, handle, plan):
        self.handle, self.plan = handle, plan

    def __del__(self):
        bl.blast_graph_destroy(self.handle)


def _basis_range(rng):
    return K_MIN * (1.0 + 0.2 * rng.random()), K_MAX * (1.0 - 0.2 * rng.random())


def run(st):
    case, h = st.case, st.plan.h
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "basis":
        st.plan.precompute(bl.BLAST_BASIS_FP64, stream)
        bl._check(bl.lib().blast_basis_get(h, ctypes.c_void_p(st.out.data_ptr()), 1, stream), "blast_basis_get")
        return {"gg": st.out[0], "gs": st.out[1], "ss": st.out[2]}
    if case["graph"]:
        rc = bl.blast_graph_launch(st.graph.handle, stream)
    elif case["kind"] == "nonsep":
        rc = bl.blast_cl_nonsep(h, st.reqs[0], st.extra.data_ptr(), st.ptrs[0], 1, stream)
    elif case["kind"] == "nonlinear":
        rc = bl.blast_cl_nonlinear(h, st.reqs[0], st.prec, st.extra.data_ptr(), st.ptrs[0], 1, stream)
    elif case["n"] == 1:
        rc = bl.blast_cl(h, st.reqs[0], st.prec, st.ptrs[0], int(not case["host"]), stream)
    else:
        rc = bl.blast_cl_batch(h, st.reqs, st.prec, st.ptrs, int(not case["host"]), stream)
    bl._check(rc, case["kind"])
    return _by_type(case, st.out)


def _by_type(case, out):
    """The three kinds of spectra apart: they lie decades apart in size."""
    if case["ragged"]:
        return {"cl": out}
    ng, ns = case["clust"], case["lens"]
    gg, gs = ng * (ng + 1) // 2, ng * ns
    v = out.view(case["n"], -1, case["n_ell"])
    return {"gg": v[:, :gg], "gs": v[:, gg:gg + gs], "ss": v[:, gg + gs:]}


def work(case):
    L, Q, N, n, X = case["n_ell"], case["n_chi"] * case["n_R"], case["n_cheb"], case["n"], case["n_chi"]
    ng, ns = case["clust"], case["lens"]
    size = {"fp64": 8, "fp32": 4, "mixed": 10}[case["prec"]]   # bytes of a basis entry
    if case["kind"] == "basis":
        Nk = synth.kquad_points(K_MIN, K_MAX, CHI_MAX, 1.8)
        return {"bytes": 24.0 * L * N * Q, "flops": 2.0 * 3 * L * N * Q * Nk}
    if case["ragged"]:   # tracers and ells as drawn on average
        ng, ns = (2 + ng) // 2, (2 + ns) // 2
    share = 0.625 if case["ragged"] else 1.0
    pairs, b_side = bl.blast_npairs(ng, ns), ng + 2 * ns
    data = 8.0 * n * ((ng + ns + 1) * (X + Q) + 2 * N_TAB + share * pairs * L) + 3.0 * L * N * Q * size
    if case["kind"] == "nonsep":
        data += 8.0 * Q * N
    if case["kind"] == "nonlinear":
        data += 8.0 * L * X
    return {"bytes": data, "flops": 2.0 * n * share * L * (3.0 * N * Q + b_side * Q + pairs * X)}


# ------------------------------------------------------------------ 64-bit values
def _spline(u, v):
    """Second derivatives of the natural cubic spline through (u, v)."""
    n = u.numel()
    h = u[1:] - u[:-1]
    A = torch.zeros(n, n, dtype=F64, device="cuda")
    i = torch.arange(1, n - 1, device="cuda")
    A[0, 0] = A[-1, -1] = 1.0
    A[i, i - 1], A[i, i], A[i, i + 1] = h[:-1], 2.0 * (h[:-1] + h[1:]), h[1:]
    d = torch.zeros(n, dtype=F64, device="cuda")
    d[1:-1] = 6.0 * ((v[2:] - v[1:-1]) / h[1:] - (v[1:-1] - v[:-2]) / h[:-1])
    return torch.linalg.solve(A, d)


def _spline_P(a, k):
    """P(k) by the natural spline of (ln k, ln P), zero outside the table."""
    u, v = torch.log(a["k_tab"]), torch.log(a["p_tab"])
    M, x = _spline(u, v), torch.log(k)
    hi = torch.searchsorted(u, x.reshape(-1)).clamp(1, u.numel() - 1).view(x.shape)
    lo = hi - 1
    h = u[hi] - u[lo]
    t = (x - u[lo]) / h
    s = 1.0 - t
    val = s * v[lo] + t * v[hi] + h * h / 6.0 * ((s ** 3 - s) * M[lo] + (t ** 3 - t) * M[hi])
    return torch.where((k >= a["k_tab"][0]) & (k <= a["k_tab"][-1]), torch.exp(val), torch.zeros_like(val))


def _dct(P):
    """Chebyshev coefficients from samples at the nodes (last axis)."""
    N = P.shape[-1]
    j = torch.arange(N, dtype=F64, device="cuda")
    C = torch.cos(math.pi * j[:, None] * (2.0 * j + 1.0) / (2.0 * N)) * (2.0 / N)
    C[0] *= 0.5
    return P @ C.T


def _prefactors(case):
    l = torch.tensor(_ells(case), device="cuda")
    f = (l + 2.0) * (l + 1.0) * l * (l - 1.0)
    return l, f


def _spectra(case, c, a, w_of):
    """C[pair][ell] from w_of(type, ell index), the projected density without growth, [n_chi][n_R]."""
    chi, wchi, _, wR, _ = (torch.tensor(x, device="cuda") for x in _nodes(case))
    X, n_R, ng, ns = case["n_chi"], case["n_R"], c["ng"], c["ns"]
    U = wchi * chi * a["growth_chi"] * a["kern_chi"]
    V = (a["growth_Rchi"] * a["kern_Rchi"]).view(ng + ns, X, n_R) * wR
    _, f = _prefactors(case)
    pref = (torch.ones_like(f), torch.sqrt(f), f)
    sel = range(case["n_ell"]) if c["sel"] is None else c["sel"]
    cols = []
    for e in sel:
        parts = []
        for t in range(3):
            A = slice(0, ng) if t < 2 else slice(ng, ng + ns)
            B = slice(0, ng) if t == 0 else slice(ng, ng + ns)
            w = w_of(t, e)
            S = U[A] @ torch.einsum("jar,ar->aj", V[B], w)
            if case["r_form"]:
                S = S + (U[B] @ torch.einsum("iar,ar->ai", V[A], w)).T
            S = S * (2.0 / math.pi * pref[t][e])
            if t != 1:
                iu = torch.triu_indices(S.shape[0], S.shape[1], device="cuda")
                S = S[iu[0], iu[1]]
            parts.append(S.reshape(-1))
        cols.append(torch.cat(parts))
    return torch.stack(cols, dim=1)


def _limber(case, c, a, P):
    """The Limber sum with P[ell][chi]."""
    chi, wchi = (torch.tensor(x, device="cuda") for x in _nodes(case)[:2])
    ng = c["ng"]
    W = a["kern_chi"].clone()
    W[ng:] *= chi * chi
    l, f = _prefactors(case)
    nu = l + 0.5
    pref = (torch.ones_like(f), torch.sqrt(f) / nu ** 2, f / nu ** 4)
    parts = []
    for t in range(3):
        A, B = (W[:ng], W[:ng]) if t == 0 else (W[:ng], W[ng:]) if t == 1 else (W[ng:], W[ng:])
        S = torch.einsum("ia,ja,ea->ije", A * (wchi / chi ** 2), B, P) * pref[t]
        if t != 1:
            iu = torch.triu_indices(S.shape[0], S.shape[1], device="cuda")
            S = S[iu[0], iu[1]]
        parts.append(S.reshape(-1, case["n_ell"]))
    return torch.cat(parts)


def _bessel(ells, x):
    """j_l(x) for ascending integer ells: the recurrence upwards past x = l, Miller's downwards before it."""
    j0 = torch.sin(x) / x
    j1 = torch.where(x < 1e-2, x / 3.0 * (1.0 - x * x / 10.0 + x ** 4 / 280.0), (j0 - torch.cos(x)) / x)
    at, inv = {int(l): i for i, l in enumerate(ells)}, 1.0 / x
    up, down, shift = [None] * len(at), [None] * len(at), [None] * len(at)
    jm, jc = j0, j1
    for l in range(1, int(ells[-1])):
        jm, jc = jc, (2 * l + 1) * inv * jc - jm
        if l + 1 in at:
            up[at[l + 1]] = jc
    f, above, n = torch.full_like(x, 1e-250), torch.zeros_like(x), torch.zeros_like(x)
    for l in range(int(ells[-1] + 40 + 12 * ells[-1] ** (1.0 / 3.0)), 0, -1):
        if l in at:
            down[at[l]], shift[at[l]] = f, n.clone()
        f, above = (2 * l + 1) * inv * f - above, f
        big = torch.abs(f) > 1e200                     # both terms scaled down, counted
        f, above, n = torch.where(big, f * 1e-200, f), torch.where(big, above * 1e-200, above), n + big
    m = torch.maximum(torch.abs(f), torch.abs(above))
    f, above = f / m, above / m
    scale = (j0 * f + j1 * above) / ((f * f + above * above) * m)
    for l, i in at.items():
        up[i] = torch.where(x > l, up[i], down[i] * 1e-200 ** (n - shift[i]) * scale)
    return up


def _integrals(case, seed):
    """The basis integrals by Clenshaw-Curtis in k, as ``run`` returns them."""
    lo, hi = _basis_range(np.random.default_rng([2410, seed]))
    chi, _, R, _, _ = _nodes(case)
    n = synth.kquad_points(K_MIN, K_MAX, CHI_MAX, 1.8) - 1
    b = 2.0 / (4.0 * np.arange(0, n // 2 + 1) ** 2 - 1.0)
    b[0], b[-1] = 0.0, 0.5 * b[-1]
    w = (1.0 - np.fft.rfft(np.concatenate([b, np.zeros(n - b.size)]), n).real) / n   # cosine sums, first half
    w = np.concatenate([w, w[-2::-1]]) * 2.0
    w[0], w[-1] = 0.5 * w[0], 0.5 * w[-1]
    x = np.cos(np.pi * np.arange(n + 1) / n)
    k = torch.tensor(0.5 * (lo + hi) + 0.5 * (hi - lo) * x, device="cuda")
    w = torch.tensor(0.5 * (hi - lo) * w, device="cuda")
    u = (2.0 * (torch.log(k) - math.log(lo)) / (math.log(hi) - math.log(lo)) - 1.0).clamp(-1.0, 1.0)
    cheb = torch.cos(torch.arange(case["n_cheb"], dtype=F64, device="cuda")[:, None] * torch.arccos(u))
    A = torch.cat([cheb * (w * k ** p) for p in (2, 0, -2)])
    c, r = torch.tensor(chi, device="cuda"), torch.tensor(R, device="cuda")
    T = torch.empty(3, case["n_ell"], case["n_cheb"], len(chi), len(R), dtype=F64, device="cuda")
    for a in range(len(chi)):
        j = _bessel(_ells(case), k[:, None] * torch.cat([c[a:a + 1], r * c[a]]))
        for e in range(case["n_ell"]):
            T[:, e, :, a] = (A @ (j[e][:, :1] * j[e][:, 1:])).view(3, case["n_cheb"], len(R))
    T = T.view(3, case["n_ell"], case["n_cheb"], -1)
    return {"gg": T[0], "gs": T[1], "ss": T[2]}


def exact(case, seed):
    if case["kind"] == "basis":
        return _integrals(case, seed)
    T = _table(case)
    X, n_R = case["n_chi"], case["n_R"]
    out = []
    for c in _cosmologies(case, seed):
        a = _arrays(case, c)
        if case["kind"] == "nonsep":
            coef = _dct(_node_samples(case, c)).T                         # [n_cheb][q]
            C = _spectra(case, c, a, lambda t, e: (coef * T[t, e]).sum(0).view(X, n_R))
        else:
            an = _dct(_spline_P(a, torch.tensor(_nodes(case)[4], device="cuda")))
            C = _spectra(case, c, a, lambda t, e: (an @ T[t, e]).view(X, n_R))
        if case["kind"] == "nonlinear":
            chi = torch.tensor(_nodes(case)[0], device="cuda")
            k = (torch.tensor(_ells(case), device="cuda")[:, None] + 0.5) / chi
            C = C + _limber(case, c, a, _limber_samples(case, c)) - _limber(
                case, c, a, _spline_P(a, k) * a["growth_chi"] ** 2)
        out.append(C.reshape(-1))
    out = torch.cat(out)
    return _by_type(case, out.cpu() if case["host"] else out)
