"""Timed cases: the work that users of this framework have it do, through its public entry points.

A dp-adaptive topology-optimization run repeats, per design iteration, filter -> build -> solve ->
sensitivity -> (filter adjoint) -> optimality-criteria update, and per adaptive cycle the indicators
with the map update.  The cases are those steps one by one, over meshes from the smallest example
(20 x 10 Q2) to the 1024 x 512 Q3 beam, and a whole iteration.  Designs are of four stages of a run:
"early" (near its uniform start), "midway" and "graded" (smooth 0/1-like fields with grey
transitions, densities from 0.02 and 1e-3) and "binary" (0/1).

A case is a dict of plain values with a "kind":
  gradient   differentiable compliance and its backward pass: build + solve + sensitivity
  solve      build + solve
  batch      build + solve + sensitivity of several uneven instances together
  operator   build + one product with the stiffness operator
  sens       design sensitivities of a displacement (self-adjoint, or with an adjoint field)
  indicator  Kelly, density and QR indicators with the dp map update
  filter     P2 density filter and its adjoint
  oc         optimality-criteria design update
  step       one whole design iteration: build, solve, sensitivities, indicators, design update
"p" or "d" = 0 means a smooth random map of orders 1..4 / design counts 1, 2, 4, 8.
"""
import math

import numpy as np
import torch

import paper_1811_09821_gb300 as mto

DEV = torch.device("cuda", 0)
P_LEVELS, D_LEVELS = (1, 2, 3, 4), (1, 2, 4, 8)


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest call: the gradient of the first example (20 x 10 Q2, 4 x 4 design points) as a
        # user's own optimizer asks for it; launches and host latency count
        dict(name="gradient_20x10_p2_d4", kind="gradient", nx=20, ny=10, p=2, d=4, design="early", load="cantilever",
             rtol=1e-10),
        # a solve with the library's default options (FP64, element-block preconditioner) on sides that
        # do not halve, an odd design count
        dict(name="solve_33x17_p3_d5_default", kind="solve", nx=33, ny=17, p=3, d=5, design="early",
             load="cantilever", precision="fp64", precond="schwarz", norm="l2", smoother="jacobi", operator="auto",
             degree=0, rtol=1e-11),
        # the ordinary beam (160 x 80 Q3) half-way through its run, with the settings of the benchmark's
        # iterations
        dict(name="solve_160x80_p3_d8", kind="solve", nx=160, ny=80, p=3, d=8, design="midway", load="mbb",
             precision="mixed", precond="mg", norm="l2", smoother="block", operator="lead", degree=2, rtol=1e-8),
        # an adaptive cycle's solve: mixed orders with hanging nodes, mixed design counts, the settings of
        # the adaptive driver
        dict(name="solve_dp_320x160", kind="solve", nx=320, ny=160, p=0, d=0, design="early", load="cantilever",
             precision="mixed", precond="mg", norm="l2", smoother="jacobi", operator="auto", degree=0, rtol=1e-10),
        # independent instances of uneven sizes, orders and design counts solved together
        dict(name="batch_8", kind="batch", sizes="40x20:1:8 40x20:2:4 80x40:2:8 40x20:4:4 80x40:3:8 40x20:3:2 "
             "160x80:1:4 80x40:4:8", design="early", rtol=1e-10),
        # the element build of the large beam's class (mixed precision), then the PCG's operator
        dict(name="operator_480x240_p3_d8", kind="operator", nx=480, ny=240, p=3, d=8, design="binary",
             precision="mixed", op="split"),
        # the same on adaptive maps: many small classes, hanging nodes, the FP64 path
        dict(name="operator_dp_320x160_fp64", kind="operator", nx=320, ny=160, p=0, d=0, design="graded",
             precision="fp64", op="fp64"),
        # sensitivities on the large beam's class
        dict(name="sens_480x240_p3_d8", kind="sens", nx=480, ny=240, p=3, d=8, design="graded", adjoint=False),
        # indicators and map update at the end of an adaptive cycle
        dict(name="indicator_dp_320x160", kind="indicator", nx=320, ny=160, p=0, d=0, design="graded", cycle=2),
        # the filter of the densities and of the sensitivities, radius of a few subcells
        dict(name="filter_320x160_d4", kind="filter", nx=320, ny=160, p=2, d=4, design="graded", radius=0.6),
        # design update of 8.4 million values
        dict(name="oc_512x256_d8", kind="oc", nx=512, ny=256, p=1, d=8, design="graded"),
        # a whole design iteration of the benchmark's beam (524,288 Q3 elements, 33.5 million design
        # values) with the benchmark's settings, early in its run
        dict(name="step_1024x512_p3_d8", kind="step", nx=1024, ny=512, p=3, d=8, design="early", load="mbb"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any size in between, odd ones included, orders 1..5 (and
    mixed maps), design counts 1..12 (and mixed maps)."""
    kind = rng.choice(["gradient", "solve", "batch", "operator", "operator", "sens", "sens", "indicator", "indicator",
                       "filter", "oc", "step"])
    if kind == "batch":
        n = rng.randint(3, 10)
        sizes = []
        for _ in range(n):
            nx, ny = rng.choice([(40, 20), (56, 24), (80, 40), (104, 56), (160, 80)])
            sizes.append("%dx%d:%d:%d" % (nx, ny, rng.randint(1, 4), rng.choice([2, 3, 4, 8])))
        return dict(kind=kind, sizes=" ".join(sizes), design="early", rtol=1e-10)
    ny = _log_int(rng, 10, 250)
    nx = max(4, int(ny * rng.uniform(1.0, 2.5)))
    p = rng.choice([0, 1, 2, 3, 3, 4, 5])
    d = rng.choice([0, 1, 2, 3, 4, 5, 6, 8, 8, 12])
    if (nx * ny) * max(p, 2) ** 2 > 400000:   # the largest meshes at the orders they are run at
        p, d = rng.choice([0, 2, 3]), rng.choice([0, 4, 8])
    design = rng.choice(["early", "graded", "binary"])
    if kind in ("gradient", "step", "solve"):
        lev = rng.randint(0, 2)   # sides that halve `lev` times (the multigrid coarsens to 2048 DOFs)
        cy = rng.randint(5, 22)
        cx = rng.randint(cy, min(2 * cy + 9, 1023 // (cy + 1)))
        nx, ny = cx << lev, cy << lev
        load = rng.choice(["cantilever", "mbb"])
        p, d = rng.choice([0, 1, 2, 3, 4]), rng.choice([0, 2, 3, 4, 8])
        if kind == "gradient":
            return dict(kind=kind, nx=nx, ny=ny, p=p, d=d, design="early", load=load, rtol=1e-10)
        if kind == "step":
            return dict(kind=kind, nx=nx, ny=ny, p=p, d=d, design="early", load=load)
        prec = rng.choice(["mixed", "mixed", "fp64"])
        smoother = rng.choice(["jacobi", "block"])
        return dict(kind=kind, nx=nx, ny=ny, p=p, d=d, design="early", load=load, precision=prec, precond="mg",
                    norm="l2", smoother=smoother, operator=rng.choice(["auto", "split"]), degree=rng.choice([0, 2]),
                    rtol=1e-10)
    if kind == "operator":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        return dict(kind=kind, nx=nx, ny=ny, p=p, d=d, design=design, precision=prec,
                    op=rng.choice(["split", "lead"]) if prec == "mixed" else "fp64")
    if kind == "sens":
        return dict(kind=kind, nx=nx, ny=ny, p=p, d=d, design=design, adjoint=rng.random() < 0.3)
    if kind == "indicator":
        return dict(kind=kind, nx=nx, ny=ny, p=p, d=d, design="graded", cycle=rng.randint(1, 4))
    if kind == "filter":
        d = rng.choice([2, 3, 4, 5, 8])
        return dict(kind=kind, nx=nx, ny=ny, p=1, d=d, design=design, radius=round(rng.uniform(0.3, 1.2), 2))
    return dict(kind="oc", nx=_log_int(rng, 8, 600), ny=_log_int(rng, 8, 300), p=1, d=d, design="graded")


# ------------------------------------------------------------------------------------------ inputs
def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * (int(seed) % 2_000_000_011) + stream)


def _noise(gen, ny, nx, sigma):
    """Smoothed white noise (periodic Gaussian, std sigma cells) of zero mean and unit std."""
    w = torch.randn(ny, nx, generator=gen, device=DEV, dtype=torch.float64)
    ky = torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None]
    kx = torch.fft.rfftfreq(nx, device=DEV, dtype=torch.float64)[None, :]
    g = torch.exp(-2.0 * (math.pi * sigma) ** 2 * (kx ** 2 + ky ** 2))
    s = torch.fft.irfft2(torch.fft.rfft2(w) * g, s=(ny, nx))
    return (s - s.mean()) / s.std()


def _map(stream, nx, ny, levels):
    """Smooth random map of the levels over the elements (host int32), the same for every seed of a
    case: a run's maps stay while its designs change."""
    s = _noise(_gen(1, stream), ny, nx, min(6.0, 0.15 * min(nx, ny))).cpu().numpy()
    q = np.clip(np.floor((s + 2.0) / 4.0 * len(levels)), 0, len(levels) - 1).astype(int)
    return np.asarray(levels, np.int32)[q].ravel()


def _maps(case):
    nel = case["nx"] * case["ny"]
    p = _map(11, case["nx"], case["ny"], P_LEVELS) if case["p"] == 0 else np.full(nel, case["p"], np.int32)
    d = _map(12, case["nx"], case["ny"], D_LEVELS) if case["d"] == 0 else np.full(nel, case["d"], np.int32)
    return p, d


def _fine_density(gen, design, ny, nx, r):
    """Densities on a fine grid of r x r cells per element."""
    s = _noise(gen, ny * r, nx * r, 8.0)
    if design == "early":
        return (0.45 + 0.1 * s).clamp(0.1, 0.9)
    w = max(r, ny * r // 40)
    frame = torch.zeros_like(s)
    frame[:w], frame[-w:], frame[:, :w], frame[:, -w:] = 1.0, 1.0, 1.0, 1.0
    if design == "binary":
        s = s + 100.0 * frame
        sub = s.reshape(-1)[:: max(1, s.numel() // 1_000_000)]
        return (s > torch.quantile(sub, 0.6)).double()
    s = s + 4.0 * frame
    sub = s.reshape(-1)[::97]
    lo, hi = -10.0, 10.0
    for _ in range(30):   # the logistic's offset for a mean density of 0.35
        t = 0.5 * (lo + hi)
        if float(torch.sigmoid((sub - t) / 0.35).mean()) > 0.35:
            lo = t
        else:
            hi = t
    return torch.sigmoid((s - 0.5 * (lo + hi)) / 0.35).clamp(2e-2 if design == "midway" else 1e-3, 1.0)


def _pack(fine, nx, ny, d, r):
    """Packed design of the per-element counts d: subcell (i, j) takes the fine cell at its centre."""
    F = fine.reshape(ny, r, nx, r).permute(0, 2, 1, 3).reshape(ny * nx, r, r)
    if len(np.unique(d)) == 1 and int(d[0]) == r:
        return F.reshape(-1).contiguous()
    off = np.concatenate([[0], np.cumsum(d.astype(np.int64) ** 2)])
    rho = torch.empty(int(off[-1]), dtype=torch.float64, device=DEV)
    for dd in np.unique(d):
        e = np.flatnonzero(d == dd)
        c = torch.as_tensor(((np.arange(dd) + 0.5) * r / dd).astype(np.int64), device=DEV)
        v = F[torch.as_tensor(e, device=DEV)][:, c][:, :, c].reshape(len(e), -1)
        rho[torch.as_tensor(off[e], device=DEV)[:, None] + torch.arange(int(dd) ** 2, device=DEV)] = v
    return rho


def _density(case, seed, d):
    r = int(d.max())
    return _pack(_fine_density(_gen(seed, 13), case["design"], case["ny"], case["nx"], r), case["nx"], case["ny"], d, r)


def _displacement(mesh, gen):
    """A bending-like field with waves of a few elements' length and a little roughness, as solved
    displacements of a truss-like design have."""
    x, y = mesh.coords[:, 0], mesh.coords[:, 1]
    nx, ny = mesh.nx, mesh.ny
    a = torch.rand(8, generator=gen, device=DEV, dtype=torch.float64) + 0.5
    ux = a[0] * x * (y - 0.5 * ny) / nx + 0.5 * a[1] * torch.sin(0.7 * a[2] * x + 0.4 * y)
    uy = -0.5 * a[3] * x * x / nx + 0.5 * a[4] * torch.cos(0.6 * a[5] * y - 0.3 * a[6] * x)
    u = torch.stack([ux, uy], 1).reshape(-1)
    return u + 2e-2 * a[7] * torch.randn(u.numel(), generator=gen, device=DEV, dtype=torch.float64)


PREC = {"fp64": mto.MTO_FP64, "mixed": mto.MTO_MIXED}
PRECOND = {"mg": mto.PREC_MG, "schwarz": mto.PREC_SCHWARZ, "jacobi": mto.PREC_JACOBI}
NORM = {"l2": mto.NORM_L2, "jacobi": mto.NORM_JACOBI, "energy": mto.NORM_ENERGY}
SMOOTH = {"jacobi": mto.SMOOTH_JACOBI, "block": mto.SMOOTH_BLOCK}
MGOP = {"auto": mto.MG_OP_AUTO, "split": mto.MG_OP_SPLIT, "lead": mto.MG_OP_LEAD}
OP = {"fp64": mto.OP_FP64, "split": mto.OP_SPLIT, "lead": mto.OP_LEAD}


def _handle(nx, ny, p, d, load=None):
    h = mto.Handle(0)
    h.setup(nx, ny, p, d)
    fixed, f = mto.load_case(h, load or "cantilever")
    h.set_supports(fixed)
    return h, f


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, case=case, mat=mto.material())
    if kind == "batch":
        st["h"], st["f"], st["rho"], st["u"], st["dc"] = [], [], [], [], []
        for k, (nx, ny, p, d) in enumerate(_instances(case)):
            pm, dm = np.full(nx * ny, p, np.int32), np.full(nx * ny, d, np.int32)
            h, f = _handle(nx, ny, pm, dm, "cantilever" if k % 2 == 0 else "mbb")
            st["h"].append(h)
            st["f"].append(f)
            st["rho"].append(_density(dict(case, nx=nx, ny=ny), seed + 7919 * k, dm))
            st["u"].append(torch.zeros(h.ndof, dtype=torch.float64, device=DEV))
            st["dc"].append(torch.zeros(h.design_len, dtype=torch.float64, device=DEV))
        return st
    nx, ny = case["nx"], case["ny"]
    p, d = _maps(case)
    h, f = _handle(nx, ny, p, d, case.get("load"))
    rho = _density(case, seed, d)
    st.update(h=h, f=f, rho=rho)
    if kind in ("solve", "step"):
        st["u"] = torch.zeros(h.ndof, dtype=torch.float64, device=DEV)
    if kind == "operator":
        st["x"] = torch.randn(h.ndof, generator=_gen(seed, 14), device=DEV, dtype=torch.float64)
        st["y"] = torch.zeros_like(st["x"])
    if kind in ("sens", "indicator"):
        mesh = _Mesh(nx, ny, p, d)
        st["u"] = _displacement(mesh, _gen(seed, 15))
        if case.get("adjoint"):
            st["v"] = _displacement(mesh, _gen(seed, 16))
    if kind in ("sens", "step"):
        st["dc"] = torch.zeros(h.design_len, dtype=torch.float64, device=DEV)
    if kind == "indicator":
        h.build_elements(rho, st["mat"], mto.MTO_MIXED)   # the indicators follow a solved iteration
    if kind == "filter":
        st["g"] = -torch.rand(h.design_len, generator=_gen(seed, 17), device=DEV, dtype=torch.float64)
        st["out"] = [torch.empty_like(rho), torch.empty_like(rho)]
    if kind == "oc":   # sensitivities spread over several decades, as on a late design
        z = torch.randn(h.design_len, generator=_gen(seed, 18), device=DEV, dtype=torch.float64)
        st["dc"] = -torch.exp(2.0 * z) * rho * rho
    if kind in ("oc", "step"):
        st["vol"] = float(rho.sum() / len(rho)) if case["d"] else 0.35
        st["rho_new"] = torch.empty_like(rho)
    return st


def _instances(case):
    for s in case["sizes"].split():
        xy, p, d = s.split(":")
        nx, ny = xy.split("x")
        yield int(nx), int(ny), int(p), int(d)


# ------------------------------------------------------------------------------------------ passes
def run(st):
    kind, case, h, mat = st["kind"], st["case"], st["h"], st["mat"]
    if kind == "gradient":
        r = st["rho"].detach().requires_grad_(True)
        C = mto.compliance(h, r, st["f"], mat, precision=mto.MTO_MIXED, rtol=case["rtol"], precond=mto.PREC_MG,
                           check_every=16)
        C.backward()
        return dict(C=C.detach(), grad=r.grad)
    if kind == "solve":
        prec = PREC[case["precision"]]
        h.build_elements(st["rho"], mat, prec)
        h.solve(st["f"], st["u"], precision=prec, rtol=case["rtol"], norm=NORM[case["norm"]],
                precond=PRECOND[case["precond"]], check_every=16, mg_degree=case["degree"],
                mg_smoother=SMOOTH[case["smoother"]], mg_operator=MGOP[case["operator"]])
        return dict(u=st["u"])
    if kind == "batch":
        mto.build_elements_batched(h, st["rho"], mat)
        mto.solve_batched(h, st["f"], st["u"], rtol=case["rtol"], norm=mto.NORM_L2)
        C = mto.sensitivity_batched(h, st["u"], st["f"], st["rho"], mat, st["dc"])
        return dict(C=C, u=st["u"], dc=st["dc"])
    if kind == "operator":
        h.build_elements(st["rho"], mat, PREC[case["precision"]])
        xKx = h.apply_operator(st["x"], st["y"], OP[case["op"]])
        return dict(y=st["y"], xKx=xKx)
    if kind == "sens":
        if case["adjoint"]:
            return dict(dc=h.sensitivity_adjoint(st["u"], st["v"], st["rho"], mat, st["dc"]))
        C = h.sensitivity(st["u"], st["f"], st["rho"], mat, st["dc"])
        return dict(dc=st["dc"], C=C)
    if kind == "indicator":
        return h.indicator(st["u"], st["rho"], mat, mto.IndicatorOpts.paper(case["cycle"]))
    if kind == "filter":
        a, b = st["out"]
        return dict(rho=h.filter(st["rho"], a, case["radius"]), g=h.filter_adjoint(st["g"], b, case["radius"]))
    if kind == "oc":
        h.oc_update(st["rho"], st["dc"], st["vol"], st["rho_new"], want_lambda=False)
        return dict(rho_new=st["rho_new"])
    # step: the benchmark's iteration
    h.build_elements(st["rho"], mat, mto.MTO_MIXED)
    h.solve(st["f"], st["u"], precision=mto.MTO_MIXED, rtol=1e-8, norm=mto.NORM_ENERGY, check_every=32,
            precond=mto.PREC_MG, mg_degree=2, mg_smoother=mto.SMOOTH_BLOCK, mg_operator=mto.MG_OP_LEAD)
    h.sensitivity(st["u"], st["f"], st["rho"], mat, st["dc"], want_C=False)
    ind = h.indicator(st["u"], st["rho"], mat)
    h.oc_update(st["rho"], st["dc"], st["vol"], st["rho_new"], want_lambda=False)
    return dict(ind, u=st["u"], dc=st["dc"], rho_new=st["rho_new"])


# ------------------------------------------------------------------------------------------ work
def _sizes(nx, ny, p, d):
    """(elements, DOFs, design values, packed matrix entries, build FMAs) of a uniform mesh; mixed
    maps count at their mean levels (orders 1..4, counts 1, 2, 4, 8)."""
    ps, ds = P_LEVELS if p == 0 else (p,), D_LEVELS if d == 0 else (d,)
    nel = nx * ny
    mean = lambda f, v: sum(f(k) for k in v) / len(v)
    S = mean(lambda k: k * k, ds)
    P = mean(lambda k: (k + 1) ** 2 * (2 * (k + 1) ** 2 + 1), ps)
    nodes = mean(lambda k: (nx * k + 1) * (ny * k + 1), ps)
    return nel, 2 * nodes, nel * S, nel * P, nel * P * S


def work(case):
    """Each input read once and each output written once.  A build also writes its element matrices
    (FP64, and the FP32 pair of a mixed build), which stay in the handle; a solve reads them once at the
    least.  The flops are those of the definitions: the build's sums over the subcells, one operator
    product, one quadratic form per subcell."""
    kind = case["kind"]
    if kind == "batch":
        parts = [work(dict(kind="gradient", nx=nx, ny=ny, p=p, d=d)) for nx, ny, p, d in _instances(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    nel, ndof, S, P, fma = _sizes(case["nx"], case["ny"], case["p"], case["d"])
    mat = P * (8 if case.get("precision") == "fp64" else 16)
    if kind == "operator":
        return dict(bytes=8 * S + mat + 16 * ndof, flops=2 * fma + 4 * P)
    if kind == "solve":
        return dict(bytes=8 * S + 2 * mat + 16 * ndof, flops=2 * fma + 4 * P)
    if kind == "gradient":
        return dict(bytes=24 * S + 2 * mat + 16 * ndof, flops=2 * fma + 4 * P + 4 * fma)
    if kind == "sens":
        return dict(bytes=16 * S + (16 if case["adjoint"] else 8) * ndof, flops=4 * fma)
    if kind == "indicator":
        return dict(bytes=8 * S + 8 * ndof + 8 * P + 33 * nel, flops=2 * fma)
    if kind == "filter":
        cells = math.pi * (case["radius"] * case["d"]) ** 2
        return dict(bytes=32 * S, flops=8 * cells * S)
    if kind == "oc":
        return dict(bytes=24 * S, flops=8 * S)
    return dict(bytes=40 * S + 3 * mat + 16 * ndof + 33 * nel, flops=8 * fma + 4 * P)


# ------------------------------------------------------------------------------------------ 64 bits
def _gll(p):
    """Gauss-Lobatto-Legendre nodes of order p."""
    c = np.zeros(p + 1)
    c[p] = 1.0
    inner = np.sort(np.real(np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c)))) if p > 1 else []
    return np.concatenate([[-1.0], inner, [1.0]])


def _lagrange(z, t):
    """(values, derivatives) [len(t), len(z)] of the Lagrange polynomials on nodes z at points t."""
    n = len(z)
    t = np.asarray(t, float)
    V, D = np.ones((len(t), n)), np.zeros((len(t), n))
    for k in range(n):
        for j in range(n):
            if j != k:
                V[:, k] *= (t - z[j]) / (z[k] - z[j])
        for i in range(n):
            if i == k:
                continue
            w = np.full(len(t), 1.0 / (z[k] - z[i]))
            for j in range(n):
                if j not in (i, k):
                    w *= (t - z[j]) / (z[k] - z[j])
            D[:, k] += w
    return V, D


def _k0(p, d, nu=0.3):
    """Subcell stiffness tables [d^2, n_e, n_e] of unit modulus on the unit square, plane stress."""
    z, n = _gll(p), p + 1
    gx, gw = np.polynomial.legendre.leggauss(n)
    LL, DD, DL = [], [], []
    for i in range(d):
        V, D = _lagrange(z, -1.0 + (2.0 * i + 1.0 + gx) / d)
        w = gw / (2.0 * d)
        D = 2.0 * D
        LL.append(V.T @ (w[:, None] * V))
        DD.append(D.T @ (w[:, None] * D))
        DL.append(D.T @ (w[:, None] * V))
    LL, DD, DL = (np.stack(a) for a in (LL, DD, DL))
    f = 1.0 / (1.0 - nu * nu)
    D11, D12, D33 = f, f * nu, f * 0.5 * (1.0 - nu)
    kr = lambda Y, X: np.einsum("jbB,iaA->jibaBA", Y, X).reshape(d * d, n * n, n * n)
    T = lambda A: A.transpose(0, 2, 1)
    K = np.zeros((d * d, n * n, 2, n * n, 2))
    K[:, :, 0, :, 0] = D11 * kr(LL, DD) + D33 * kr(DD, LL)
    K[:, :, 1, :, 1] = D11 * kr(DD, LL) + D33 * kr(LL, DD)
    K[:, :, 0, :, 1] = D12 * kr(T(DL), DL) + D33 * kr(DL, T(DL))
    K[:, :, 1, :, 0] = K[:, :, 0, :, 1].transpose(0, 2, 1)
    return torch.as_tensor(K.reshape(d * d, 2 * n * n, 2 * n * n), device=DEV)


class _Mesh:
    """The documented node numbering (vertices, horizontal and vertical edge interiors, cell
    interiors), node coordinates, and the elements' minimum-rule node maps."""

    def __init__(self, nx, ny, p, d):
        self.nx, self.ny, self.p, self.d = nx, ny, np.asarray(p), np.asarray(d)
        P = self.p.reshape(ny, nx)
        pH, pV = np.empty((ny + 1, nx), np.int64), np.empty((ny, nx + 1), np.int64)
        pH[0], pH[ny], pH[1:ny] = P[0], P[-1], np.minimum(P[:-1], P[1:])
        pV[:, 0], pV[:, nx], pV[:, 1:nx] = P[:, 0], P[:, -1], np.minimum(P[:, :-1], P[:, 1:])
        self.pH, self.pV = pH.ravel(), pV.ravel()
        base = lambda n, first: first + np.concatenate([[0], np.cumsum(n)])
        h = base(self.pH - 1, (nx + 1) * (ny + 1))
        v = base(self.pV - 1, h[-1])
        i = base((self.p.astype(np.int64) - 1) ** 2, v[-1])
        self.hb, self.vb, self.ib, self.nodes = h[:-1], v[:-1], i[:-1], int(i[-1])
        self.off = np.concatenate([[0], np.cumsum(self.d.astype(np.int64) ** 2)])
        xy = np.empty((self.nodes, 2))
        V = np.arange((nx + 1) * (ny + 1))
        xy[V, 0], xy[V, 1] = V % (nx + 1), V // (nx + 1)
        for q in range(2, int(self.p.max()) + 1):
            t = 0.5 * (1.0 + _gll(q)[1:-1])
            k = np.arange(q - 1)
            e = np.flatnonzero(self.pH == q)
            g = self.hb[e][:, None] + k
            xy[g, 0], xy[g, 1] = (e % nx)[:, None] + t, (e // nx)[:, None] + 0.0 * t
            e = np.flatnonzero(self.pV == q)
            g = self.vb[e][:, None] + k
            xy[g, 0], xy[g, 1] = (e % (nx + 1))[:, None] + 0.0 * t, (e // (nx + 1))[:, None] + t
            e = np.flatnonzero(self.p == q)
            a, b = np.meshgrid(k, k)
            g = self.ib[e][:, None] + (b * (q - 1) + a).ravel()
            xy[g, 0], xy[g, 1] = (e % nx)[:, None] + t[a.ravel()], (e // nx)[:, None] + t[b.ravel()]
        self.coords = torch.as_tensor(xy, device=DEV)

    def elements(self, q):
        return np.flatnonzero(self.p == q)

    def local(self, q):
        """(nodes, weights) [n, (q+1)^2, q+1] of the order-q elements' local nodes."""
        e, nx = self.elements(q), self.nx
        ex, ey = e % nx, e // nx
        g, w = np.zeros((len(e), (q + 1) ** 2, q + 1), np.int64), np.zeros((len(e), (q + 1) ** 2, q + 1))
        vert = lambda x, y: y * (nx + 1) + x
        z = _gll(q)
        for b in range(q + 1):
            for a in range(q + 1):
                ln = b * (q + 1) + a
                if a in (0, q) and b in (0, q):
                    g[:, ln, 0], w[:, ln, 0] = vert(ex + a // q, ey + b // q), 1.0
                elif a in (0, q) or b in (0, q):
                    if b in (0, q):
                        x0, y0, x1, y1, t = ex, ey + b // q, ex + 1, ey + b // q, a
                        eid = y0 * nx + x0
                        o, first = self.pH[eid], self.hb[eid]
                    else:
                        x0, y0, x1, y1, t = ex + a // q, ey, ex + a // q, ey + 1, b
                        eid = y0 * (nx + 1) + x0
                        o, first = self.pV[eid], self.vb[eid]
                    s = o == q
                    g[s, ln, 0], w[s, ln, 0] = first[s] + t - 1, 1.0
                    for r in np.unique(o[~s]):
                        s = o == r
                        c = _lagrange(_gll(r), [z[t]])[0][0]
                        for k in range(r + 1):
                            node = vert(x0[s], y0[s]) if k == 0 else vert(x1[s], y1[s]) if k == r else first[s] + k - 1
                            g[s, ln, k], w[s, ln, k] = node, c[k]
                else:
                    g[:, ln, 0], w[:, ln, 0] = self.ib[e] + (b - 1) * (q - 1) + a - 1, 1.0
        return torch.as_tensor(g, device=DEV), torch.as_tensor(w, device=DEV)

    def gather(self, q, u):
        """Local displacements [n, 2 (q+1)^2] of the order-q elements."""
        g, w = self.local(q)
        return (u.reshape(-1, 2)[g] * w[..., None]).sum(2).reshape(len(g), -1)

    def classes(self):
        for q in np.unique(self.p):
            for d in np.unique(self.d[self.p == q]):
                e = np.flatnonzero((self.p == q) & (self.d == d))
                yield int(q), int(d), e, np.searchsorted(self.elements(q), e)

    def cells(self, e, d):
        return torch.as_tensor(self.off[e], device=DEV)[:, None] + torch.arange(d * d, device=DEV)


def _modulus(rho):
    return 1e-9 + rho ** 3 * (1.0 - 1e-9)


def _deform(q, U):
    """U [n, n_e] without its least-squares rigid motion about the element centre."""
    z = 0.5 * _gll(q)
    x = torch.as_tensor(np.tile(z, q + 1), device=DEV)
    y = torch.as_tensor(np.repeat(z, q + 1), device=DEV)
    ux, uy = U[:, 0::2], U[:, 1::2]
    om = ((x * uy - y * ux).sum(1) / (x * x + y * y).sum())[:, None]
    return torch.stack([ux - ux.mean(1, keepdim=True) + om * y, uy - uy.mean(1, keepdim=True) - om * x], 2).reshape(len(U), -1)


def _exact_sens(mesh, rho, u, v):
    dc = torch.empty_like(rho)
    for q, d, e, slot in mesh.classes():
        slot = torch.as_tensor(slot, device=DEV)
        U = _deform(q, mesh.gather(q, u))[slot]
        Vv = U if v is u else _deform(q, mesh.gather(q, v))[slot]
        K0 = _k0(q, d).permute(1, 0, 2).reshape(U.shape[1], -1)
        at = mesh.cells(e, d)
        for k in range(0, len(e), 4096):
            s = slice(k, k + 4096)
            w = ((Vv[s] @ K0).reshape(len(U[s]), d * d, -1) * U[s][:, None, :]).sum(2)
            dc[at[s]] = -3.0 * rho[at[s]] ** 2 * (1.0 - 1e-9) * w
    return dc


def _exact_operator(mesh, rho, x):
    y = torch.zeros_like(x).reshape(-1, 2)
    for q in np.unique(mesh.p):
        g, w = mesh.local(int(q))
        X = mesh.gather(int(q), x)
        Y = torch.zeros_like(X)
        for qq, d, e, slot in mesh.classes():
            if qq != q:
                continue
            K0 = _k0(qq, d).reshape(d * d, -1)
            at, slot = mesh.cells(e, d), torch.as_tensor(slot, device=DEV)
            for k in range(0, len(e), 8192):
                s = slice(k, k + 8192)
                K = (_modulus(rho[at[s]]) @ K0).reshape(-1, X.shape[1], X.shape[1])
                Y[slot[s]] = (K @ X[slot[s]][:, :, None])[:, :, 0]
        y.index_add_(0, g.reshape(-1), (Y.reshape(len(X), -1, 1, 2) * w[..., None]).reshape(-1, 2))
    return y.reshape(-1)


def _exact_kelly(mesh, u):
    nx, ny, nel = mesh.nx, mesh.ny, mesh.nx * mesh.ny
    ga = torch.zeros(nel, dtype=torch.float64, device=DEV)
    U, slot = {}, np.zeros(nel, np.int64)
    for q in np.unique(mesh.p):
        U[int(q)] = mesh.gather(int(q), u)
        slot[mesh.elements(q)] = np.arange(len(mesh.elements(q)))
    E = np.arange(nel).reshape(ny, nx)
    for A, B, vertical in ((E[:, :-1].ravel(), E[:, 1:].ravel(), True), (E[:-1].ravel(), E[1:].ravel(), False)):
        for qa in np.unique(mesh.p):
            for qb in np.unique(mesh.p):
                s = (mesh.p[A] == qa) & (mesh.p[B] == qb)
                if not s.any():
                    continue
                qf = int(max(qa, qb))
                gx, gw = np.polynomial.legendre.leggauss(qf + 1)
                jump = 0.0
                for q, els, end, sign in ((int(qa), A[s], 1.0, 1.0), (int(qb), B[s], -1.0, -1.0)):
                    z = _gll(q)
                    T, N = _lagrange(z, gx)[0], 2.0 * _lagrange(z, [end])[1][0]
                    W = np.einsum("gb,a->gba" if vertical else "ga,b->gba", T, N).reshape(qf + 1, -1)
                    Ue = U[q][torch.as_tensor(slot[els], device=DEV)].reshape(len(els), -1, 2)
                    jump = jump + sign * torch.einsum("gn,enc->egc", torch.as_tensor(W, device=DEV), Ue)
                val = (jump ** 2).sum(2) @ torch.as_tensor(gw, device=DEV) * 0.5 * math.sqrt(2.0) / (2.0 * qf)
                for els in (A[s], B[s]):
                    ga.index_add_(0, torch.as_tensor(els, device=DEV), val)
    return ga


def _exact_gamma_d(mesh, rho, cycle):
    lo, hi = float(rho.min()), float(rho.max())
    avg = 0.5 * (lo + hi)
    fac = avg * math.exp(-0.8 * (cycle - 1))
    rl, ru, cl, cu = lo + 0.8 * fac, hi - 0.8 * fac, lo + 0.2 * fac, hi - 0.2 * fac
    a = (rl <= rho) & (rho <= avg)
    b = ~a & (avg < rho) & (rho <= ru)
    c = ~a & ~b & (rho <= cl)
    e = ~a & ~b & ~c & (rho >= cu)
    t = a * (rho - rl) + b * (ru - rho) - c * (cl - rho) - e * (rho - cu)
    out = torch.zeros(mesh.nx * mesh.ny, dtype=torch.float64, device=DEV)
    for _, d, els, _ in mesh.classes():
        out[torch.as_tensor(els, device=DEV)] = t[mesh.cells(els, d)].sum(1) / (d * d)
    return out


def _exact_qr(mesh, rho, u):
    eps = torch.zeros(mesh.nx * mesh.ny, dtype=torch.float64, device=DEV)
    for q, d, e, slot in mesh.classes():
        U = _deform(q, mesh.gather(q, u)[torch.as_tensor(slot, device=DEV)])
        n0, n1 = U.shape[1], 2 * (q + 2) ** 2
        # f^(q+1) = M^(q+1,q) M^(q)^-1 f^(q), per component
        gx, gw = np.polynomial.legendre.leggauss(q + 2)
        A, B = _lagrange(_gll(q), gx)[0], _lagrange(_gll(q + 1), gx)[0]
        R1 = np.linalg.solve(A.T @ (gw[:, None] * A), A.T @ (gw[:, None] * B)).T
        R = torch.as_tensor(np.kron(R1, R1), device=DEV)
        fx = torch.tensor([0, 1, 2 * (q + 1) + 1], device=DEV)
        fr = torch.as_tensor(np.setdiff1d(np.arange(n1), [0, 1, 2 * (q + 1) + 1]), device=DEV)
        K0a, K0b = _k0(q, d).reshape(d * d, -1), _k0(q + 1, d).reshape(d * d, -1)
        at, els = mesh.cells(e, d), torch.as_tensor(e, device=DEV)
        for k in range(0, len(e), 4096):
            s = slice(k, k + 4096)
            Em, ue = _modulus(rho[at[s]]), U[s]
            f = ((Em @ K0a).reshape(-1, n0, n0) @ ue[:, :, None])[:, :, 0]
            jp = 0.5 * (ue * f).sum(1)
            f1 = torch.einsum("jk,ekc->ejc", R, f.reshape(len(ue), -1, 2)).reshape(len(ue), -1)
            K1 = (Em @ K0b).reshape(-1, n1, n1)
            u1 = torch.zeros_like(f1)
            u1[:, fx] = ue[:, [0, 1, 2 * q + 1]]
            rhs = f1[:, fr] - (K1[:, fr][:, :, fx] @ u1[:, fx][:, :, None])[:, :, 0]
            u1[:, fr] = torch.linalg.solve(K1[:, fr][:, :, fr], rhs)
            j1 = 0.5 * (u1 * (K1 @ u1[:, :, None])[:, :, 0]).sum(1)
            eps[els[s]] = torch.where(j1 == 0, torch.zeros_like(j1), 1.0 - jp / j1)
    return eps


def _exact_filter(case, rho, g):
    nx, ny, d, R = case["nx"], case["ny"], case["d"], case["radius"]
    grid = lambda v: v.reshape(ny, nx, d, d).permute(0, 2, 1, 3).reshape(1, 1, ny * d, nx * d)
    pack = lambda v: v.reshape(ny, d, nx, d).permute(0, 2, 1, 3).reshape(-1)
    k = int(R * d) + 1
    o = torch.arange(-k, k + 1, device=DEV, dtype=torch.float64) / d
    H = (R - torch.sqrt(o[:, None] ** 2 + o[None, :] ** 2)).clamp(min=0.0)
    conv = lambda v: sum(H[a, b] * torch.nn.functional.pad(v, (k, k, k, k))[..., a:a + ny * d, b:b + nx * d]
                         for a in range(2 * k + 1) for b in range(2 * k + 1) if H[a, b] > 0)
    x = grid(rho)
    W = conv(torch.ones_like(x))
    return pack(conv(x) / W), pack(conv(grid(g) / W))


def _exact_oc(mesh, rho, dc, vol):
    dv = torch.as_tensor(np.repeat(1.0 / mesh.d.astype(float) ** 2, mesh.d.astype(np.int64) ** 2), device=DEV)
    t = rho * torch.sqrt((-dc).clamp(min=0.0) / dv)
    lo, hi = (rho - 0.2).clamp(min=0.0), (rho + 0.2).clamp(max=1.0)
    l1, l2 = 0.0, 1e9
    new = lambda lam: torch.minimum(torch.maximum(t / math.sqrt(lam), lo), hi)
    while (l2 - l1) / (l1 + l2) > 1e-10:
        lam = 0.5 * (l1 + l2)
        if float((new(lam) * dv).sum()) > vol * mesh.nx * mesh.ny:
            l1 = lam
        else:
            l2 = lam
    return new(0.5 * (l1 + l2))


def _exact_solution(mesh, rho, load):
    """Dense solve of a uniform-order mesh."""
    nx, ny, q = mesh.nx, mesh.ny, int(mesh.p[0])
    g, _ = mesh.local(q)
    dof = (2 * g[:, :, 0][:, :, None] + torch.arange(2, device=DEV)).reshape(len(g), -1)
    d = int(mesh.d[0])
    Ke = (_modulus(rho.reshape(len(g), -1)) @ _k0(q, d).reshape(d * d, -1)).reshape(len(g), dof.shape[1], -1)
    n = 2 * mesh.nodes
    K = torch.zeros(n * n, dtype=torch.float64, device=DEV)
    K.index_add_(0, (dof[:, :, None] * n + dof[:, None, :]).reshape(-1), Ke.reshape(-1))
    K = K.reshape(n, n)
    left = torch.nonzero(mesh.coords[:, 0] == 0)[:, 0]
    f = torch.zeros(n, dtype=torch.float64, device=DEV)
    if load == "cantilever":
        fixed = torch.cat([2 * left, 2 * left + 1])
        f[2 * ((ny // 2) * (nx + 1) + nx) + 1] = -1.0
    else:
        fixed = torch.cat([2 * left, torch.tensor([2 * nx + 1], device=DEV)])
        f[2 * (ny * (nx + 1)) + 1] = -1.0
    free = torch.ones(n, dtype=torch.bool, device=DEV)
    free[fixed] = False
    u = torch.zeros_like(f)
    A = K[free][:, free]
    r = f[free]
    L = torch.linalg.cholesky(A)
    x = torch.cholesky_solve(r[:, None], L)[:, 0]
    x = x + torch.cholesky_solve((r - A @ x)[:, None], L)[:, 0]
    u[free] = x
    return f, u


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "step"):
        return None   # as many unknowns as a direct solve does not take in seconds
    p, d = _maps(case)
    nx, ny = case["nx"], case["ny"]
    rho = _density(case, seed, d)
    mesh = _Mesh(nx, ny, p, d)
    if kind in ("gradient", "solve"):
        if case["p"] == 0 or case["d"] == 0 or mesh.nodes > 6000:
            return None
        f, u = _exact_solution(mesh, rho, case["load"])
        return dict(u=u) if kind == "solve" else dict(C=torch.dot(f, u), grad=_exact_sens(mesh, rho, u, u))
    if kind == "operator":
        x = torch.randn(2 * mesh.nodes, generator=_gen(seed, 14), device=DEV, dtype=torch.float64)
        y = _exact_operator(mesh, rho, x)
        return dict(y=y, xKx=float(torch.dot(x, y)))
    if kind in ("sens", "indicator"):
        u = _displacement(mesh, _gen(seed, 15))
        if kind == "sens":
            v = _displacement(mesh, _gen(seed, 16)) if case["adjoint"] else u
            dc = _exact_sens(mesh, rho, u, v)
            if case["adjoint"]:
                return dict(dc=dc)
            return dict(dc=dc, C=-float(u[2 * ((ny // 2) * (nx + 1) + nx) + 1]))
        return dict(gamma_a=_exact_kelly(mesh, u), gamma_d=_exact_gamma_d(mesh, rho, case["cycle"]),
                    eps_qr=_exact_qr(mesh, rho, u), p_new=None, d_new=None, theta=None)
    if kind == "filter":
        g = -torch.rand(len(rho), generator=_gen(seed, 17), device=DEV, dtype=torch.float64)
        a, b = _exact_filter(case, rho, g)
        return dict(rho=a, g=b)
    z = torch.randn(len(rho), generator=_gen(seed, 18), device=DEV, dtype=torch.float64)
    vol = float(rho.sum() / len(rho)) if case["d"] else 0.35
    return dict(rho_new=_exact_oc(mesh, rho, -torch.exp(2.0 * z) * rho * rho, vol))
