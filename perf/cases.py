"""The calls that users of this library make, as measurable cases.

Every case is one pass of a program that holds a grid context (grid, options, solvent, output buffers) and hands
it a new solute, the way a scan over conformations, a geometry optimisation or a screen over solutes does:
``set_solute`` and then the initialization, its parts, its reverse mode, the batched launch, the reciprocal-space
asymptotics or the all-space integral.  The solutes are seeded globules and ellipsoids at protein density; sizes,
grids, solvents and options are those of this repository's benchmark, tests and workload definitions, odd and
ragged grids among them.

Precision of what a pass returns: with FP64 pairs the grids as the library wrote them.  With FP32 pairs the
library rounds each grid value once to single precision and widens it to its FP64 storage, so the program keeps
single-precision grids (one pass over them, part of the measured call); sums of FP32 pair terms (gradients, the
all-space integral) are kept in single precision too.  The LJ truncation integrals are FP64 with either.
"""
import math

import numpy as np
import torch

from paper_2109_09772_gb300 import rism

DENSITY = 0.116  # atoms / A^3 (protein)
MOLAR = 6.02214076e-4  # 1/A^3 per mol/L
# water and 0.1 M salt: q (e), sigma (A), eps (kcal/mol), rho (1/A^3), ionic
SITES = [(-0.8476, 3.166, 0.1553, 55.2 * MOLAR, 0), (0.4238, 1.0, 0.01, 110.4 * MOLAR, 0),
         (1.0, 2.16, 0.35, 0.1 * MOLAR, 1), (-1.0, 4.83, 0.01, 0.1 * MOLAR, 1)]
K_E, K_B, T, EPS_R, ETA = 332.0522173, 0.0019872041, 298.0, 78.44, 1.0


def listed():
    return [
        # A small-molecule solute on a small ragged grid: launches and latency are what it costs.
        dict(name="init_150", kind="init", atoms=150, nx=37, ny=21, nz=13, h=0.45, sites=4, lj="rcut", cut=4.0,
             method="tree", precision=32, degree=8, theta=0.7),
        # A mid-sized globule, the size of a small protein: the whole initialization (u, c, h, LJ tail).
        dict(name="init_2000", kind="init", atoms=2000, nx=128, ny=128, nz=128, h=0.5, sites=4, lj="rcut", cut=9.0,
             method="tree", precision=32, degree=8, theta=0.7),
        # The tubulin-dimer-sized ellipsoid of the benchmark.
        dict(name="init_13600", kind="init", atoms=13600, shape="ellipsoid", nx=224, ny=192, nz=160, h=0.5, sites=4,
             lj="rcut", cut=9.0, method="tree", precision=32, degree=8, theta=0.7),
        # A program that calls the potential and the asymptotics separately, with the tolerance-driven LJ cut-offs
        # of the parameter guide and an odd grid.
        dict(name="parts_1324_tol", kind="parts", atoms=1324, nx=107, ny=99, nz=93, h=0.5, sites=4, lj="tol", cut=1e-3,
             method="tree", precision=32, degree=8, theta=0.7),
        # The FP64 direct sum without cut-off, two water sites: the high-precision reference a user checks with.
        dict(name="direct64_200", kind="init", atoms=200, nx=64, ny=64, nz=64, h=0.5, sites=2, lj="none", cut=0.0,
             method="direct", precision=64),
        # The FP32 direct sum: the treecode's check at full size.
        dict(name="direct32_2000", kind="init", atoms=2000, nx=128, ny=128, nz=128, h=0.5, sites=4, lj="rcut", cut=9.0,
             method="direct", precision=32),
        # Forces and charge / LJ gradients of a mid-sized solute, every cotangent.
        dict(name="backward_2000", kind="backward", atoms=2000, nx=128, ny=128, nz=128, h=0.5, sites=4, lj="rcut",
             cut=9.0, method="tree", precision=32, degree=8, theta=0.7, with_h=True),
        # The largest solute differentiated: four ellipsoids stacked along z, u and c cotangents.
        dict(name="backward_55000", kind="backward", atoms=55000, shape="stack", nx=320, ny=320, nz=384, h=0.5,
             sites=4, lj="rcut", cut=9.0, method="tree", precision=32, degree=8, theta=0.7, with_h=False),
        # A screen: 32 uneven solutes, each on its own grid, in one batched launch.
        dict(name="batched_32", kind="batched", count=32, lo=500, hi=8000, sizes=0, buffer=12.0, h=0.5, sites=4,
             lj="rcut", cut=9.0, method="tree", precision=32, degree=8, theta=0.7),
        # Reciprocal-space asymptotics of the tubulin-sized solute on the whole half spectrum.
        dict(name="kspace_13600", kind="kspace", atoms=13600, shape="ellipsoid", nx=224, ny=192, nz=160, h=0.5,
             sites=4, lj="rcut", cut=9.0, method="tree", precision=32, k_tol=0.0),
        # The same of a mid-sized solute with the frequency cut-off, odd lattice sizes.
        dict(name="kspace_2000_cut", kind="kspace", atoms=2000, nx=135, ny=121, nz=120, h=0.5, sites=4, lj="rcut",
             cut=9.0, method="tree", precision=32, k_tol=1.0),
        # The all-space long-range integral of the excess chemical potential with its per-atom sums.
        dict(name="lra_13600", kind="lra", atoms=13600, shape="ellipsoid", nx=224, ny=192, nz=160, h=0.5, sites=4,
             lj="rcut", cut=9.0, method="tree", precision=32),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def grid(points, ragged=0.3):
        e = points ** (1.0 / 3.0)
        return dict(zip(("nx", "ny", "nz"), (max(9, int(e * math.exp(rng.uniform(-ragged, ragged)))) for _ in range(3))))

    kind = rng.choice(["init", "init", "parts", "direct64", "direct32", "backward", "batched", "kspace", "lra"])
    sites = rng.choice([1, 2, 4, 4, 4, 6])
    lj = rng.choice([("rcut", rng.choice([6.0, 9.0, 12.0])), ("rcut", 9.0), ("tol", rng.choice([1e-2, 1e-3])), ("none", 0.0)])
    c = dict(kind=kind, h=rng.choice([0.25, 0.4, 0.5, 0.5, 0.5]), sites=sites, lj=lj[0], cut=lj[1], method="tree",
             precision=32, degree=rng.choice([4, 6, 8, 8, 8, 10]), theta=rng.choice([0.5, 0.6, 0.7, 0.7, 0.8]))
    if kind == "direct64":
        n, m = int(log(20, 800)), log(4e3, 3e5)
        c.update(kind="init", method="direct", precision=64, atoms=n, **grid(min(m, 1.2e8 / n)))
    elif kind == "direct32":
        n, m = int(log(20, 8000)), log(4e3, 3e6)
        c.update(kind="init", method="direct", atoms=n, **grid(min(m, 1e10 / n)))
    elif kind == "batched":
        c.update(count=rng.choice([2, 5, 8, 16]), lo=rng.choice([60, 200, 500]), hi=rng.choice([1000, 4000]),
                 sizes=rng.randrange(1000), buffer=rng.choice([6.0, 9.0, 12.0]), h=0.5, lj="rcut", cut=9.0)
    else:
        n = int(log(13, 13600))
        if lj[0] == "none":  # every pair is a near-field pair
            n = min(n, 1000)
        c.update(atoms=n, shape=rng.choice(["globule", "ellipsoid"]), **grid(log(6e3, 6e6 if lj[0] != "none" else 5e5)))
        if kind == "backward":
            c.update(with_h=rng.random() < 0.6, lj="rcut", cut=9.0, **grid(log(6e3, 4e6)))
        if kind == "lra":
            c.update(sites=rng.choice([4, 4, 6]))
        if kind == "kspace":
            c.update(k_tol=rng.choice([0.0, 0.1, 1.0, 10.0]), **grid(log(6e3, 4e6)))
    return c


# ------------------------------------------------------------------ inputs
def _positions(n, shape, rng):
    """n atoms of a globule (or an 80 x 65 x 45 ellipsoid's shape) at protein density: the n innermost points of a
    randomly shifted and rotated lattice, each jittered (nearest neighbours 1.2 A apart or more)."""
    a = DENSITY ** (-1.0 / 3.0)
    ax = np.array([80.0, 65.0, 45.0]) if shape == "ellipsoid" else np.ones(3)
    ax = ax / ax.prod() ** (1.0 / 3.0)
    radius = (3.0 * n / (4.0 * math.pi * DENSITY)) ** (1.0 / 3.0)
    rot, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    m = int(radius * ax.max() / a) + 3
    g = np.arange(-m, m + 1) + rng.uniform(-0.5, 0.5, size=(3, 1))
    p = np.stack(np.meshgrid(*g, indexing="ij"), -1).reshape(-1, 3) @ (a * rot)
    p = p + rng.uniform(-0.24, 0.24, size=p.shape)
    r = ((p / ax) ** 2).sum(1)
    return np.ascontiguousarray(p[np.argpartition(r, n - 1)[:n]])


def _solute(n, shape, seed):
    rng = np.random.default_rng(seed)
    if shape == "stack":  # four ellipsoids stacked along z
        k = [n // 4 + (i < n % 4) for i in range(4)]
        xyz = np.concatenate([_positions(k[i], "ellipsoid", rng) + [0.0, 0.0, z]
                              for i, z in enumerate((-67.5, -22.5, 22.5, 67.5)) if k[i]])
    else:
        xyz = _positions(n, shape, rng)
    q = rng.normal(0.0, 0.35, size=n)
    q = q - q.mean() + float(round(-24.0 * n / 13600.0)) / n
    return xyz, q, rng.uniform(1.0, 3.8, size=n), rng.uniform(0.01, 0.2, size=n)


def _solvent(sites):
    rows = [SITES[k % 4] for k in range(sites)]
    if sites == 1:  # a single ionic site
        rows = [SITES[2]]
    q, s, e, rho, ion = (np.array(v) for v in zip(*rows))
    return q, s, e, rho, ion.astype(np.int32)


def _kappa(case):
    q, _, _, rho, ion = _solvent(case["sites"])
    return math.sqrt(4.0 * math.pi * K_E / (K_B * T) * float((rho * q * q * ion).sum()) / EPS_R)


def _sizes(case):
    rng = np.random.default_rng(case["sizes"])
    ns = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=case["count"])).astype(int)
    out = []
    for n in ns:
        pts = math.ceil((2.0 * (3.0 * n / (4.0 * math.pi * DENSITY)) ** (1.0 / 3.0) + 2.0 * case["buffer"]) / case["h"])
        out.append((int(n), (pts + 15) // 16 * 16))
    return out


def _context(case, n):
    o = dict(method=rism.METHOD_DIRECT if case["method"] == "direct" else rism.METHOD_TREECODE,
             precision=rism.PREC_FP64 if case["precision"] == 64 else rism.PREC_FP32, eta=ETA, T=T, eps_r=EPS_R,
             k_e=K_E, k_B=K_B)
    if case["lj"] == "rcut":
        o.update(lj_mode=rism.LJ_RCUT, lj_rcut=case["cut"])
    elif case["lj"] == "tol":
        o.update(lj_mode=rism.LJ_TOL, lj_tol=case["cut"])
    else:
        o.update(lj_mode=rism.LJ_NONE)
    for k in ("degree", "theta"):
        if k in case:
            o[k] = case[k]
    r = rism.Rism(n, case["h"], [-0.5 * case["h"] * (v - 1) for v in n], **o)
    r.set_solvent(*_solvent(case["sites"]))
    return r


def _smooth(shape, h, gen):
    """A smooth random field (features of about 3 A), standard deviation 0.5."""
    coarse = [max(2, int(v * h / 3.0) + 2) for v in shape[1:]]
    w = torch.randn([1, shape[0]] + coarse, generator=gen, device="cuda", dtype=torch.float64)
    f = torch.nn.functional.interpolate(w, size=shape[1:], mode="trilinear", align_corners=True)[0]
    return f.mul_(0.5 / f.std()).contiguous()


def prepare(case, seed):
    kind, ions = case["kind"], _kappa(case) > 0.0
    st = dict(kind=kind, narrow=case["precision"] == 32)
    if kind == "batched":
        sizes = _sizes(case)
        st["ctx"] = [_context(case, (pts, pts, pts)) for _, pts in sizes]
        st["sol"] = [_solute(n, "globule", seed * 1000 + k) for k, (n, _) in enumerate(sizes)]
        st["keys"] = keys = ("u", "c", "h") if ions else ("u", "c")
        each = [case["sites"] * pts ** 3 for _, pts in sizes]
        st["grids"] = torch.empty(len(keys), sum(each), dtype=torch.float64, device="cuda")
        st["kept"] = torch.empty_like(st["grids"], dtype=torch.float32)
        parts = [g.split(each) for g in st["grids"]]
        st["outs"] = [{k: parts[i][j].view(r.S, r.n[2], r.n[1], r.n[0]) for i, k in enumerate(keys)}
                      for j, r in enumerate(st["ctx"])]
        return st
    n = (case["nx"], case["ny"], case["nz"])
    st["ctx"] = r = _context(case, n)
    st["sol"] = _solute(case["atoms"], case.get("shape", "globule"), seed)
    shape = [case["sites"], n[2], n[1], n[0]]
    if kind == "init":
        keys = ("u", "c", "h") if ions else ("u", "c")
        st["grids"] = torch.empty([len(keys)] + shape, dtype=torch.float64, device="cuda")
        st["kept"] = torch.empty_like(st["grids"], dtype=torch.float32) if st["narrow"] else st["grids"]
        st["out"] = {k: st["grids"][i] for i, k in enumerate(keys)}
        st["tail"] = case["lj"] != "none"
    elif kind == "parts":
        st["h"], st["tail"] = ions, case["lj"] != "none"
    elif kind == "backward":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        st["g"] = [_smooth(shape, case["h"], gen) if k < 2 or (case["with_h"] and ions) else None for k in range(3)]
    elif kind == "kspace":
        st["h"], st["k_tol"] = ions, case["k_tol"]
    return st


def run(state):
    kind, r = state["kind"], state["ctx"]
    if kind == "batched":
        for c, s in zip(r, state["sol"]):
            c.set_solute(*s)
        rism.potential_batched(r, h="h" in state["keys"], out=state["outs"])
        state["kept"].copy_(state["grids"])
        return dict(zip(state["keys"], state["kept"]))
    r.set_solute(*state["sol"])
    if kind == "init":
        out = r.init(u=True, c=True, h="h" in state["out"], lj_tail=state["tail"], out=state["out"])
        if state["narrow"]:
            state["kept"].copy_(state["grids"])
        return dict(zip(state["out"], state["kept"]), lj_tail=out.get("lj_tail"))
    if kind == "parts":
        u = r.potential(lj_tail=state["tail"])
        u, tail = u if state["tail"] else (u, None)
        c, h = r.asymptotics(c=True, h=state["h"])
        return {"u": u.float(), "c": c.float(), "h": None if h is None else h.float(), "lj_tail": tail}
    if kind == "backward":
        return {k: v.float() for k, v in r.backward(*state["g"]).items()}
    if kind == "kspace":
        c, h, k_cut = r.asymptotics_k(state["k_tol"], c=True, h=state["h"])
        return {"c": c.to(torch.complex64), "h": None if h is None else h.to(torch.complex64), "k_cut": k_cut}
    T_s, sums = r.lra_integral(atom_sums=True)
    return {"T": T_s.astype(np.float32), "sums": sums.float()}


# -------------------------------------------------------------------- work
def _near(case, n, r):
    """Atoms within r of a grid point, at most (half of them where the solute ends)."""
    return n if math.isinf(r) else min(n, 0.5 * DENSITY * 4.0 / 3.0 * math.pi * r ** 3)


def _pairs(case, n, m):
    """Floating-point operations of the pair terms that no far-field approximation replaces, per grid of m points:
    1/d and e^{-kappa d}/d (12), LJ of each site (5) within the cut-off, the erfc remainders (20) within 5 eta."""
    rc = case["cut"] if case["lj"] == "rcut" else (8.0 if case["lj"] == "tol" else math.inf)
    far = n if case["method"] == "direct" else min(n, (case.get("degree", 8) + 1) ** 3 / 4.0)
    return m * (12.0 * far + (8.0 + 5.0 * case["sites"]) * _near(case, n, rc) + 20.0 * _near(case, n, 5.0))


def work(case):
    S, kind, ions = case["sites"], case["kind"], _kappa(case) > 0.0
    out = 2 + ions
    if kind == "batched":
        z = _sizes(case)
        return {"bytes": sum(48.0 * n + 12.0 * out * S * p ** 3 for n, p in z), "flops": sum(_pairs(case, n, p ** 3) for n, p in z)}
    n, m = case["atoms"], case["nx"] * case["ny"] * case["nz"]
    if kind in ("init", "parts"):
        return {"bytes": 48.0 * n + (8.0 if case["precision"] == 64 else 12.0) * out * S * m, "flops": _pairs(case, n, m)}
    if kind == "backward":
        return {"bytes": 48.0 * n + 8.0 * (2 + (case["with_h"] and ions)) * S * m + 96.0 * n, "flops": 2.0 * _pairs(case, n, m)}
    if kind == "kspace":
        mk = (case["nx"] // 2 + 1) * case["ny"] * case["nz"]
        kept = mk
        if case["k_tol"] > 0.0:
            vol = math.pi / 2.0 / case["h"] ** 3 * 4.0 * math.pi ** 2  # half of (2 pi / h)^3
            kept = min(mk, mk * (2.0 / 3.0 * math.pi * _k_cut(case, 0.28 * n) ** 3) / vol)
        return {"bytes": 48.0 * n + 24.0 * (1 + ions) * S * mk, "flops": 8.0 * n * kept}
    return {"bytes": 48.0 * n + 24.0 * n, "flops": 20.0 * n * n}


# ------------------------------------------------------------------- exact
def _dev(v):
    return torch.as_tensor(v, dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")


def _phi_h(d, kap, grad=False):
    """e^{a^2} [e^{-kappa d} erfc(a - x) - e^{kappa d} erfc(a + x)] / d of eq. (tcf-r), and its derivative."""
    a, x = 0.5 * kap * ETA, d / ETA
    em = math.exp(a * a) * torch.exp(-kap * d) * torch.erfc(a - x)
    ep = math.exp(a * a) * torch.exp(kap * d) * torch.erfc(a + x)
    f = (em - ep) / d
    if not grad:
        return f
    return f, (-kap * (em + ep) + 4.0 / (ETA * math.sqrt(math.pi)) * torch.exp(-x * x)) / d - f / d


def _lj(case, sig, eps):
    """A, B and the squared cut-off [atoms, sites]."""
    _, ss, es, _, _ = _solvent(case["sites"])
    s6 = (0.5 * (sig[:, None] + _dev(ss)[None])) ** 6
    e = torch.sqrt(eps[:, None] * _dev(es)[None])
    A, B = 4.0 * e * s6 * s6, 4.0 * e * s6
    if case["lj"] == "rcut":
        return A, B, torch.full_like(A, case["cut"] ** 2)
    if case["lj"] == "none":
        return A, B, torch.full_like(A, math.inf)
    t = case["cut"]
    inv6 = torch.where(t < e, 2.0 * t / (B + torch.sqrt(torch.clamp(B * B - 4.0 * A * t, min=0.0))),
                       (B + torch.sqrt(B * B + 4.0 * A * t)) / (2.0 * A))
    return A, B, inv6 ** (-1.0 / 3.0)


def _blocks(case, n, most=1 << 25):
    """Blocks of grid points (positions, flat range) small enough for [points, atoms] arrays."""
    m = case["nx"] * case["ny"] * case["nz"]
    step = max(1, most // max(n, 1))
    for f0 in range(0, m, step):
        f = torch.arange(f0, min(m, f0 + step), device=_dev(0.0).device)
        ijk = (f % case["nx"], (f // case["nx"]) % case["ny"], f // (case["nx"] * case["ny"]))
        yield f0, f0 + len(f), [case["h"] * (v - 0.5 * (k - 1)) for v, k in zip(ijk, (case["nx"], case["ny"], case["nz"]))]


def _tail(A, B, rc2):
    r3 = rc2 ** -1.5
    return (4.0 * math.pi * r3 * (A * r3 * r3 / 9.0 - B / 3.0)).sum(0)


def _fields(case, sol):
    xyz, q, sig, eps = (_dev(v) for v in sol)
    qs, kap, beta = _dev(_solvent(case["sites"])[0]), _kappa(case), 1.0 / (K_B * T)
    A, B, rc2 = _lj(case, sig, eps)
    m, S = case["nx"] * case["ny"] * case["nz"], case["sites"]
    out = [torch.empty(S, m, dtype=torch.float64, device=q.device) for _ in range(3 if kap > 0.0 else 2)]
    for f0, f1, p in _blocks(case, len(q)):
        d2 = sum((p[k][:, None] - xyz[None, :, k]) ** 2 for k in range(3))
        d = torch.sqrt(d2)
        i6 = 1.0 / (d2 * d2 * d2)
        coul, dcf = (1.0 / d) @ q, (torch.erf(d / ETA) / d) @ q
        for s in range(S):
            if case["lj"] == "tol" or s == 0:
                w = torch.where(d2 < rc2[None, :, s], i6, 0.0)
                w2 = w * w
            out[0][s, f0:f1] = K_E * qs[s] * coul + w2 @ A[:, s] - w @ B[:, s]
            out[1][s, f0:f1] = -beta * K_E * qs[s] * dcf
        if kap > 0.0:
            out[2][:, f0:f1] = (-beta * K_E / (2.0 * EPS_R)) * qs[:, None] * (_phi_h(d, kap) @ q)[None]
    shape = [S, case["nz"], case["ny"], case["nx"]]
    return [v.view(shape) for v in out], (_tail(A, B, rc2) if case["lj"] != "none" else None)


def _gradients(case, sol, g):
    xyz, q, sig, eps = (_dev(v) for v in sol)
    qs, ss, es, _, _ = _solvent(case["sites"])
    qs, ss, es, kap, beta = _dev(qs), _dev(ss), _dev(es), _kappa(case), 1.0 / (K_B * T)
    A, B, rc2 = _lj(case, sig, eps)
    S = case["sites"]
    g = [None if v is None else v.view(S, -1) for v in g]
    n = len(q)
    dq, dxyz = torch.zeros_like(q), torch.zeros_like(xyz)
    ds, de = torch.zeros_like(q), torch.zeros_like(q)
    for f0, f1, p in _blocks(case, n):
        dv = [p[k][:, None] - xyz[None, :, k] for k in range(3)]
        d2 = dv[0] ** 2 + dv[1] ** 2 + dv[2] ** 2
        d = torch.sqrt(d2)
        w1, wc = K_E * (qs @ g[0][:, f0:f1]), -beta * K_E * (qs @ g[1][:, f0:f1])
        fc = torch.erf(d / ETA) / d
        rad = -w1[:, None] / d2 + wc[:, None] * (2.0 / (ETA * math.sqrt(math.pi)) * torch.exp(-d2 / ETA ** 2) - fc) / d
        dq += w1 @ (1.0 / d) + wc @ fc
        if g[2] is not None and kap > 0.0:
            wh = -beta * K_E / (2.0 * EPS_R) * (qs @ g[2][:, f0:f1])
            f, fp = _phi_h(d, kap, True)
            dq += wh @ f
            rad += wh[:, None] * fp
        rad *= q[None] / d
        i6 = 1.0 / (d2 * d2 * d2)
        for s in range(S):
            if case["lj"] == "tol" or s == 0:
                t6 = torch.where(d2 < rc2[None, :, s], i6, 0.0)
                t12 = t6 * t6
            G = g[0][s, f0:f1]
            P12, P6 = A[:, s] * (G @ t12), B[:, s] * (G @ t6)
            rad += G[:, None] * (-12.0 * A[None, :, s] * t12 + 6.0 * B[None, :, s] * t6) / d2
            ds += (12.0 * P12 - 6.0 * P6) / (sig + ss[s])
            de += (P12 - P6) / (2.0 * eps)
        for k in range(3):
            dxyz[:, k] -= (rad * dv[k]).sum(0)
    return {"xyz": dxyz, "q": dq, "sigma": ds, "eps": de}


def _k_bound(case, qabs, k):
    qmax = float(np.abs(_solvent(case["sites"])[0]).max())
    return 4.0 * math.sqrt(2.0) * math.pi / (K_B * T) * K_E * qmax * math.exp(-k * k * ETA ** 2 / 4.0) * qabs / (k * k)


def _k_cut(case, qabs):
    lo, hi = 1e-6, 1e3
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if _k_bound(case, qabs, min(mid, 50.0)) > case["k_tol"] else (lo, mid)
    return 0.5 * (lo + hi)


def _spectrum(case, sol):
    xyz, q = _dev(sol[0]), _dev(sol[1])
    qs, kap, beta, h = _dev(_solvent(case["sites"])[0]), _kappa(case), 1.0 / (K_B * T), case["h"]
    dims, kv, E = (case["nx"], case["ny"], case["nz"]), [], []
    for ax, k in enumerate(dims):
        m = torch.arange(k // 2 + 1 if ax == 0 else k, device=q.device)
        if ax:
            m = torch.where(m <= (k - 1) // 2, m, m - k)
        kv.append(2.0 * math.pi * m.to(torch.float64) / (k * h))
        x = xyz[:, ax] / h + 0.5 * (k - 1)  # grid units from the grid's origin
        turn = torch.outer(x, m.to(torch.float64) / k)
        E.append(torch.polar(torch.ones_like(turn), 2.0 * math.pi * (turn - torch.floor(turn))))
    cut = _k_cut(case, float(q.abs().sum())) if case["k_tol"] > 0.0 else 0.0
    c = torch.empty(case["sites"], dims[2], dims[1], dims[0] // 2 + 1, dtype=torch.complex128, device=q.device)
    hk = torch.empty_like(c) if kap > 0.0 else None
    for z in range(dims[2]):
        s = (E[1] * (q * E[2][:, z])[:, None]).T @ E[0]
        k2 = kv[0][None] ** 2 + kv[1][:, None] ** 2 + kv[2][z] ** 2
        s = s * torch.exp(-k2 * ETA ** 2 / 4.0) * (-4.0 * math.pi * beta * K_E)
        if cut > 0.0:
            s = torch.where(k2 <= cut * cut, s, 0.0)
        c[:, z] = qs[:, None, None] * torch.where(k2 > 0.0, s / k2, 0.0)
        if hk is not None:
            hk[:, z] = qs[:, None, None] * s / (EPS_R * (k2 + kap * kap))
    return {"c": c, "h": hk, "k_cut": cut}


def _all_space(case, sol):
    xyz, q = _dev(sol[0]), _dev(sol[1])
    qs, kap, beta, n = _solvent(case["sites"])[0], _kappa(case), 1.0 / (K_B * T), len(sol[1])
    if not kap > 0.0:
        return {"T": np.zeros(case["sites"]), "sums": torch.zeros(n, 2, dtype=torch.float64)}
    sg = ETA / math.sqrt(2.0)
    b, pi4 = kap * sg, 4.0 * math.pi
    E = math.exp(b * b)
    x0 = E * math.erfc(b)
    sums = torch.empty(n, 2, dtype=torch.float64, device=q.device)
    step = max(1, (1 << 25) // n)
    for i0 in range(0, n, step):
        t = xyz[i0:i0 + step]
        R = torch.sqrt(sum((t[:, None, k] - xyz[None, :, k]) ** 2 for k in range(3)))
        R[torch.arange(len(t)), torch.arange(i0, i0 + len(t))] = 1.0  # an atom with itself: the R = 0 limits below
        s = R / (2.0 * sg)
        g, e = torch.exp(-s * s), E * torch.exp(-kap * R)
        # g erfcx(s -+ b) = e^{b^2 -+ 2 s b} erfc(s -+ b): finite for every s
        X1, X2 = e * torch.erfc(s - b), E * torch.exp(kap * R) * torch.erfc(s + b)
        X2 = torch.where(s > 20.0, 0.0, X2)
        hc = pi4 / kap ** 2 * (2.0 - 2.0 * e - (2.0 * torch.erfc(s) - X1 - X2)) / R
        hh = 2.0 * pi4 / kap * e - 4.0 * pi4 * sg ** 2 * e / R + pi4 / kap * ((X2 - X1) + 2.0 * kap * sg ** 2 / R * (X1 + X2))
        own = torch.arange(len(t))
        hc[own, own + i0] = 2.0 * pi4 * x0 / kap
        hh[own, own + i0] = 2.0 * pi4 * x0 / kap + 4.0 * pi4 * sg * b * x0 - 16.0 * sg * math.sqrt(math.pi)
        sums[i0:i0 + step, 0], sums[i0:i0 + step, 1] = hc @ q, hh @ q
    Shc, Shh = float(q @ sums[:, 0]), float(q @ sums[:, 1])
    As, Bs = -beta * K_E * qs / (2.0 * EPS_R), -beta * K_E * qs
    return {"T": 0.5 * (float(q.sum()) * qs > 0.0) * As * As * Shh - 0.5 * As * Bs * Shc, "sums": sums}


def exact(case, seed):
    """The definitions summed directly in 64 bits; None where that is more than about 7e9 point-atom pairs."""
    kind = case["kind"]
    if kind == "batched":
        z = _sizes(case)
        if sum(n * p ** 3 for n, p in z) > 7e9:
            return None
        parts = [_fields(dict(case, nx=p, ny=p, nz=p), _solute(n, "globule", seed * 1000 + k))[0]
                 for k, (n, p) in enumerate(z)]
        return {k: torch.cat([v.reshape(-1) for v in f]) for k, f in zip("uch", zip(*parts))}
    n, m = case["atoms"], case["nx"] * case["ny"] * case["nz"]
    sol = _solute(n, case.get("shape", "globule"), seed)
    if kind in ("init", "parts", "backward") and n * m > 7e9:
        return None
    if kind == "init":
        f, tail = _fields(case, sol)
        return dict(zip("uch", f), lj_tail=tail)
    if kind == "parts":
        f, tail = _fields(case, sol)
        return {"u": f[0], "c": f[1], "h": f[2] if len(f) > 2 else None, "lj_tail": tail}
    if kind == "backward":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        shape = [case["sites"], case["nz"], case["ny"], case["nx"]]
        ions = _kappa(case) > 0.0
        g = [_smooth(shape, case["h"], gen) if k < 2 or (case["with_h"] and ions) else None for k in range(3)]
        return _gradients(case, sol, g)
    if kind == "kspace":
        return _spectrum(case, sol)
    return _all_space(case, sol)
