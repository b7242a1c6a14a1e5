"""The work whose speed is watched: calls of the library's public entry points at the sizes,
functionals and precisions that its users run.

A case is a dict of plain values; `op` says which entry point a pass goes through:
  eval   Grid.energy_potential: one energy and potential of a density (the inner call of every
         density optimisation)
  batch  energy_potential_batched over snapshots of uneven grid sizes, with forces
  step   OFDFTEnergy forward and backward: one geometry step (new ions, E, V and forces)
  td     Grid.td_propagate: real-time steps of a kicked cluster
  opt    Grid.optimize_density: a few iterations of the density optimiser
Systems are FCC Al (a = 7.65 bohr, Z = 3, r_c = 0.8) with jittered ions and a Gaussian model
density with multiplicative noise; `td` runs an isolated Mg-like cluster.  `exact` is a plain
torch FP64 statement of the same functional.
"""
import math

import numpy as np
import torch

import paper_2002_02985_gb300 as ofd
from paper_2002_02985_gb300 import _lib as L

A_AL = 7.65
FCC = ((0.0, 0.0, 0.0), (0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))
KEYS = ("total", "TF", "vW", "NL", "H", "PP", "XC")


def _case(op, n, **kw):
    c = dict(op=op, n0=n[0], n1=n[1], n2=n[2], pts=20, tile=1, tilt=0.0, knots=16, fp64=False, xc=False,
             interp=False, mgp=False)
    c.update(kw)
    return c


def listed():
    return [
        # a unit cell: one evaluation of a small periodic cell, where launches and latency count
        dict(_case("eval", (32, 32, 32), knots=10, ), name="cell-32"),
        # the ordinary bulk evaluation: 256 atoms on 128^3, the headline benchmark's size
        dict(_case("eval", (128, 128, 128)), name="bulk-128"),
        # the same evaluation in full FP64, the plain path that results are checked with
        dict(_case("eval", (128, 128, 128), fp64=True), name="bulk-128-fp64"),
        # a finer grid with the knots of a wide density range and LDA exchange-correlation
        dict(_case("eval", (192, 192, 192), knots=30, xc=True), name="bulk-192-xc"),
        # a sheared cell whose three grid lengths differ, with the interpolated potential
        dict(_case("eval", (90, 100, 108), tilt=0.15, interp=True), name="sheared-interp"),
        # odd lengths on every axis, LMGP kernels
        dict(_case("eval", (75, 81, 125), knots=12, mgp=True), name="odd-mgp"),
        # a large supercell with the direct structure factor
        dict(_case("eval", (256, 256, 256)), name="bulk-256"),
        # the scale of the large-system runs: 131,072 atoms, PME structure factor, 16 points per cell edge
        dict(_case("eval", (512, 512, 512), pts=16, tile=8, knots=12), name="pme-512"),
        # snapshots of 108-atom cells on grids of four sizes, with forces (training-set labelling)
        dict(_case("batch", (64, 80, 120), snaps=16), name="snapshots-16"),
        # one relaxation or dynamics step of a 108-atom cell through autograd
        dict(_case("step", (96, 96, 96)), name="geometry-96"),
        # real-time propagation of an isolated 55-atom cluster after a kick
        dict(_case("td", (128, 128, 128), xc=True, steps=2), name="td-128"),
        # the start of a density optimisation in FP64 on a unit cell: many small dependent calls
        dict(_case("opt", (32, 32, 32), knots=10, fp64=True, iters=4), name="optimise-32-fp64"),
    ]


def _smooth(lo, hi):
    return [n for n in range(lo, hi + 1) if not [p for p in (7, 11, 13, 17, 19, 23) if n % p == 0] and _is235(n)]


def _is235(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


def draw(rng):
    """A case of the listed ranges: 24 to 320 points per axis (lengths 2^a 3^b 5^c, odd ones too)."""
    op = rng.choice(["eval"] * 7 + ["batch", "step", "td", "opt"])
    top = {"eval": 320, "batch": 120, "step": 128, "td": 150, "opt": 48}[op]
    base = math.exp(rng.uniform(math.log(24), math.log(top)))
    near = [n for n in _smooth(20, top) if 0.75 * base <= n <= 1.3 * base] or [32]
    n = [rng.choice(near) for _ in range(3)]
    knots = rng.randint(6, 24)
    if op == "batch":
        return _case(op, (rng.choice(near), rng.choice(near), rng.choice(near)), snaps=rng.randint(4, 12))
    if op == "td":
        n = [max(n)] * 3
        return _case(op, n, knots=min(knots, 16), xc=rng.random() < 0.5, steps=1)
    if op == "opt":
        return _case(op, n, knots=min(knots, 12), fp64=True, iters=rng.randint(2, 4))
    if op == "step":
        return _case(op, n, knots=knots, xc=rng.random() < 0.3)
    fp64 = max(n) <= 128 and rng.random() < 0.15
    tile = 1
    if not fp64 and rng.random() < 0.2:
        n = [2 * (x // 2) if _is235(2 * (x // 2)) else 96 for x in n]
        tile = 2
    return _case(op, n, knots=knots, fp64=fp64, tile=tile, pts=16 if tile > 1 else 20,
                 tilt=rng.choice([0.0, 0.0, 0.12]) if tile == 1 else 0.0, xc=rng.random() < 0.3,
                 interp=rng.random() < 0.25, mgp=rng.random() < 0.2)


# ------------------------------------------------------------------ inputs
def _cells(case, n):
    return [max(1, round(x / case["tile"] / case["pts"])) for x in n]


def _geometry(case, n, rng):
    """Lattice vectors (rows), ion positions, and the block of ions that is repeated tile^3 times."""
    t = case["tile"]
    nc = _cells(case, n)
    if case["op"] == "td":
        side = 40.0
        r = np.array([[i, j, k] for i in range(-4, 5) for j in range(-4, 5) for k in range(-4, 5)
                      if (i + j + k) % 2 == 0 and i * i + j * j + k * k <= 8], dtype=float)     # 55 sites
        pos = 0.5 * side + r * (5.5 / math.sqrt(2.0)) + rng.normal(0.0, 0.1, r.shape)
        return np.diag([side] * 3), pos, np.diag([side] * 3), pos
    block = np.diag(np.array(nc) * A_AL)
    block[1, 0] = case["tilt"] * block[0, 0]
    block[2, 1] = -case["tilt"] * block[1, 1]
    ijk = np.stack(np.meshgrid(*[np.arange(c) for c in nc], indexing="ij"), -1).reshape(-1, 1, 3)
    frac = ((ijk + np.array(FCC)) / np.array(nc)).reshape(-1, 3)
    bpos = frac @ block + rng.normal(0.0, 0.2, (len(frac), 3))
    if t == 1:
        return block, bpos, block, bpos
    shift = np.stack(np.meshgrid(*[np.arange(t)] * 3, indexing="ij"), -1).reshape(-1, 1, 3) @ block
    return block * t, (shift + bpos).reshape(-1, 3), block, bpos


def _phases(frac, n, half):
    m = np.arange(n // 2 + 1) if half else np.where(np.arange(n) <= n // 2, np.arange(n), np.arange(n) - n)
    a = torch.from_numpy(np.outer(frac, m)).cuda() * (-2.0 * math.pi)
    return torch.complex(torch.cos(a), torch.sin(a))


def _structure_factor(cell, pos, n):
    """sum_I e^{-iG.R_I} on the half spectrum, FP64."""
    f = pos @ np.linalg.inv(cell)
    p0, p1, p2 = (_phases(f[:, a], n[a], a == 2) for a in range(3))
    out = torch.empty((n[0], n[1], n[2] // 2 + 1), dtype=torch.complex128, device="cuda")
    for k in range(n[0]):
        out[k] = (p0[:, k, None] * p1).T @ p2
    return out


def _gvectors(cell, n):
    b = 2.0 * math.pi * np.linalg.inv(cell).T
    m = [torch.from_numpy(np.where(np.arange(x) <= x // 2, np.arange(x), np.arange(x) - x).astype(float)).cuda()
         for x in n]
    m[2] = torch.arange(n[2] // 2 + 1, dtype=torch.float64, device="cuda")
    g = [m[0][:, None, None] * b[0, d] + m[1][None, :, None] * b[1, d] + m[2][None, None, :] * b[2, d]
         for d in range(3)]
    return g


def _species(case):
    return (2.0, 1.0, 1.4) if case["op"] == "td" else (3.0, 0.8, 1.0)     # Z, r_c, width of the model density


def _density(case, n, block, bpos, seed):
    """The sum of normalised Gaussians on the ions (band-limited sum), noise, and the electron count."""
    Z, _, sigma = _species(case)
    t = case["tile"]
    nb = [x // t for x in n]
    g = _gvectors(block, nb)
    S = _structure_factor(block, bpos, nb)
    om = abs(np.linalg.det(block))
    rho = torch.fft.irfftn(S * (Z / om) * torch.exp(-0.5 * sigma * sigma * (g[0] ** 2 + g[1] ** 2 + g[2] ** 2)),
                           s=nb, dim=(0, 1, 2), norm="forward")
    rho = rho.clamp_min(1e-8 if case["op"] == "td" else 1e-4)
    dt = torch.float64 if case["fp64"] else torch.float32
    rho = rho.to(dt).repeat(t, t, t)
    if case["op"] != "td":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        rho *= 1.0 + 0.02 * (2.0 * torch.rand(rho.shape, generator=gen, device="cuda", dtype=dt) - 1.0)
    ne = Z * len(bpos) * t ** 3
    rho *= ne / (float(rho.sum(dtype=torch.float64)) * om * t ** 3 / rho.numel())
    return rho.contiguous(), ne


def _sizes(case):
    n = (case["n0"], case["n1"], case["n2"])
    if case["op"] != "batch":
        return [n]
    # snapshots on cubic grids of four sizes, as a mixed labelling set has them
    s = sorted(set(n))
    s.append(s[-1] if len(s) > 3 else _smooth(s[0], s[-1])[len(_smooth(s[0], s[-1])) // 2])
    return [(s[i % len(s)],) * 3 for i in range(case["snaps"])]


def _functional(case):
    terms = L.TERMS_ALL | (L.TERM_XC if case["xc"] else 0)
    if case["op"] == "td":
        terms &= ~L.TERM_NL            # spectra are taken with the semilocal functional
    return ofd.Functional(terms=terms, n_knots=case["knots"], precision=L.FP64 if case["fp64"] else L.FP32_MIXED,
                          nl_potential=L.NLPOT_INTERP if case["interp"] else L.NLPOT_EXACT,
                          **(ofd.MGP if case["mgp"] else {}))


def _inputs(case, seed):
    out = []
    for i, n in enumerate(_sizes(case)):
        rng = np.random.default_rng([seed, i])
        cell, pos, block, bpos = _geometry(case, n, rng)
        rho, ne = _density(case, n, block, bpos, seed * 64 + i)
        out.append(dict(n=n, cell=cell, pos=pos, block=block, bpos=bpos, rho=rho, ne=ne))
    return out


def prepare(case, seed):
    sys_ = _inputs(case, seed)
    Z, rc, _ = _species(case)
    st = dict(case=case, func=_functional(case), sys=sys_, grids=[])
    for s in sys_:
        g = ofd.Grid(s["cell"], s["n"])
        spec = (np.zeros(len(s["pos"]), dtype=np.int32), [Z], [rc])
        if case["op"] != "step":
            g.set_ions(s["pos"], *spec, pme_order=10 if case["tile"] > 1 else 0)
        st["grids"].append(g)
        s["spec"] = spec
    s = sys_[0]
    if case["op"] == "batch":
        st["rhos"] = [x["rho"] for x in sys_]
        st["V"] = [torch.empty_like(x) for x in st["rhos"]]
    elif case["op"] == "step":
        st["rho"] = s["rho"].clone().requires_grad_(True)
        st["R"] = torch.from_numpy(s["pos"]).requires_grad_(True)
    elif case["op"] == "td":
        st["psi"] = s["rho"].sqrt()
    elif case["op"] == "opt":
        st["psi"] = s["rho"].sqrt()
    return st


def _e(E, dtype):
    return np.array([E[k] for k in KEYS], dtype=dtype)


def run(st):
    case, f, g, s = st["case"], st["func"], st["grids"][0], st["sys"][0]
    dt = np.float64 if case["fp64"] else np.float32
    if case["op"] == "eval":
        E, V = g.energy_potential(s["rho"], f)
        return {"E": _e(E, dt), "V": V}
    if case["op"] == "batch":
        E, V, F = ofd.energy_potential_batched(st["grids"], st["rhos"], f, want_forces=True, V_out=st["V"])
        return {"E": E.astype(dt), "V": V, "F": np.concatenate(F).astype(dt)}
    if case["op"] == "step":
        st["rho"].grad = st["R"].grad = None
        E = ofd.OFDFTEnergy.apply(st["rho"], st["R"], g, f, s["spec"])
        E.backward()
        return {"E": E.detach().to(torch.float32), "dE_drho": st["rho"].grad,
                "dE_dR": st["R"].grad.to(torch.float32)}
    if case["op"] == "td":
        re, im = st["psi"].clone(), torch.zeros_like(st["psi"])
        g.td_kick(re, im, (0.1, 0.0, 0.0))
        mu, _ = g.td_propagate(re, im, s["rho"], f, 0.1, case["steps"], solver_tol=1e-7,
                               raise_on_not_converged=False)
        return {"re": re, "im": im, "dipole_x": mu[1:, 0].astype(dt)}
    psi = st["psi"].clone()
    rep = g.optimize_density(psi, f, s["ne"], tol_per_atom=1e-14, max_iter=case["iters"])
    return {"E": _e(rep["energies"], dt), "psi": psi}


# ------------------------------------------------------------------ work
def _eval_work(case, n):
    N = n[0] * n[1] * n[2]
    NH = n[0] * n[1] * (n[2] // 2 + 1)
    M = case["knots"] if case["op"] != "td" else 0
    # real transforms: density, psi, rho^beta (and the knot fields unless interpolated) forward; the
    # Hartree + ions, vW and knot fields (and the exact potential's second term) back
    nf, ni = (2, 2) if not M else (3, 2 + M) if case["interp"] else (3 + M, 3 + M)
    b = 8 if case["fp64"] else 4
    return 2.0 * b * N, (nf + ni) * 2.5 * N * math.log2(N) + 24.0 * M * NH + 60.0 * N


def work(case):
    b = f = 0.0
    for n in _sizes(case):
        eb, ef = _eval_work(case, n)
        ions = 4 * case["tile"] ** 3 * np.prod(_cells(case, n))
        if case["op"] in ("batch", "step"):
            ef += 8.0 * ions * n[0] * n[1] * (n[2] // 2 + 1)      # forces: one complex product per ion and G
        if case["op"] == "step":
            ef += 8.0 * ions * n[0] * n[1] * (n[2] // 2 + 1)      # and the structure factor
        N = n[0] * n[1] * n[2]
        if case["op"] == "td":
            # per step two potentials and two solves of two real systems: 6 operator applications each
            eb, ef = case["steps"] * 16.0 * N, case["steps"] * (2 * ef + 48 * 2.5 * N * math.log2(N))
        if case["op"] == "opt":
            eb, ef = 16.0 * N, ef * 3.0 * case["iters"]
        b, f = b + eb, f + ef
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact values
def _rfft(x):
    return torch.fft.rfftn(x, dim=(0, 1, 2), norm="forward")


def _irfft(x, n):
    return torch.fft.irfftn(x, s=n, dim=(0, 1, 2), norm="forward")


def _series(z, c):
    p = torch.full_like(z, c[-1])
    for v in reversed(c[:-1]):
        p = p * z + v
    return p * z


def _gnl(eta):
    """G_NL = 1/F - 3 eta^2 - 1 of the Lindhard function, by series where the closed form cancels."""
    a = [1.0 / (4.0 * m * m - 1.0) for m in range(1, 42)]
    y = (eta * eta).clamp_max(0.25)
    lo = _series(y, [-8.0 / 3.0] + [a[m] + 3.0 * a[m - 1] for m in range(1, 36)]) / (1.0 - _series(y, a[:36]))
    x = 1.0 / (eta * eta).clamp_min(4.0)
    hi = -_series(x, [a[m] + 3.0 * a[m + 1] for m in range(36)]) / _series(x, a[:36])
    e = eta.clamp(0.5, 2.0)
    F = 0.5 + (1.0 - e * e) / (4.0 * e) * torch.log(((1.0 + e) / (1.0 - e)).abs())
    mid = torch.where(e == 1.0, torch.full_like(e, -2.0), 1.0 / F - 3.0 * e * e - 1.0)
    return torch.where(eta < 0.5, lo, torch.where(eta > 2.0, hi, mid))


_TABLE = {}


def _mgp_table(y, n=(1 << 18) + 1):
    """J_y(eta) = 2 int_0^1 r^(6y-1) G_NL(eta/r^2) dr at eta = u/(1-u), u uniform: Gauss-Legendre
    panels halving toward the kink at r = sqrt(eta) and toward both ends."""
    if y not in _TABLE:
        x, w = (torch.from_numpy(v).cuda() for v in np.polynomial.legendre.leggauss(8))
        u = torch.arange(1, n - 1, dtype=torch.float64, device="cuda") / (n - 1)
        eta = u / (1.0 - u)
        k = eta.sqrt().clamp_max(1.0)
        J = torch.zeros_like(eta)
        edges = [0.0] + [0.5 ** j for j in range(24, 0, -1)]
        edges = edges + [1.0 - e for e in reversed(edges[:-1])]
        for lo, hi in ((torch.zeros_like(k), k), (k, torch.ones_like(k))):
            for a, b in zip(edges[:-1], edges[1:]):
                c, h = lo + (hi - lo) * (0.5 * (a + b)), (hi - lo) * (0.5 * (b - a))
                for q in range(8):
                    r = c + h * x[q]
                    J += torch.where(h > 0.0, 2.0 * h * w[q] * r ** (6.0 * y - 1.0) * _gnl(eta / (r * r).clamp_min(1e-300)),
                                     torch.zeros_like(h))
        ends = [torch.tensor([v], dtype=torch.float64, device="cuda") for v in (0.0, -8.0 / (15.0 * y))]
        _TABLE[y] = torch.cat([ends[0], J, ends[1]])
    return _TABLE[y]


def _kernel(case, eta):
    c = 0.24 * (3.0 * math.pi ** 2) ** (2.0 / 3.0)
    if not case["mgp"]:
        return c * _gnl(eta)
    # (x, y) = (1, 5/6): the G_NL part drops out; quadratic interpolation of the table
    t = _mgp_table(5.0 / 6.0)
    p = eta / (1.0 + eta) * (len(t) - 1)
    i = p.long().clamp(1, len(t) - 2)
    d = p - i
    return c * 2.5 * (t[i] + 0.5 * d * (t[i + 1] - t[i - 1]) + 0.5 * d * d * (t[i + 1] - 2.0 * t[i] + t[i - 1]))


def _vext(case, s, g2):
    Z, rc, _ = _species(case)
    om, t, n = abs(np.linalg.det(s["cell"])), case["tile"], s["n"]
    v = torch.where(g2 > 0.0, -4.0 * math.pi * Z * torch.exp(-0.25 * rc * rc * g2) / g2.clamp_min(1e-300),
                    torch.full_like(g2, math.pi * Z * rc * rc)) / om
    if t == 1:
        return v * _structure_factor(s["cell"], s["pos"], n)
    S = torch.zeros(g2.shape, dtype=torch.complex128, device="cuda")
    # a block repeated t^3 times scatters at multiples of t; on the block's own (wider) set of integers
    nb = [2 * (x // (2 * t)) + 1 for x in n]
    sb = _structure_factor(s["block"], s["bpos"], nb)
    m = [torch.arange(-(x // (2 * t)), x // (2 * t) + 1, device="cuda") for x in n[:2]]
    m = [a[(a * t >= -((x - 1) // 2)) & (a * t <= x // 2)] for a, x in zip(m, n)]
    k2 = torch.arange(0, (n[2] // 2) // t + 1, device="cuda")
    src = sb[(m[0] % nb[0])[:, None, None], (m[1] % nb[1])[None, :, None], k2[None, None, :]]
    S[((m[0] * t) % n[0])[:, None, None], ((m[1] * t) % n[1])[None, :, None], (k2 * t)[None, None, :]] = src * t ** 3
    return v * S


def _evaluate(case, s, rho, vext, vw=True):
    """Energies (total, TF, vW, NL, H, PP, XC) and the potential of the functional, FP64."""
    n, cell = s["n"], s["cell"]
    om = abs(np.linalg.det(cell))
    dv = om / rho.numel()
    g2 = sum(x * x for x in _gvectors(cell, n))
    w = torch.full((n[2] // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    if n[2] % 2 == 0:
        w[-1] = 1.0
    E = dict.fromkeys(KEYS, 0.0)
    ctf = 0.3 * (3.0 * math.pi ** 2) ** (2.0 / 3.0)
    E["TF"] = ctf * float((rho ** (5.0 / 3.0)).sum()) * dv
    V = (5.0 / 3.0) * ctf * rho ** (2.0 / 3.0)
    if vw:
        psi = rho.sqrt()
        h = _rfft(psi)
        E["vW"] = 0.5 * om * float((w * g2 * (h.real ** 2 + h.imag ** 2)).sum())
        V += _irfft(g2 * h, n) / (2.0 * psi)
    h = _rfft(rho)
    k = torch.where(g2 > 0.0, 4.0 * math.pi / g2.clamp_min(1e-300), torch.zeros_like(g2))
    E["H"] = 0.5 * om * float((w * k * (h.real ** 2 + h.imag ** 2)).sum())
    E["PP"] = om * float((w * (h.real * vext.real + h.imag * vext.imag)).sum())
    V += _irfft(k * h + vext, n)
    if case["xc"]:
        # Dirac exchange and the Perdew-Zunger fit of the correlation energy
        c = rho ** (1.0 / 3.0)
        ex = -0.75 * (3.0 / math.pi) ** (1.0 / 3.0) * c
        rs = (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0) / c
        den = 1.0 + 1.0529 * rs.sqrt() + 0.3334 * rs
        ln = rs.log()
        ec = torch.where(rs >= 1.0, -0.1423 / den, 0.0311 * ln - 0.048 + 0.0020 * rs * ln - 0.0116 * rs)
        vc = torch.where(rs >= 1.0,
                         -0.1423 / den ** 2 * (1.0 + 7.0 / 6.0 * 1.0529 * rs.sqrt() + 4.0 / 3.0 * 0.3334 * rs),
                         0.0311 * ln - 0.048 - 0.0311 / 3.0 + 2.0 / 3.0 * 0.0020 * rs * ln
                         + (2.0 * -0.0116 - 0.0020) / 3.0 * rs)
        E["XC"] = float((rho * (ex + ec)).sum()) * dv
        V += 4.0 / 3.0 * ex + vc
    if case["op"] != "td":
        _nonlocal(case, s, rho, g2, E, V)
    E["total"] = sum(E[q] for q in KEYS[1:])
    return E, V


def _nonlocal(case, s, rho, g2, E, V):
    # knots in kF, linear spline weights
    n, M, dv = s["n"], case["knots"], abs(np.linalg.det(s["cell"])) / rho.numel()
    kf = (3.0 * math.pi ** 2 * rho) ** (1.0 / 3.0)
    k0, k1 = float(kf.min()), float(kf.max())
    knots = k0 * np.exp(np.arange(M) * (math.log(k1 / k0) / (M - 1)))
    knots[-1] = k1
    kt = torch.from_numpy(knots).cuda()
    j = (torch.searchsorted(kt, kf, right=True) - 1).clamp(0, M - 2)
    idk = 1.0 / (kt[1:] - kt[:-1])[j]
    t = (kf - kt[j]) * idk
    ra = rho ** (5.0 / 6.0)
    rb = _rfft(ra)
    g = g2.sqrt()
    phi, slope, t2 = torch.zeros_like(rho), torch.zeros_like(rho), torch.zeros_like(rb)
    for m in range(M):
        K = _kernel(case, g / (2.0 * knots[m]))
        y = _irfft(K * rb, n)
        hm = (j == m) * (1.0 - t) + (j == m - 1) * t
        phi += hm * y
        if not case["interp"]:
            slope += ((j == m - 1).double() - (j == m).double()) * idk * y
            t2 += K * _rfft(hm * ra)
        del K, y, hm
    E["NL"] = float((ra * phi).sum()) * dv
    p = rho ** (-1.0 / 6.0)
    if case["interp"]:
        V += (5.0 / 3.0) * p * phi
    else:
        V += (5.0 / 6.0) * p * (phi + _irfft(t2, n)) + p * slope * kf / 3.0


def _forces(case, s, rho):
    Z, rc, _ = _species(case)
    n = s["n"]
    g = _gvectors(s["cell"], n)
    g2 = sum(x * x for x in g)
    w = torch.full((n[2] // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1.0
    if n[2] % 2 == 0:
        w[-1] = 1.0
    c = w * torch.where(g2 > 0.0, -4.0 * math.pi * Z * torch.exp(-0.25 * rc * rc * g2) / g2.clamp_min(1e-300),
                        torch.zeros_like(g2)) * _rfft(rho).conj()
    f = s["pos"] @ np.linalg.inv(s["cell"])
    p0, p1, p2 = (_phases(f[:, a], n[a], a == 2) for a in range(3))
    F = np.zeros((len(f), 3))
    # F_I = -sum_G G w v Im[conj(rho_hat) e^{-iG.R}], the three phase factors contracted axis by axis
    for d in range(3):
        a = torch.einsum("ijk,Ik->Iij", c * g[d], p2)
        a = torch.einsum("Iij,Ij->Ii", a, p1)
        F[:, d] = -(a * p0).sum(1).imag.cpu().numpy()
    return F


def _propagate(case, s, rho, vext):
    """Crank-Nicolson with one corrector pass, (1 + tau^2 H^2) x = (1 - i tau H)^2 psi by preconditioned CG."""
    n, om, tau = s["n"], abs(np.linalg.det(s["cell"])), 0.05
    g2 = sum(x * x for x in _gvectors(s["cell"], n))
    r = [(torch.arange(m, dtype=torch.float64, device="cuda") / m - 0.5) * s["cell"][a, a] for a, m in enumerate(n)]
    x0 = r[0][:, None, None]
    psi = rho.sqrt() * torch.exp(1j * 0.1 * x0.expand(tuple(n)))

    def spec(v, f):
        return torch.complex(_irfft(f * _rfft(v.real), n), _irfft(f * _rfft(v.imag), n))

    def solve(v, psi):
        def H(u):
            return spec(u, 0.5 * g2) + v * u
        vb = float((v * psi.abs() ** 2).sum() / (psi.abs() ** 2).sum())
        pre = 1.0 / (1.0 + tau ** 2 * (0.5 * g2 + vb) ** 2)
        b = psi - 1j * tau * H(psi)
        b = b - 1j * tau * H(b)
        x = psi.clone()
        res = b - (x + tau ** 2 * H(H(x)))
        z = spec(res, pre)
        p, rz, nb = z.clone(), float((res.conj() * z).sum().real), float(b.abs().square().sum())
        for _ in range(60):
            q = p + tau ** 2 * H(H(p))
            a = rz / float((p.conj() * q).sum().real)
            x, res = x + a * p, res - a * q
            if float(res.abs().square().sum()) <= 1e-24 * nb:
                break
            z = spec(res, pre)
            new = float((res.conj() * z).sum().real)
            p, rz = z + (new / rz) * p, new
        return x

    def veff(p):
        return _evaluate(case, s, p.abs() ** 2, vext, vw=False)[1]

    v, mu = veff(psi), []
    for _ in range(case["steps"]):
        x = solve(v, psi)
        x = solve(0.5 * (v + veff(x)), psi)
        psi, v = x, veff(x)
        mu.append(float((x0 * (psi.abs() ** 2 - rho)).sum()) * om / rho.numel())
    return psi, np.array(mu)


def exact(case, seed):
    if case["op"] == "opt":
        return None                    # a fixed number of line searches has no value of its own
    E, V, F = [], [], []
    for s in _inputs(case, seed):
        rho = s["rho"].double()
        g2 = sum(x * x for x in _gvectors(s["cell"], s["n"]))
        vext = _vext(case, s, g2)
        del g2
        if case["op"] == "td":
            psi, mu = _propagate(case, s, rho, vext)
            return {"re": psi.real.contiguous(), "im": psi.imag.contiguous(), "dipole_x": mu}
        e, v = _evaluate(case, s, rho, vext)
        E.append(_e(e, np.float64))
        V.append(v)
        if case["op"] in ("batch", "step"):
            F.append(_forces(case, s, rho))
    if case["op"] == "eval":
        return {"E": E[0], "V": V[0]}
    if case["op"] == "batch":
        return {"E": np.array(E), "V": V, "F": np.concatenate(F)}
    om = abs(np.linalg.det(s["cell"]))
    return {"E": torch.tensor(E[0][0], dtype=torch.float64), "dE_drho": V[0] * (om / rho.numel()),
            "dE_dR": torch.from_numpy(-F[0])}
