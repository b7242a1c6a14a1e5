"""The any-length kernels (csrc/any.cuh, plain.cu) at the lengths where they can go wrong: two and three
passes, odd lengths, lengths with and without compiled plans, the shortest and longest of their range,
rows of a ragged last pair and column tiles that do not divide the columns.  Bounds: FP64 1e-10 relative
and 1e-9 Ha, FP32-mixed 1e-6 Ha/atom per term and 1e-4 of the potential away from the knots, as for every
other kernel; a transform there and back returns the field to 100 roundings."""
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2002_02985_gb300 as ofd  # noqa: E402
import workloads as W  # noqa: E402
from oracle import functionals as ofn  # noqa: E402
from oracle import td as otd  # noqa: E402
from oracle.evaluate import Functional as OFunc  # noqa: E402
from oracle.grid import Grid as OGrid  # noqa: E402
from paper_2002_02985_gb300 import _lib as L  # noqa: E402
from test_gpu_parity import _config_case, _n_configurations, _role_cases, knot_mask, lattice_positions, run_both  # noqa: E402

LENGTHS = (16, 18, 24, 27, 45, 75, 81, 90, 125, 162, 243, 250, 256, 270, 320, 375, 486, 512)
ROLES = {"rows": ((5, 9), L.OPTION_PICK_ROWS), "pencil": ((9, 10), L.OPTION_PICK_PENCIL),
         "recip": ((9, 12), L.OPTION_PICK_RECIP)}


def _case(role, n):
    a, b = ROLES[role][0]
    shape = {"rows": (a, b, n), "pencil": (a, n, b), "recip": (n, a, b)}[role]
    cell = np.diag([0.3 * max(m, 12) for m in shape])
    cell[1, 0] = 0.1
    counts = [max(1, round(m * 0.3 / 4.8)) if m == n else 1 for m in shape]
    pos = lattice_positions(cell, counts, n + 3)
    rho = W.renormalise(W.apply_noise(W.gaussian_density(cell, shape, pos, 3.0, 1.0) + 5e-3, 0.03, n), cell,
                        3.0 * len(pos))
    return cell, shape, pos, rho


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("role", sorted(ROLES))
def test_any_length_kernels_match_oracle(role, n):
    cell, shape, pos, rho = _case(role, n)
    kw = dict(n_knots=7)
    E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, kw, L.FP64, Z=(3.0,), rc=(0.8,))
    assert abs(E["total"] - Eo["total"]) <= 1e-10 * max(1.0, abs(Eo["total"]))
    assert np.max(np.abs(V - Vo)) <= 1e-9 * max(1.0, np.max(np.abs(Vo)))
    for pick in range(3):                      # (indices past the candidates run the first one)
        E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, kw, L.FP32_MIXED, Z=(3.0,), rc=(0.8,),
                                       options=((ROLES[role][1], pick),))
        for k in ("TF", "vW", "NL", "H", "PP", "total"):
            assert abs(E[k] - Eo[k]) / len(pos) <= 1e-6, (pick, k, E[k], Eo[k])
        m = knot_mask(rho.astype(np.float32).astype(np.float64), 7)
        assert np.linalg.norm((V - Vo)[m]) / np.linalg.norm(Vo[m]) <= 1e-4, pick


@pytest.mark.parametrize("n", (72, 128, 180, 256))
@pytest.mark.parametrize("cols", [(3, 5), (15, 8)])
def test_every_reciprocal_space_tile_width_matches_oracle(n, cols):
    """All candidates of the pass (16 and 8 columns, shared and single tiles) where the last tile is ragged."""
    shape = (n,) + cols
    cell = np.diag([0.3 * max(m, 12) for m in shape])
    pos = lattice_positions(cell, (max(1, round(n * 0.3 / 4.8)), 1, 1), n + 3)
    rho = W.renormalise(W.apply_noise(W.gaussian_density(cell, shape, pos, 3.0, 1.0) + 5e-3, 0.03, n), cell,
                        3.0 * len(pos))
    kw = dict(n_knots=7)
    for pick in range(10):                     # (indices past the candidates run the first one)
        E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, kw, L.FP32_MIXED, Z=(3.0,), rc=(0.8,),
                                       options=((L.OPTION_PICK_RECIP, pick),))
        for k in ("TF", "vW", "NL", "H", "PP", "total"):
            assert abs(E[k] - Eo[k]) / len(pos) <= 1e-6, (pick, k, E[k], Eo[k])
        m = knot_mask(rho.astype(np.float32).astype(np.float64), 7)
        assert np.linalg.norm((V - Vo)[m]) / np.linalg.norm(Vo[m]) <= 1e-4, pick


@pytest.mark.parametrize("kw", [dict(n_knots=19, nl_potential=L.NLPOT_INTERP), dict(n_knots=5, kernel=L.KERNEL_WT_GLOBAL),
                                dict(n_knots=6, mgp_x=1.0), dict(n_knots=40)])
def test_any_length_modes_match_oracle(kw):
    shape = (45, 25, 54)
    cell = np.diag([0.35 * m for m in shape])
    pos = lattice_positions(cell, (3, 2, 4), 5)
    rho = W.renormalise(W.apply_noise(W.gaussian_density(cell, shape, pos, 3.0, 1.0) + 2e-3, 0.03, 9), cell,
                        3.0 * len(pos))
    E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, kw, L.FP32_MIXED, Z=(3.0,), rc=(0.8,))
    for k in ("TF", "vW", "NL", "H", "PP", "total"):
        assert abs(E[k] - Eo[k]) / len(pos) <= 1e-6, (k, E[k], Eo[k])
    m = knot_mask(rho.astype(np.float32).astype(np.float64), kw["n_knots"])
    assert np.linalg.norm((V - Vo)[m]) / np.linalg.norm(Vo[m]) <= 1e-4


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("shape", [(4, 4, 4), (16, 9, 15), (27, 10, 125), (162, 6, 8), (5, 81, 243), (64, 12, 512),
                                   (1024, 4, 6), (6, 8, 1024), (2, 3, 5)])
def test_plain_transforms_return_the_field(shape, dtype):
    g = ofd.Grid(np.diag([5.0, 6.0, 7.0]), shape)
    x = torch.from_numpy(np.random.default_rng(sum(shape)).normal(0.3, 1.0, shape)).to("cuda", dtype)
    y = g.interpolate(x, g)
    eps = torch.finfo(dtype).eps
    assert float((y - x).abs().max()) <= 100 * eps * float(x.abs().max())


def _shared_tile_picks(cell, shape, precision):
    """Indices of the reciprocal-space candidates in which several blocks share a column tile (the list is in
    the report of a grid whose kernels are all forced, which times nothing)."""
    g = ofd.Grid(cell, shape)
    for option in (L.OPTION_PICK_ROWS, L.OPTION_PICK_PENCIL, L.OPTION_PICK_RECIP):
        g.set_option(option, 0)
    dt = torch.float64 if precision == L.FP64 else torch.float32
    g.energy_potential(torch.full(shape, 0.01, dtype=dt, device="cuda"),
                       ofd.Functional(n_knots=9, terms=L.TERMS_ALL & ~L.TERM_PP, precision=precision))
    seg = [x for x in g.tuning_report(precision).split(";") if x.strip().startswith("recip")][0]
    names = re.findall(r"\[([^\]]*)\]", seg)
    return [i for i, x in enumerate(names) if re.search(r" s[2-8]$", x)]


def _long_n0(n, cols):
    shape = (n,) + cols
    cell = np.diag([0.3 * max(m, 12) for m in shape])
    pos = lattice_positions(cell, (max(1, round(n * 0.3 / 4.8)), 1, 1), n + 3)
    rho = W.renormalise(W.apply_noise(W.gaussian_density(cell, shape, pos, 3.0, 1.0) + 5e-3, 0.03, n), cell,
                        3.0 * len(pos))
    return cell, shape, pos, rho


def _close(E, V, Eo, Vo, rho, n_atoms, knots):
    for k in ("TF", "vW", "NL", "H", "PP", "total"):
        assert abs(E[k] - Eo[k]) / n_atoms <= 1e-6, (k, E[k], Eo[k])
    m = knot_mask(rho.astype(np.float32).astype(np.float64), knots)
    assert np.linalg.norm((V - Vo)[m]) / np.linalg.norm(Vo[m]) <= 1e-4


def test_tiles_are_not_shared_where_memory_does_not_allow_their_slots():
    """A cap between twelve channels and the eight slots more of a tile shared by eight blocks."""
    cell, shape, pos, rho = _long_n0(375, (3, 8))
    pick = _shared_tile_picks(cell, shape, L.FP32_MIXED)[-1]
    NH = 375 * 3 * 5
    # (the channels and V_ext, the ions' phase tables in both precisions, 128 KB for the small arrays)
    cap = 8 * NH * (12 + 1) + 24 * len(pos) * (375 + 3 + 5) + (1 << 17)
    E, V, Eo, Vo, og, g = run_both(cell, shape, pos, rho, dict(n_knots=9), L.FP32_MIXED, Z=(3.0,), rc=(0.8,),
                                   options=((L.OPTION_PICK_RECIP, pick), (L.OPTION_ALLOC_CAP, cap)))
    _close(E, V, Eo, Vo, rho, len(pos), 9)


@pytest.mark.parametrize("n,cols,precision", [
    (n, cols, p) for n, cols in ((45, (15, 8)), (128, (3, 5)), (225, (3, 5)), (250, (15, 8)), (375, (3, 5)), (486, (5, 8)))
    for p in (L.FP32_MIXED, L.FP64) if (n, p) != (375, L.FP64)])          # (no FP64 form: too many threads)
def test_shared_tiles_match_oracle(n, cols, precision):
    """Every candidate whose column tiles are shared by several blocks: nine knots for up to eight blocks,
    plans of two and three passes with radices 2, 3 and 5, the last tile ragged."""
    cell, shape, pos, rho = _long_n0(n, cols)
    picks = _shared_tile_picks(cell, shape, precision)
    assert picks
    for pick in picks:
        E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, dict(n_knots=9), precision, Z=(3.0,), rc=(0.8,),
                                       options=((L.OPTION_PICK_RECIP, pick),))
        if precision == L.FP64:
            assert abs(E["total"] - Eo["total"]) <= 1e-10 * max(1.0, abs(Eo["total"])), pick
            assert np.max(np.abs(V - Vo)) <= 1e-9 * max(1.0, np.max(np.abs(Vo))), pick
        else:
            _close(E, V, Eo, Vo, rho, len(pos), 9)


@pytest.mark.parametrize("n", (64, 80, 96, 120, 192, 1024))
@pytest.mark.parametrize("role", range(3))
def test_configurations_past_the_fifth_match_oracle(n, role):
    """The candidates that the tests of the first five leave out."""
    shape, option = _role_cases(n)[role]
    count = _n_configurations(shape, ("rows", "pencil", "recip")[role])
    cell, pos, rho = _config_case(shape)
    for pick in range(5, count):
        E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, dict(n_knots=6), L.FP32_MIXED, Z=(3.0,), rc=(0.8,),
                                       options=((option, pick),))
        _close(E, V, Eo, Vo, rho, len(pos), 6)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("role", sorted(ROLES))
def test_any_length_configurations_past_the_third_match_oracle(role, n):
    cell, shape, pos, rho = _case(role, n)
    for pick in range(3, _n_configurations(shape, role)):
        E, V, Eo, Vo, og, _ = run_both(cell, shape, pos, rho, dict(n_knots=7), L.FP32_MIXED, Z=(3.0,), rc=(0.8,),
                                       options=((ROLES[role][1], pick),))
        _close(E, V, Eo, Vo, rho, len(pos), 7)


# odd rows (the scalar accesses) and rows of four points, a ragged last row pair, n0 of two and three passes
FILTER_SHAPES = [(27, 25, 45), (125, 9, 15), (162, 6, 8), (16, 15, 250)]


def _filter_case(shape, precision, sheared=True):
    cell = np.diag([0.45 * max(m, 12) for m in shape])
    if sheared:
        cell[1, 0], cell[2, 1] = 0.6, -0.4
    pos = np.array([[0.45, 0.5, 0.5], [0.55, 0.5, 0.5]]) @ cell
    rho = W.renormalise(W.gaussian_density(cell, shape, pos, 2.0, 1.5) + 1e-4, cell, 4.0)
    dt = torch.float64 if precision == L.FP64 else torch.float32
    return cell, pos, rho, torch.from_numpy(np.ascontiguousarray(rho)).to("cuda", dt)


def _propagate(cell, shape, pos, rho, precision, kernels):
    g = ofd.Grid(cell, shape)
    g.set_option(L.OPTION_KERNELS, kernels)
    g.set_ions(pos, [0, 0], [2.0], [1.0])
    re, im = rho.sqrt(), torch.zeros_like(rho)
    g.td_kick(re, im, [0.05, 0.02, -0.03])
    start = (re + 1j * im).to(torch.complex128).cpu().numpy()
    f = ofd.Functional(terms=L.TERM_TF | L.TERM_VW | L.TERM_HARTREE | L.TERM_PP, precision=precision)
    g.td_propagate(re, im, rho, f, 0.05, 2, solver_tol=1e-12 if precision == L.FP64 else 1e-7)
    return start, (re + 1j * im).to(torch.complex128).cpu().numpy()


@pytest.mark.parametrize("precision,tol", [(L.FP64, 1e-9), (L.FP32_MIXED, 2e-4)])
@pytest.mark.parametrize("sheared", [True, False])
@pytest.mark.parametrize("shape", FILTER_SHAPES)
def test_filters_of_a_propagation_match_oracle_and_general_path(shape, sheared, precision, tol):
    """H, H^2 and the preconditioner of both components (two fields, potential and base in the epilogue)."""
    cell, pos, rho, rho_d = _filter_case(shape, precision, sheared)
    start, psi = _propagate(cell, shape, pos, rho_d, precision, L.KERNELS_AUTO)
    scale = np.max(np.abs(psi))
    _, general = _propagate(cell, shape, pos, rho_d, precision, L.KERNELS_GENERIC)
    assert np.max(np.abs(psi - general)) < tol * scale
    if sheared and any(m % 2 == 0 for m in shape):
        return          # on the Nyquist planes of a sheared cell the oracle's splitting iteration does not converge
    og = OGrid(cell, shape)
    Vg = ofn.external_potential_G(og, pos, [0, 0], [2.0], [1.0])
    ref, _ = otd.propagate(og, start, rho_d.double().cpu().numpy(), OFunc(terms=("TF", "VW", "HARTREE", "PP")), Vg,
                           0.05, 2, n_corrector=1)
    assert np.max(np.abs(psi - ref)) < tol * scale


@pytest.mark.parametrize("precision,tol", [(L.FP64, 1e-9), (L.FP32_MIXED, 1e-3)])
@pytest.mark.parametrize("shape", FILTER_SHAPES)
def test_preconditioned_iterations_match_general_path(shape, precision, tol):
    """Three preconditioned iterations (FP32: each potential within 1e-4, as for every kernel)."""
    cell, pos, rho, rho_d = _filter_case(shape, precision)
    out = []
    for kernels in (L.KERNELS_AUTO, L.KERNELS_GENERIC):
        g = ofd.Grid(cell, shape)
        g.set_option(L.OPTION_KERNELS, kernels)
        g.set_ions(pos, [0, 0], [2.0], [1.0])
        psi = (rho_d + 1e-3).sqrt()
        f = ofd.Functional(terms=L.TERM_TF | L.TERM_VW | L.TERM_HARTREE | L.TERM_PP, precision=precision)
        g.optimize_density(psi, f, 4.0, max_iter=3, precondition=True, raise_on_not_converged=False)
        out.append(psi.double())
    assert float((out[0] - out[1]).norm() / out[1].norm()) < tol
