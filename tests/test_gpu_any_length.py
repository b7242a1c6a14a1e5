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
from paper_2002_02985_gb300 import _lib as L  # noqa: E402
from test_gpu_parity import knot_mask, lattice_positions, run_both  # noqa: E402

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
    seg = [x for x in g.tuning_report().split(";") if x.strip().startswith("recip")][0]
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
