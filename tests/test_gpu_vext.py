"""V_ext(G) of the FP32-mixed path with several species (vext_fast_kernel<true>): the species' terms are
summed in FP64 and rounded once, whatever cancels between them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2002_02985_gb300 as ofd  # noqa: E402
from paper_2002_02985_gb300 import _lib as L  # noqa: E402

PP = dict(terms=L.TERM_PP)


def _potential(cell, shape, pos, species, Z, rc):
    g = ofd.Grid(cell, shape)
    g.set_ions(pos, species, Z, rc)
    _, V = g.energy_potential(torch.full(shape, 0.01, dtype=torch.float32, device="cuda"), ofd.Functional(**PP))
    return V.double()


@pytest.mark.parametrize("shape", [(24, 20, 18), (9, 15, 250)])
def test_species_that_cancel_leave_the_difference(shape):
    """Ions of charge 1000 and -999 on the same sites are ions of charge 1: each coefficient is one FP64
    difference (1000 x 2^-53) rounded to FP32 once, so at most one FP32 unit away from the single
    species' and, over the transform, 2^-22 of its norm.  Rounding after each species would leave
    1000 units."""
    cell = np.diag([0.4 * n for n in shape])
    pos = np.random.default_rng(3).uniform(0.0, 1.0, (5, 3)) @ cell
    one = _potential(cell, shape, pos, np.zeros(5, np.int32), (1.0,), (0.8,))
    two = _potential(cell, shape, np.concatenate([pos, pos]), np.repeat(np.arange(2, dtype=np.int32), 5),
                     (1000.0, -999.0), (0.8, 0.8))
    assert float((two - one).norm() / one.norm()) <= 2.0 ** -22


@pytest.mark.parametrize("counts", [(1, 70), (33, 0, 5), (1, 1, 1, 1, 1)])
def test_equal_species_match_one_species(counts):
    """Ions labelled as several species of one charge and radius: groups around the tile of 32 and the
    group of 8, a species without ions, as many species as ions.  Only the FP32 groups of 8 differ, so
    every structure factor by at most ten roundings of terms whose norm is its own: 16 x 2^-24."""
    shape, n = (20, 12, 27), sum(counts)
    cell = np.diag([0.7 * m for m in shape])
    pos = np.random.default_rng(n).uniform(0.0, 1.0, (n, 3)) @ cell
    species = np.random.default_rng(n).permutation(np.repeat(np.arange(len(counts), dtype=np.int32), counts))
    one = _potential(cell, shape, pos, np.zeros(n, np.int32), (3.0,), (0.8,))
    many = _potential(cell, shape, pos, species, (3.0,) * len(counts), (0.8,) * len(counts))
    assert float((many - one).norm() / one.norm()) <= 16 * 2.0 ** -24


@pytest.mark.parametrize("n_species", [1, 8])
def test_form_factors_in_place_match_the_table(n_species):
    """Under a cap that admits the workspace but not the FP64 form factors the kernel evaluates them in
    place, in FP64 too: at most one FP32 unit of a coefficient."""
    shape = (32, 32, 32)
    cell, NH = np.diag([9.0, 10.0, 11.0]), 32 * 32 * 17
    pos = np.random.default_rng(n_species).uniform(0.0, 1.0, (24, 3)) @ cell
    species = np.arange(24, dtype=np.int32) % n_species
    Z, rc = tuple(1.0 + np.arange(n_species)), tuple(0.6 + 0.1 * np.arange(n_species))
    V = []
    for cap in (0, (3 + 1) * NH * 8 + (3 << 15 if n_species == 1 else 1 << 19)):
        g = ofd.Grid(cell, shape)
        g.set_ions(pos, species, Z, rc)
        g.set_option(L.OPTION_ALLOC_CAP, cap)
        V.append(g.energy_potential(torch.full(shape, 0.01, dtype=torch.float32, device="cuda"),
                                    ofd.Functional(**PP))[1].double())
    assert float((V[1] - V[0]).norm() / V[0].norm()) <= 2.0 ** -23


def _group_error(chain_of_four):
    """rms error, against FP64, of the FP32 sum of eight products of phases p q (complex, so two products per
    component): each product rounded and then added, or fused into two chains of four."""
    f = np.float32
    rng = np.random.default_rng(11)
    p, q = (np.exp(2j * np.pi * rng.uniform(0.0, 1.0, (8, 200000))) for _ in range(2))
    a, b, c, d = p.real.astype(f), p.imag.astype(f), q.real.astype(f), q.imag.astype(f)
    fma = lambda x, y, z: (x.astype(np.float64) * y + z).astype(f)
    exact = (a.astype(np.float64) * c - b.astype(np.float64) * d).sum(0)
    if chain_of_four:
        s = [np.zeros(p.shape[1], f) for _ in range(2)]
        for i in range(8):
            s[i // 4] = fma(-b[i], d[i], fma(a[i], c[i], s[i // 4]))
        s = s[0] + s[1]
    else:
        s = np.zeros(p.shape[1], f)
        for i in range(8):
            s = s + fma(a[i], c[i], -(b[i] * d[i]))
    return np.sqrt(np.mean((s - exact) ** 2))


def test_groups_of_ions_lose_no_more_than_rounded_products():
    """Ions of charge Z and, in another order, of charge -Z on the same sites: what is left of S(G) is the
    rounding of the FP32 groups alone (the phases and their products are the same).  It is no larger than
    with every product rounded and then added (a margin of 10 % for the 3000 samples; fused into one chain
    of eight it would be 1.2 times that)."""
    shape, n = (16, 18, 20), 480
    cell = np.diag([8.0, 9.0, 10.0])
    rng = np.random.default_rng(2)
    pos = rng.uniform(0.0, 1.0, (n, 3)) @ cell
    both = np.concatenate([pos, pos[rng.permutation(n)]])
    V = _potential(cell, shape, both, np.repeat(np.arange(2, dtype=np.int32), n), (3.0, -3.0), (0.3, 0.3))
    h = torch.fft.rfftn(V.reshape(shape), norm="forward").cpu().numpy()
    m = [np.fft.fftfreq(x, 1.0 / x) for x in shape[:2]] + [np.arange(shape[2] // 2 + 1)]
    q2 = sum(((2 * np.pi * k / cell[i, i]) ** 2).reshape([-1 if j == i else 1 for j in range(3)])
             for i, k in enumerate(m))
    q2[0, 0, 0] = 1.0
    S = h / (-4.0 * np.pi * 3.0 * np.exp(-0.25 * 0.3 ** 2 * q2) / q2 / 720.0)
    inner = np.ones(S.shape, bool)
    inner[0, 0, 0] = inner[8] = inner[:, 9] = inner[:, :, 10] = False      # (Nyquist planes come back real)
    rms = np.sqrt(np.mean(np.abs(S[inner]) ** 2) / 2.0)                    # per component
    groups = 2 * n / 8
    assert _group_error(True) <= 1.02 * _group_error(False)
    assert rms <= 1.1 * np.sqrt(groups) * _group_error(False)
