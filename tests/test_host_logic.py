"""Host logic of the library on a machine without a GPU: its objects linked against a stand-in for
the CUDA runtime (host_cuda.cpp) that keeps device memory on the host, runs no kernel and logs every
copy, memset, launch and wait."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

from paper_2002_02985_gb300 import _lib as L
from paper_2002_02985_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
STREAM = 0x5000                                # a stream of the caller's that is not the legacy one


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    B.build()
    out = str(tmp_path_factory.mktemp("host") / "libofdft_host.so")
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.sources()]
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc, "-o", out,
                    os.path.join(HERE, "host_cuda.cpp"), *objs, "-lpthread"], check=True)
    saved, L._lib = L._lib, None
    try:
        lib = L.load(out)
    finally:
        L._lib = saved
    lib.host_cuda_log.restype = ct.c_char_p
    lib.host_cuda_cost.argtypes = [ct.c_char_p, ct.c_double]
    return lib


class Grid:
    """A grid of the library on the stand-in runtime, with host arrays in the place of device ones."""

    def __init__(self, lib, shape, side=8.0, stream=STREAM):
        self.lib, self.shape = lib, shape
        self.h = ct.c_void_p()
        cell = (ct.c_double * 9)(*np.diag([side] * 3).ravel())
        assert lib.ofdft_grid_create(cell, (ct.c_int * 3)(*shape), ct.c_void_p(stream), ct.byref(self.h)) == 0

    def close(self):
        self.lib.ofdft_grid_destroy(self.h)

    def set_ions(self, n_species=1, pme=0):
        n = max(4, n_species)
        pos, sp = np.random.default_rng(n).uniform(0.0, 8.0, (n, 3)), np.arange(n, dtype=np.int32) % n_species
        Z, rc = 1.0 + np.arange(n_species), 0.7 + 0.1 * np.arange(n_species)
        ptr = lambda a, t: a.ctypes.data_as(ct.POINTER(t))
        ions = L.CIons(n, ptr(pos, ct.c_double), ptr(sp, ct.c_int))
        spec = L.CSpecies(n_species, ptr(Z, ct.c_double), ptr(rc, ct.c_double))
        call = (ct.byref(ions), ct.byref(spec)) + ((pme,) if pme else ())
        return (self.lib.ofdft_set_ions_pme if pme else self.lib.ofdft_set_ions)(self.h, *call)

    def functional(self, precision=L.FP32_MIXED, knots=6, terms=L.TERMS_ALL):
        return L.CFunctional(terms, 5.0 / 6.0, 5.0 / 6.0, knots, L.KNOTS_LOG, None, L.NLPOT_EXACT, L.KERNEL_LWT,
                             precision, 0.0, 0.0, 0.0)

    def density(self, precision=L.FP32_MIXED):
        self.rho = np.full(self.shape, 0.01, np.float64 if precision == L.FP64 else np.float32)
        return ct.c_void_p(self.rho.ctypes.data)

    def evaluate(self, precision=L.FP32_MIXED, **kw):
        E = (ct.c_double * L.N_ENERGIES)()
        f = self.functional(precision, **kw)
        return self.lib.ofdft_energy_potential(self.h, self.density(precision), ct.byref(f), E, None)


def log(lib):
    return [x.split() for x in lib.host_cuda_log().decode().splitlines()]


def test_host_data_reaches_the_device_on_the_grids_stream(lib):
    """Uploads and clears that kernels of the grid's stream read are made on that stream: a copy from
    pageable memory (or a memset) on the legacy stream may still be under way when the call returns,
    and a non-blocking stream does not wait for it."""
    lib.host_cuda_reset()
    a, b = Grid(lib, (24, 20, 18)), Grid(lib, (24, 20, 18))
    for g in (a, b):
        assert g.set_ions(2) == 0
        for p in (L.FP32_MIXED, L.FP64):
            assert g.evaluate(p) == 0
    hs, f = (ct.c_void_p * 2)(a.h, b.h), a.functional()
    rho = (ct.c_void_p * 2)(a.density(), b.density())
    E = (ct.c_double * (2 * L.N_ENERGIES))()
    assert lib.ofdft_energy_potential_batched(2, hs, rho, ct.byref(f), E, None, None) == 0
    assert a.set_ions(1, pme=6) == 0 and a.evaluate() == 0
    ops = log(lib)
    assert [x for x in ops if x[0] in ("memcpy", "memset") and x[1] != "d2h"] == []
    up = [x for x in ops if x[0] == "memcpyAsync" and x[1] == "h2d"]
    assert up and {x[2] for x in up} == {"%x" % STREAM}
    a.close(), b.close()


@pytest.mark.parametrize("kernels", [L.KERNELS_AUTO, L.KERNELS_GENERIC])
@pytest.mark.parametrize("shape", [(192, 16, 192), (200, 16, 250)])
def test_every_device_allows_the_kernels_shared_memory(lib, shape, kernels):
    """More than 48 KB of dynamic shared memory is allowed per kernel and device: a grid on a second device
    sets the attribute of every kernel that a grid on the first one did."""
    seen = []
    for device in (0, 1):
        lib.host_cuda_device(device)
        lib.host_cuda_reset()
        g = Grid(lib, shape)
        assert lib.ofdft_set_option(g.h, L.OPTION_KERNELS, ct.c_longlong(kernels)) == 0
        for p, t in ((L.FP32_MIXED, np.float32), (L.FP64, np.float64)):
            x = np.zeros(shape, t)
            assert lib.ofdft_interpolate(g.h, ct.c_void_p(x.ctypes.data), g.h, ct.c_void_p(x.ctypes.data), p) == 0
        ops = log(lib)
        allowed = {x[1] for x in ops if x[0] == "attribute" and x[3] == str(device)}
        assert {x[1] for x in ops if x[0] == "launch" and ("plain_" in x[1] or "axis0_fft" in x[1])
                and "mean" not in x[1]} <= allowed
        seen.append(allowed)
        g.close()
    lib.host_cuda_device(0)
    assert seen[0] == seen[1]


def test_form_factor_table_is_optional(lib):
    """A cap that admits the workspace of an FP32 evaluation but not the FP64 form factors: the kernel
    evaluates them in place.  One that does not admit the workspace is out of memory as before, and
    without a cap the table is made once and kept."""
    shape, species = (32, 32, 32), 8
    NH = 32 * 32 * 17
    need, table = (3 + 1) * NH * 8 + (1 << 19), species * NH * 8     # three spectra, V_ext, small arrays
    assert (1 << 19) < table
    for cap, rc, tables in ((need, 0, 0), (3 * NH * 8, L.OFDFT_ERR_OOM, 0), (0, 0, species)):
        g = Grid(lib, shape)
        assert g.set_ions(species) == 0
        assert lib.ofdft_set_option(g.h, L.OPTION_ALLOC_CAP, ct.c_longlong(cap)) == 0
        lib.host_cuda_reset()
        for _ in range(2):
            assert g.evaluate(terms=L.TERM_PP) == rc, cap
        ops = [x for x in log(lib) if x[0] == "launch"]
        assert sum("form_table" in x[1] for x in ops) == tables
        if rc == 0:
            assert sum("vext_fast" in x[1] for x in ops) == 1
        g.close()


def test_new_species_are_evaluated_inside_a_capture(lib):
    """After one ordinary call an asynchronous evaluation can be captured, also when the ions have
    become ions of more or other species since: no table is allocated, and none counts as made by a
    launch that has only been captured."""
    g = Grid(lib, (24, 20, 18))
    f, E = g.functional(), np.zeros(L.N_ENERGIES)
    call = lambda: lib.ofdft_energy_potential_async(g.h, g.density(), ct.byref(f), ct.c_void_p(E.ctypes.data), None)
    made = lambda: sum(x[0] == "launch" and "form_table" in x[1] for x in log(lib))
    assert g.set_ions(1) == 0 and g.evaluate() == 0
    for n_species in (3, 2):
        assert g.set_ions(n_species) == 0
        lib.host_cuda_reset()
        lib.host_cuda_capture(1)
        rc = call()
        lib.host_cuda_capture(0)
        assert rc == 0 and made() == 0 and [x for x in log(lib) if x[0] == "refused"] == []
    assert g.set_ions(2) == 0 and call() == 0 and made() == 2
    g.close()


def test_slots_of_shared_tiles_are_optional(lib):
    """The term-2 slots of blocks that share a column tile (32^3 has fewer tiles than SMs): none where
    the knots are too few to be shared out, none where a cap does not admit them, and none added
    inside a capture; the call itself succeeds as it did without shared tiles."""
    NH, small = 32 * 32 * 17, 1 << 17
    made = lambda: [int(x[3]) // (8 * NH) for x in log(lib) if x[0] == "malloc" and int(x[3]) >= 4 * 8 * NH]
    terms = L.TERMS_ALL & ~L.TERM_PP
    g = Grid(lib, (32, 32, 32))
    lib.host_cuda_reset()
    assert g.evaluate(knots=10, terms=terms) == 0 and made()[0] > 13
    g.close()
    for knots, slots in ((6, 9), (10, 13)):
        g = Grid(lib, (32, 32, 32))
        assert lib.ofdft_set_option(g.h, L.OPTION_ALLOC_CAP, ct.c_longlong(8 * NH * slots + small)) == 0
        lib.host_cuda_reset()
        assert g.evaluate(knots=knots, terms=terms) == 0 and made() == [slots]
        assert g.evaluate(knots=knots, terms=terms) == 0 and made() == [slots]
        g.close()
    g = Grid(lib, (32, 32, 32))
    f, E = g.functional(knots=10, terms=terms), np.zeros(L.N_ENERGIES)
    f.nl_potential = L.NLPOT_INTERP
    call = lambda: lib.ofdft_energy_potential_async(g.h, g.density(), ct.byref(f), ct.c_void_p(E.ctypes.data), None)
    lib.host_cuda_reset()
    assert call() == 0 and made() == [13]
    f.nl_potential = L.NLPOT_EXACT
    lib.host_cuda_capture(1)
    rc = call()
    lib.host_cuda_capture(0)
    assert rc == 0 and [x for x in log(lib) if x[0] == "refused"] == []
    g.close()


def test_tuner_runs_a_large_candidate_that_is_behind_once(lib):
    """Beyond 2^24 points a configuration whose warm-up is clearly behind the best of its role is not timed
    further, and the pick is the one that timing all of them would make; one that is ahead or level is."""
    lib.host_cuda_cost(b"kernel", 1.0)
    lib.host_cuda_cost(b"_any_kernel", 3.0)
    try:
        g = Grid(lib, (1024, 18, 1024))
        lib.host_cuda_reset()
        assert g.evaluate(knots=4, terms=L.TERMS_ALL & ~L.TERM_PP) == 0
        report = lib.ofdft_tuning_report(g.h, L.FP32_MIXED).decode()
        g.close()
    finally:
        lib.host_cuda_cost(b"", 0.0)
    segments = {s.split(":")[0].strip(): s for s in report.split(";")}
    launches = [x[1] for x in log(lib) if x[0] == "launch"]
    for role, part in (("recip", "axis0_any_kernel"), ("rows", "row_fwd_any_kernel")):
        behind = segments[role].count("[any")
        assert behind > 0 and "-> any" not in segments[role], report
        assert sum(part in x for x in launches) == behind, report
    names = [x for x in segments["rows"].split("->")[0].split("[")[1:] if not x.startswith("any")]
    assert len(names) > 1
    level = sum("row_fwd" in x and "_any_kernel" not in x for x in launches)
    assert level >= 3 * len(names)


@pytest.mark.parametrize("n2,cost,pick", [(30, 0.92, "pencil"), (27, 0.5, "ctpencil")])
def test_tuner_keeps_the_earlier_of_two_level_candidates_on_small_grids(lib, n2, cost, pick):
    """Where an evaluation takes less than 0.1 ms a candidate replaces an earlier one only when it is ahead by
    more than such short timings scatter, so that the picks, and with them the results' last bits, are those
    of every process."""
    lib.host_cuda_cost(b"kernel", 0.01)
    lib.host_cuda_cost(b"pencil_ct_kernel", 0.01 * cost)
    try:
        g = Grid(lib, (24, 32, n2))
        assert g.evaluate(knots=5, terms=L.TERMS_ALL & ~L.TERM_PP) == 0
        report = lib.ofdft_tuning_report(g.h, L.FP32_MIXED).decode()
        g.close()
    finally:
        lib.host_cuda_cost(b"", 0.0)
    assert [s for s in report.split(";") if s.strip().startswith("pencil")][0].split("-> ")[1].split()[0] == pick, report
