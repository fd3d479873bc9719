"""Set-ups with little device memory left: what is only there for speed is left out, and the energies
come by the forms that need less."""
import numpy as np
import pytest
import torch

import paper_1611_06797_gb300 as L
from synth import ModelSolidSpec, build_model_solid
from tests.conftest import solid

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def _system(phases):
    # 3071 plane waves and 2 occupied orbitals: the virtuals and the Green's function are almost all of it
    return build_model_solid(ModelSolidSpec("mem24", a=12.0, grid=24, r2=81, wells=2, n_occ=2, n_tau=2, seed=5),
                             random_phases=phases, device="cuda")


class _Hold:
    """All of the device's free memory but `leave` bytes, in allocations of the test's own."""

    def __init__(self, leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.parts = []
        free = torch.cuda.mem_get_info()[0]
        if free > leave:
            self.parts.append(torch.empty(free - leave, dtype=torch.uint8, device="cuda"))

    def release(self):
        self.parts.clear()
        torch.cuda.empty_cache()


def test_general_orbitals_without_room_for_a_second_copy_of_the_virtuals():
    """149 MB of virtuals and 151 MB of Green's function fit in 420 MB, the virtuals by plane wave (149 MB
    more, for the tensor-core products) do not: the products run on the CUDA cores."""
    s = _system(phases=True)
    tau, w = np.array([0.5, 3.0]), np.array([0.4, 0.6])
    # load the kernels first (their code takes device memory of its own)
    small = solid("tiny", random_phases=True)
    for simt in (False, True):
        c = L.setup_from_solid(small, precision=L.FP64, real=False, simt_gemm=simt)
        L.ltmp2_energy(c, tau, w)
        L.ltmp2_destroy(c)
    c = L.setup_from_solid(s, precision=L.FP64, real=False)
    ref = L.ltmp2_energy(c, tau, w)
    L.ltmp2_destroy(c)
    hold = _Hold(420 * MIB)
    try:
        c = L.setup_from_solid(s, precision=L.FP64, real=False)
        e = L.ltmp2_energy(c, tau, w)
        L.ltmp2_destroy(c)
    finally:
        hold.release()
    # FP64 sums of 1e5 terms in another order
    assert abs(e[0] - ref[0]) < 1e-12 * abs(ref[0]) and abs(e[1] - ref[1]) < 1e-12 * abs(ref[0])
    assert np.abs(e[2] - ref[2]).max() < 1e-12 * abs(ref[0])


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture(scope="module")
def large():
    from synth import SPECS
    s = build_model_solid(SPECS["batch5"], device="cuda")   # 27^3, 64 occupied
    torch.cuda.empty_cache()
    return s


def test_pair_matrices_come_with_the_first_whole_energy(large):
    """The 27^3 system's matrices (over 4 GB in FP32): not in a context that runs shares alone, taken once by
    the first whole energy, with the levels that are set by then; small systems hold theirs from set-up."""
    s = large
    tau, w = np.array([1.5]), np.array([0.7])
    ctx = L.setup_from_solid(s, precision=L.FP32, real=True)
    n = L.ltmp2_num_primary_gprime(ctx)
    f0 = _free()
    a = L.ltmp2_energy_partial(ctx, tau, w, 0, n // 2)
    b = L.ltmp2_energy_partial(ctx, tau, w, n // 2, n)
    assert f0 - _free() < 64 * MIB
    L.ltmp2_set_extrapolation(ctx, 8, 1.05)
    f1 = _free()
    e = L.ltmp2_energy(ctx, tau, w)
    assert f1 - _free() > 4096 * MIB
    f2 = _free()
    lev = L.ltmp2_level_energies(ctx)
    again = L.ltmp2_energy(ctx, tau, w)
    assert f2 - _free() < 64 * MIB
    tol = 3e-6 * abs(e[0])   # FP32: co-densities of (j, i) from another transform
    assert abs(e[0] - a[0] - b[0]) < tol and abs(e[1] - a[1] - b[1]) < tol
    assert again[0] == e[0] and again[1] == e[1]
    halves = []
    for x, y in ((0, n // 2), (n // 2, n)):
        L.ltmp2_energy_partial(ctx, tau, w, x, y)
        halves.append(L.ltmp2_level_energies(ctx))
    for key in ("E_d", "E_x"):
        assert np.abs(lev[key] - halves[0][key] - halves[1][key]).max() < tol
    L.ltmp2_destroy(ctx)
    small = L.setup_from_solid(solid("cfg1"), precision=L.FP32, real=True)
    L.ltmp2_energy_partial(small, tau, w, 0, 1)
    f3 = _free()
    L.ltmp2_energy(small, tau, w)
    assert f3 - _free() < MIB
    L.ltmp2_destroy(small)


def test_whole_energy_without_room_for_the_matrices(large):
    """Less than four times the matrices free at the first whole energy: it goes by slabs of G'."""
    s = large
    tau, w = np.array([1.5]), np.array([0.7])
    ctx = L.setup_from_solid(s, precision=L.FP32, real=True)
    n = L.ltmp2_num_primary_gprime(ctx)
    a = L.ltmp2_energy_partial(ctx, tau, w, 0, n // 2)
    b = L.ltmp2_energy_partial(ctx, tau, w, n // 2, n)
    hold = _Hold(12288 * MIB)
    try:
        f0 = _free()
        e = L.ltmp2_energy(ctx, tau, w)
        assert f0 - _free() < 64 * MIB
    finally:
        hold.release()
    # the slabs' sums in another order
    assert abs(e[0] - a[0] - b[0]) < 1e-6 * abs(e[0]) and abs(e[1] - a[1] - b[1]) < 1e-6 * abs(e[0])
    assert np.abs(e[2] - a[2] - b[2] - a[3] - b[3]).max() < 1e-6 * abs(e[0])
    L.ltmp2_destroy(ctx)
