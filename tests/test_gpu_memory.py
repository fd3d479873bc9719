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
