"""The slabs of the outer G' loop, which ranges of G' and persistent batches take and whole energies no
longer do: the column kernel of every grid against the oracle, and the spin channels' cross term."""
import numpy as np
import pytest

import paper_1611_06797_gb300 as L
from oracle import OracleSystem, laplace_denominator, uhf_mp2_energy
from synth import SPECS, spin_polarized_pair
from tests.test_gpu_grids import GRIDS, MEV_PER_ATOM, _ragged_slab, _system
from tests.test_gpu_uhf import _quad

pytestmark = pytest.mark.gpu


def _ranges(ctx, tau, w):
    """E_d, E_x and the pair energies from three ranges of G', in ragged slabs."""
    n = L.ltmp2_num_primary_gprime(ctx)
    L.ltmp2_set_slab_size(ctx, min(_ragged_slab(n), L.ltmp2_set_slab_size(ctx, 0)))
    parts = [L.ltmp2_energy_partial(ctx, tau, w, b, e) for b, e in ((0, 1), (1, n // 2), (n // 2, n))]
    return [sum(p[k] for p in parts) for k in range(4)]


@pytest.mark.parametrize("real", [False, True], ids=["general", "real"])
@pytest.mark.parametrize("n", sorted(GRIDS))
def test_slabs_match_oracle_at_grid(n, real):
    s, tau, w, ref = _system(n, phases=not real)
    tol = {L.FP64: 1e-12 * abs(ref["E_d"]),            # FP64 sums of 1e5 terms
           L.FP32: MEV_PER_ATOM * s.n_atoms}           # the precision form's bound
    for precision in (L.FP64, L.FP32):
        ctx = L.setup_from_solid(s, precision=precision, real=real)
        ed, ex, pd, px = _ranges(ctx, tau, w)
        L.ltmp2_destroy(ctx)
        assert abs(ed - ref["E_d"]) < tol[precision] and abs(ex - ref["E_x"]) < tol[precision], precision
        assert np.abs(pd - ref["e_d"]).max() < tol[precision], precision
        assert np.abs(px - ref["e_x"]).max() < tol[precision], precision


@pytest.mark.parametrize("slab", [None, 4])
def test_cross_term_of_slabs_matches_oracle(slab):
    """The overlap route goes by slabs, also for the opposite-spin term."""
    a, b = spin_polarized_pair(SPECS["cfg1"], 5, 3)
    tau, w = _quad(a, b, 6)
    ref = uhf_mp2_energy(OracleSystem.from_solid(a), OracleSystem.from_solid(b), laplace_denominator(tau, w))
    ca, cb = (L.setup_from_solid(x, precision=L.FP64, real=True) for x in (a, b))
    for c in (ca, cb):
        L.ltmp2_set_route(c, L.ROUTE_OVERLAP)
        if slab:
            L.ltmp2_set_slab_size(c, slab)
    ed, ex, es = L.ltmp2_energy_uhf(ca, cb, tau, w)
    for c in (ca, cb):
        L.ltmp2_set_route(c, L.ROUTE_GREEN)
    again = L.ltmp2_energy_uhf(ca, cb, tau, w)         # back on the pair matrices
    L.ltmp2_destroy(ca)
    L.ltmp2_destroy(cb)
    tol = 1e-12 * abs(ref["E_d"])
    for d, x, spin in ((ed, ex, es), again):
        assert abs(d - ref["E_d"]) < tol and abs(x - ref["E_x"]) < tol
        assert np.abs(spin - [ref["E_aa"], ref["E_bb"], ref["E_ab"]]).max() < tol
