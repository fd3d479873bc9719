"""The FP64 plane kernel takes each plane's fixed-point scale from a sum over its block: block shapes
whose lines do not fill whole warps (the default on 36^3 and 40^3, on 24^3 with three occupied, and
after ltmp2_set_tuning elsewhere) must give the energies of the oracle, and those of a shape that
does fill them."""
import numpy as np
import pytest

import paper_1611_06797_gb300 as L
from oracle import OracleSystem, denominator_range, laplace_denominator, mp2_energy, sinc_laplace_quadrature
from synth import ModelSolidSpec, build_model_solid

pytestmark = pytest.mark.gpu

# grid -> (cell constant in bohr, squared sphere radius in index units), occupied orbitals
SYSTEMS = {12: (6.0, 12, 8), 18: (6.5, 16, 4), 20: (6.0, 16, 4), 24: (6.0, 12, 3), 25: (7.0, 16, 4), 27: (6.5, 16, 4),
           36: (7.0, 16, 3), 40: (6.5, 16, 3)}


def _system(n, real):
    a, r2, n_occ = SYSTEMS[n]
    s = build_model_solid(ModelSolidSpec(f"block{n}", a=a, grid=n, r2=r2, wells=2, n_occ=n_occ, n_tau=3, seed=300 + n),
                          random_phases=not real)
    o = OracleSystem.from_solid(s)
    tau, w = sinc_laplace_quadrature(3, *denominator_range(o))
    return s, o, tau, w


@pytest.mark.parametrize("real", [True, False], ids=["real", "general"])
@pytest.mark.parametrize("n", sorted(SYSTEMS))
def test_blocks_of_partial_warps(n, real):
    s, o, tau, w = _system(n, real)
    ref = mp2_energy(o, laplace_denominator(tau, w))
    ctx = L.setup_from_solid(s, precision=L.FP64, real=real)
    out = {}
    for ib in [0] + list(range(1, s.n_occ + 1)):   # 0: the default; n ib threads
        L.ltmp2_set_tuning(ctx, plane_kernel=2, plane_ib=ib)
        out[ib] = L.ltmp2_energy(ctx, tau, w)
    L.ltmp2_destroy(ctx)
    # 1e-12 of the direct term: rounding errors of FP64 sums of 1e5 terms
    tol = 1e-12 * abs(ref["E_d"])
    for ib, (ed, ex, ep) in out.items():
        assert abs(ed - ref["E_d"]) < tol and abs(ex - ref["E_x"]) < tol, (ib, ed - ref["E_d"], ex - ref["E_x"])
        assert np.abs(ep - ref["e_d"] - ref["e_x"]).max() < tol, ib
        # the planes' scales are powers of two above their norms, the same for every shape unless a norm
        # lies within its own rounding of one: the results agree to the last bits
        assert abs(ed - out[1][0]) <= 1e-15 * abs(ed) and np.abs(ep - out[1][2]).max() <= 1e-15 * abs(ed), ib
