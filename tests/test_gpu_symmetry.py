"""Whole energies by the pairs' exchange symmetry (items i <= j, the exchange term as a matrix
times its transpose) against the slabs of the outer G' loop, which every partial range takes, at
the sizes of passes where they can go wrong: one column, ragged parts of one orbital, several
orbitals with a ragged last pass, everything in one; with cutoff levels and a pair mask."""
from dataclasses import replace

import numpy as np
import pytest

import paper_1611_06797_gb300 as L
from oracle import OracleSystem, denominator_range, sinc_laplace_quadrature
from synth import SPECS, build_model_solid
from tests.conftest import solid

pytestmark = pytest.mark.gpu


def _halves(ctx, tau, w, n):
    """The energy from two ranges of G': no range holds every G', so no symmetry is used."""
    a, b = (L.ltmp2_energy_partial(ctx, tau, w, x, y) for x, y in ((0, n // 2), (n // 2, n)))
    return a[0] + b[0], a[1] + b[1], a[2] + b[2] + a[3] + b[3]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("real", [True, False], ids=["real", "general"])
@pytest.mark.parametrize("name", ["tiny2", "cfg1"])
def test_symmetric_passes_match_the_slabs(name, real, precision):
    s = solid(name) if real else solid(name, random_phases=True)
    tau, w = sinc_laplace_quadrature(3, *denominator_range(OracleSystem.from_solid(s)))
    ctx = L.setup_from_solid(s, precision=getattr(L, precision.upper()), real=real)
    n = L.ltmp2_num_primary_gprime(ctx)
    ed, ex, ep = _halves(ctx, tau, w, n)
    # FP64: sums in another order, 1e5 terms; FP32: co-densities of (j, i) from another transform
    tol = (1e-13 if precision == "fp64" else 3e-6) * abs(ed)
    for slab in (1, max(1, n // 3), n - 1, n):
        if L.ltmp2_set_slab_size(ctx, min(slab, L.ltmp2_set_slab_size(ctx, 0))) < 1:
            continue
        e = L.ltmp2_energy(ctx, tau, w)
        assert abs(e[0] - ed) < tol and abs(e[1] - ex) < tol and np.abs(e[2] - ep).max() < tol, slab
        assert np.array_equal(e[2], e[2].T)
    L.ltmp2_set_slab_size(ctx, 0)
    keep = np.ones((s.n_occ, s.n_occ), dtype=bool)
    keep[0, s.n_occ - 1] = keep[s.n_occ - 1, 0] = False
    L.ltmp2_set_pair_mask(ctx, keep)
    ed2, ex2, ep2 = _halves(ctx, tau, w, n)
    e = L.ltmp2_energy(ctx, tau, w)
    assert abs(e[0] - ed2) < tol and abs(e[1] - ex2) < tol and np.abs(e[2] - ep2).max() < tol
    L.ltmp2_destroy(ctx)


@pytest.mark.parametrize("real", [True, False], ids=["real", "general"])
def test_levels_of_the_symmetric_passes(real):
    """Cutoff levels on and off again: the rows of the lower triangle are regrouped each time."""
    s = solid("cfg1") if real else solid("cfg1", random_phases=True)
    tau, w = sinc_laplace_quadrature(2, *denominator_range(OracleSystem.from_solid(s)))
    ctx = L.setup_from_solid(s, precision=L.FP64, real=real)
    n = L.ltmp2_num_primary_gprime(ctx)
    plain = L.ltmp2_energy(ctx, tau, w)
    for n_c, alpha in ((8, 1.05), (16, 1.3), (2, 1.01)):
        L.ltmp2_set_extrapolation(ctx, n_c, alpha)
        e = L.ltmp2_energy(ctx, tau, w)
        lev = L.ltmp2_level_energies(ctx)
        halves = []
        for x, y in ((0, n // 2), (n // 2, n)):
            L.ltmp2_energy_partial(ctx, tau, w, x, y)
            halves.append(L.ltmp2_level_energies(ctx))
        for key in ("E_d", "E_x"):
            slabs = halves[0][key] + halves[1][key]
            assert np.abs(lev[key] - slabs).max() < 1e-13 * abs(plain[0]), (n_c, key)
        assert abs(e[0] - plain[0]) < 1e-13 * abs(plain[0]) and abs(e[1] - plain[1]) < 1e-13 * abs(plain[0])
    L.ltmp2_set_extrapolation(ctx, 1)
    e = L.ltmp2_energy(ctx, tau, w)
    assert abs(e[0] - plain[0]) < 1e-14 * abs(plain[0])
    L.ltmp2_destroy(ctx)


@pytest.mark.parametrize("n_occ", [1, 3, 5, 9])
@pytest.mark.parametrize("real", [True, False], ids=["real", "general"])
def test_direct_blocks(n_occ, real):
    """The direct term's 4 x 4 blocks of (i, j) at ragged orbital counts: the slabs' against the
    symmetric passes' (another kernel, with its own order of the sum)."""
    s = build_model_solid(replace(SPECS["tiny2"], wells=n_occ, n_occ=n_occ), random_phases=not real)
    tau, w = sinc_laplace_quadrature(2, *denominator_range(OracleSystem.from_solid(s)))
    ctx = L.setup_from_solid(s, precision=L.FP64, real=real)
    ed, ex, ep = _halves(ctx, tau, w, L.ltmp2_num_primary_gprime(ctx))
    e = L.ltmp2_energy(ctx, tau, w)
    tol = 1e-13 * abs(ed)   # FP64 sums of 1e5 terms in another order
    assert abs(e[0] - ed) < tol and abs(e[1] - ex) < tol and np.abs(e[2] - ep).max() < tol
    L.ltmp2_destroy(ctx)
