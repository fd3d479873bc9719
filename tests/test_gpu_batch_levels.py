"""A captured batch keeps its energies when the cutoff levels of its contexts change afterwards: the
row groups and level tables that ltmp2_set_extrapolation rewrites are the batch's own copies."""
import numpy as np
import pytest

import paper_1611_06797_gb300 as L
from oracle import OracleSystem, denominator_range, sinc_laplace_quadrature
from tests.conftest import solid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("real", [True, False], ids=["real", "general"])
@pytest.mark.parametrize("at_creation", [None, (8, 1.05), (16, 1.3)], ids=["plain", "8_levels", "16_levels"])
def test_levels_changed_after_the_capture(at_creation, real):
    solids = [solid(n) if real else solid(n, random_phases=True) for n in ("tiny2", "cfg1")]
    quads = [sinc_laplace_quadrature(3, *denominator_range(OracleSystem.from_solid(s))) for s in solids]
    ctxs = [L.setup_from_solid(s, precision=L.FP64, real=real) for s in solids]
    plain = [L.ltmp2_energy(c, *q)[:2] for c, q in zip(ctxs, quads)]
    if at_creation:
        for c in ctxs:
            L.ltmp2_set_extrapolation(c, *at_creation)
    else:
        L.ltmp2_set_slab_size(ctxs[0], 1)   # uneven rounds: one graph branch per system
    b = L.ltmp2_batch_create(ctxs, [q[0] for q in quads], [q[1] for q in quads])
    assert not b.persistent()
    # the same launches on the same tables: the same bits; against the plain energy, sums in another order
    first = b.run()
    for k, (d, x) in enumerate(plain):
        assert abs(first[0][k] - d) < 1e-13 * abs(d) and abs(first[1][k] - x) < 1e-13 * abs(d)
    for levels in ((16, 1.3), (2, 1.01), (1, 1.05), (8, 1.05)):
        for c in ctxs:
            L.ltmp2_set_extrapolation(c, *levels)
        again = b.run()
        assert np.array_equal(again[0], first[0]) and np.array_equal(again[1], first[1]), levels
        # and the contexts' own energies follow the new levels
        for c, q, (d, x) in zip(ctxs, quads, plain):
            e = L.ltmp2_energy(c, *q)
            assert abs(e[0] - d) < 1e-13 * abs(d) and abs(e[1] - x) < 1e-13 * abs(d)
    b.destroy()
    for c in ctxs:
        L.ltmp2_destroy(c)
