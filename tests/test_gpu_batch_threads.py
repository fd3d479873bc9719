"""Batches set up, captured and run from several host threads at once: the persistent kernels' twiddle
tables and shared-memory limits belong to the device and are shared by the threads."""
import threading

import numpy as np
import pytest

import paper_1611_06797_gb300 as L
from oracle import OracleSystem, denominator_range, sinc_laplace_quadrature
from tests.conftest import solid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_batches_from_several_threads(precision):
    names = ["tiny", "tiny2", "cfg1"]
    solids = {n: solid(n) for n in names}
    quads = {n: sinc_laplace_quadrature(2, *denominator_range(OracleSystem.from_solid(solids[n]))) for n in names}
    want, got, errors = {}, {}, []
    for n in names:
        c = L.setup_from_solid(solids[n], precision=getattr(L, precision.upper()), real=True)
        want[n] = L.ltmp2_energy(c, *quads[n])[:2]
        L.ltmp2_destroy(c)

    def work(t):
        try:
            n = names[t % len(names)]
            ctxs = [L.setup_from_solid(solids[n], precision=getattr(L, precision.upper()), real=True) for _ in range(2)]
            for _ in range(3):
                b = L.ltmp2_batch_create(ctxs, [quads[n][0]] * 2, [quads[n][1]] * 2)
                assert b.persistent()
                got[t] = (n, b.run())
                b.destroy()
            for c in ctxs:
                L.ltmp2_destroy(c)
        except Exception as e:   # noqa: BLE001 - reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    rel = 1e-12 if precision == "fp64" else 2e-6   # the slabs' sums against the symmetric passes'
    for n, (ed, ex) in got.values():
        assert np.abs(np.asarray(ed) - want[n][0]).max() < rel * abs(want[n][0])
        assert np.abs(np.asarray(ex) - want[n][1]).max() < rel * abs(want[n][0])
