"""The exact-slice products' forms: general orbitals as real products over interleaved real and
imaginary parts, four slices in the precision form, rows of extreme scale and rows that are
not finite."""
import numpy as np
import pytest
import torch

import paper_1611_06797_gb300 as L
from oracle import OracleSystem, denominator_range, laplace_denominator, mp2_energy, sinc_laplace_quadrature
from tests.conftest import solid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["tiny", "tiny2", "cfg1"])     # 123, 179, 515 plane waves: no multiples of a tile
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_general_products_match_real_ones(name, precision):
    """The same real orbitals through the real basis and as general ones, on the tensor cores and
    on the CUDA cores."""
    s = solid(name)
    o = OracleSystem.from_solid(s)
    tau, w = sinc_laplace_quadrature(4, *denominator_range(o))
    ref = mp2_energy(o, laplace_denominator(tau, w))
    # FP64: rounding of sums of about 1e5 terms of both signs; FP32: 2^-24 of the operands, through
    # P_v's cancellation of most of e^{-iG'r} phi_j at small tau (seen: 1e-6)
    tol = (1e-12 if precision == "fp64" else 5e-6) * abs(ref["E_d"])
    for real in (True, False):
        for simt in (False, True):
            ctx = L.setup_from_solid(s, precision=getattr(L, precision.upper()), real=real, simt_gemm=simt)
            ed, ex, ep = L.ltmp2_energy(ctx, tau, w)
            L.ltmp2_destroy(ctx)
            assert abs(ed - ref["E_d"]) < tol and abs(ex - ref["E_x"]) < tol, (real, simt)
            assert np.abs(ep - ref["e_d"] - ref["e_x"]).max() < tol, (real, simt)


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (130, 65, 17), (257, 63, 400), (64, 130, 1200)])
def test_rows_of_any_scale(m, n, k):
    """Rows times powers of two down to denormal and up to 2^1000: the product scales with them
    exactly (entries of 8 bits, so that a denormal row still holds them); a row with a NaN or an
    infinity gives a row of NaN and touches no other."""
    g = np.random.default_rng(m + n + k)
    a = g.integers(-127, 128, (m, k)).astype(float)
    b = g.integers(-127, 128, (n, k)).astype(float)
    exact = a @ b.T                                        # below 2^31: exact in FP64
    ea = g.integers(-40, 40, m)
    eb = g.integers(-40, 40, n)
    ea[0], eb[0] = -1060, 1000                             # entries down to 2^-1060, up to 2^1007
    ta = torch.from_numpy(np.ldexp(a, ea[:, None])).cuda()
    tb = torch.from_numpy(np.ldexp(b, eb[:, None])).cuda()
    c = L.ltmp2_dgemm_nt(ta, tb).cpu().numpy()
    with np.errstate(over="ignore"):
        want = np.ldexp(exact, ea[:, None] + eb[None, :])
    assert np.array_equal(c, want)
    bad = m // 2
    for value in (np.nan, np.inf, -np.inf):
        ta2 = ta.clone()
        ta2[bad, k // 2] = value
        c2 = L.ltmp2_dgemm_nt(ta2, tb).cpu().numpy()
        assert np.isnan(c2[bad]).all()
        keep = np.arange(m) != bad
        assert np.array_equal(c2[keep], want[keep])
