"""The arithmetic the exact-slice tensor-core products rest on, restated on the host in NumPy for both
forms, 8 slices in windows of 384 k (FP64) and 4 slices in windows of 640 k (FP32): rows scaled by a power
of two with |x| < 2^e and rounded to an integer below 2^(7 S), balanced digits of 7 bits, the slice
products with s + t < S accumulated per order s + t in FP32 over a window, drained as 32-bit pairs of
orders (acc_2q 2^7 + acc_2q+1) into 64-bit integers, four orders to a sum, and scaled once.
Checked: the digit bounds (|d_0| <= 128, -64 <= d_s < 64), the remainder (half a unit of the last digit),
that every partial sum of an order stays below 2^24 (so FP32 holds it exactly whatever its rounding: the
FP32 running sums here equal the exact integer sums) and every drained pair below 2^31, including the
worst case of a window, and the error of the combined product against the exact one.  The device kernel
itself is tested on the GPU (tests/test_gpu_dgemm.py, tests/test_gpu_products.py)."""
import numpy as np
import pytest

BITS = 7
# slices, window in k (DRAIN_KB blocks of 16), the type of the operands
FORMS = [(8, 384, np.float64), (4, 640, np.float32)]


def slices(x, S):
    """Rows of x -> integers d [S][rows][k] (top digit first) and exponents e [rows]."""
    m = np.abs(x).max(axis=1)
    e = np.where(m > 0, np.frexp(m)[1], 0)      # m = f 2^e with f in [1/2, 1): m < 2^e
    v = np.rint(np.ldexp(x.astype(np.longdouble), (BITS * S - e)[:, None])).astype(np.int64)
    d = np.empty((S,) + x.shape, dtype=np.int64)
    for s in range(S - 1, 0, -1):
        d[s] = ((v + 64) & 127) - 64
        v = (v - d[s]) >> BITS
    d[0] = v
    return d, e


def product(a, b, S, window):
    da, ea = slices(a, S)
    db, eb = slices(b, S)
    k = a.shape[1]
    sums = np.zeros((S // 4, a.shape[0], b.shape[0]), dtype=np.int64)
    peak = pair_peak = 0
    for w0 in range(0, k, window):
        acc = []
        for d in range(S):
            o32 = np.zeros((a.shape[0], b.shape[0]), np.float32)
            exact = np.zeros((a.shape[0], b.shape[0]), dtype=np.int64)
            for s in range(d + 1):
                for q in range(w0, min(k, w0 + window)):        # one k at a time: every partial sum
                    p = np.outer(da[s][:, q], db[d - s][:, q])
                    exact += p
                    o32 += p.astype(np.float32)
                    peak = max(peak, int(np.abs(exact).max()))
            assert np.array_equal(o32.astype(np.int64), exact)   # FP32 held every partial sum
            acc.append(exact)
        for q in range(S // 2):
            pair = acc[2 * q] * 128 + acc[2 * q + 1]
            pair_peak = max(pair_peak, int(np.abs(pair).max()))
            sums[q // 2] += pair * (1 << 14) if q % 2 == 0 else pair
    v = sums[0].astype(a.dtype)
    if S == 8:
        v = v * float(1 << 28) + sums[1].astype(np.float64)
    scale = (ea[:, None] + eb[None, :] - BITS * (S + 1)).astype(np.int32)
    return np.ldexp(v, scale), peak, pair_peak


@pytest.mark.parametrize("S,window,T", FORMS)
def test_slice_bounds_and_remainder(S, window, T):
    rng = np.random.default_rng(3)
    x = (rng.standard_normal((16, 257)) * 10.0 ** rng.uniform(-30, 30, size=(16, 1))).astype(T)
    x[2] = 0.0
    x[3, 5] = np.ldexp(T(1.0) - np.finfo(T).epsneg, 40)   # rounds up to the next power of two: digit 128
    d, e = slices(x, S)
    assert np.abs(d[0]).max() <= 128 and d[1:].min() >= -64 and d[1:].max() < 64
    recon = sum(d[s].astype(np.longdouble) * 2.0 ** (-BITS * (s + 1)) for s in range(S))
    scaled = np.ldexp(x.astype(np.longdouble), -e[:, None])
    assert np.all(np.abs(scaled - recon) <= 2.0 ** (-BITS * S - 1))
    assert np.all(d[:, 2] == 0)


@pytest.mark.parametrize("S,window,T", FORMS)
def test_order_sums_stay_exact_in_fp32_and_the_product_is_accurate(S, window, T):
    rng = np.random.default_rng(5)
    k = 2 * window + 132                      # three windows, the last one partial
    a = (rng.standard_normal((6, k)) * 10.0 ** rng.uniform(-15, 15, size=(6, 1))).astype(T)
    b = (rng.standard_normal((5, k)) * 10.0 ** rng.uniform(-15, 15, size=(5, 1))).astype(T)
    c, peak, pair_peak = product(a, b, S, window)
    assert peak < 2 ** 24 and pair_peak < 2 ** 31
    ref = a.astype(np.longdouble) @ b.astype(np.longdouble).T
    # per term, of the two rows' scales (below twice their largest magnitudes): the dropped orders, at most
    # (S - 1) 64^2 2^(-7 (S + 2)) from order S and 1/100 of that from the next ones, and half a unit of the last
    # digit of each operand; then the rounding of the result
    scale = np.abs(a).max(axis=1)[:, None].astype(np.longdouble) * np.abs(b).max(axis=1)[None, :]
    per_term = 4.0 * (1.01 * (S - 1) * 4096 * 2.0 ** (-BITS * (S + 2)) + 2.0 * 2.0 ** (-BITS * S - 1))
    bound = k * per_term * scale + np.finfo(T).eps * np.abs(ref)
    assert np.all(np.abs(c.astype(np.longdouble) - ref) <= bound)


@pytest.mark.parametrize("S,window,T", FORMS)
def test_worst_case_of_a_window(S, window, T):
    """Every digit at its largest magnitude with one sign."""
    per_k = [sum((128 if s == 0 else 64) * (128 if d - s == 0 else 64) for s in range(d + 1)) for d in range(S)]
    assert max(per_k) == per_k[S - 1] == 2 * 128 * 64 + (S - 2) * 64 * 64
    assert per_k[S - 1] * window < 2 ** 24 <= per_k[S - 1] * (window + 48)   # no whole 16-k blocks to spare but two
    for q in range(S // 2):
        assert (per_k[2 * q] * 128 + per_k[2 * q + 1]) * window < 2 ** 31, q
