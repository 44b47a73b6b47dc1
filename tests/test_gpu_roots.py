"""The roots and the reciprocal that set fixed points, against references of more precision (pt_math_check):
sqrt_full and root_full of the FP64 forms' Picard update, and the double-float iteration's reciprocal of an
unnormalised sum. eps = 2^-53; the references are NumPy's long doubles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
RCP_FULL, SQRT_FULL, ROOT_FULL, DF_RCP_SUM = 1, 15, 16, 17


def _run(fn, a, b=None):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_08716_gb300 import native as N
    ta = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    tb = None if b is None else torch.from_numpy(np.ascontiguousarray(b, dtype=np.float64)).cuda()
    out = torch.empty_like(ta)
    torch.cuda.synchronize()
    rc = N.load().pt_math_check(fn, ta.data_ptr(), None if tb is None else tb.data_ptr(), out.data_ptr(), ta.numel(),
                                None)
    assert rc == N.PT_OK, rc
    return out.cpu().numpy()


def _arguments(n=100000):
    """The range of the seeded path, half of it next to 1, with its ends and 1 itself."""
    rng = np.random.default_rng(21)
    x = np.exp2(rng.uniform(-60.0, 60.0, n))
    near = 1.0 + rng.choice([-1.0, 1.0], n) * np.exp2(rng.uniform(-53.0, -1.0, n))
    ends = np.array([2.0 ** -60, np.nextafter(2.0 ** 61, 0.0), 1.0, np.nextafter(1.0, 0.0), np.nextafter(1.0, 2.0)])
    return np.concatenate([x, near, ends])


def test_square_root():
    """s = x r rounds once and its rounding is halved by the correction, which rounds once: 1.5 eps."""
    x = _arguments()
    want = np.sqrt(x.astype(np.longdouble))
    err = np.abs(_run(SQRT_FULL, x).astype(np.longdouble) - want) / want
    assert err.max() <= 1.6 * EPS, float(err.max() / EPS)
    assert np.isnan(_run(SQRT_FULL, np.array([np.nan, -1.0]))).all()


@pytest.mark.parametrize("m", [3, 5, 10, 63, 64])
def test_mth_root(m):
    """y^m holds at most m roundings, of which the root takes 1/m, the last sum rounds once, the rest (rounding
    of t, of 1/x, the dropped term) is below 2^-12 of that: 2 eps."""
    x = _arguments()
    want = x.astype(np.longdouble) ** (np.longdouble(1) / m)
    err = np.abs(_run(ROOT_FULL, x, np.full_like(x, m)).astype(np.longdouble) - want) / want
    assert err.max() <= 2.1 * EPS, (m, float(err.max() / EPS))


@pytest.mark.parametrize("m", [3, 10, 64])
def test_mth_root_beyond_its_range(m):
    """The library's exp(log x / m): log x, 1/m and their product round by 2, 1 and 1 eps, which the exponential
    carries times |log x| / m, and rounds by 2 itself."""
    rng = np.random.default_rng(22)
    x = np.concatenate([np.exp2(rng.uniform(61.0, 1000.0, 5000)), np.exp2(rng.uniform(-1000.0, -60.0, 5000)),
                        [2.0 ** 61, np.nextafter(2.0 ** -60, 0.0)]])
    want = x.astype(np.longdouble) ** (np.longdouble(1) / m)
    err = np.abs(_run(ROOT_FULL, x, np.full_like(x, m)).astype(np.longdouble) - want) / want
    bound = (2.0 + 4.0 * np.abs(np.log(x)) / m) * EPS
    assert (err <= bound).all(), (m, float((err / bound).max()))
    odd = _run(ROOT_FULL, np.array([np.nan, -1.0, np.inf, 0.0]), np.full(4, float(m)))
    assert np.isnan(odd[:2]).all() and odd[2] == np.inf and odd[3] == 0.0


def test_double_float_reciprocal_of_a_sum():
    """u = 2^-48: the unnormalised sum is good to 2 u, d = 1 - x r to 3 u and its product with r to 2 u."""
    rng = np.random.default_rng(23)
    a = np.exp(rng.uniform(np.log(1e-10), np.log(1e10), 200000))
    b = a * np.exp2(rng.uniform(-30.0, 2.0, a.size))

    def pair(x):
        hi = x.astype(np.float32)
        return hi.astype(np.float64) + (x - hi).astype(np.float32).astype(np.float64)
    want = 1.0 / (pair(a) + pair(b))
    err = np.abs(_run(DF_RCP_SUM, a, b) - want) / want
    assert err.max() <= 8 * 2.0 ** -48, float(err.max() * 2.0 ** 48)
    assert np.isnan(_run(DF_RCP_SUM, np.array([np.nan]), np.array([1.0]))).all()


def test_reciprocal_third_order():
    """1/x: the seed's error cubed is below the rounding; e (1 + e) and the last sum round once: 1.1 eps."""
    x = _arguments()
    want = np.longdouble(1) / x.astype(np.longdouble)
    err = np.abs(_run(RCP_FULL, x).astype(np.longdouble) - want) / want
    assert err.max() <= 1.1 * EPS, float(err.max() / EPS)


def test_missing_operand_is_rejected():
    torch = pytest.importorskip("torch")
    from paper_2207_08716_gb300 import native as N
    a = torch.ones(4, dtype=torch.float64, device="cuda")
    for fn in (ROOT_FULL, DF_RCP_SUM, 18):
        assert N.load().pt_math_check(fn, a.data_ptr(), None, a.data_ptr(), 4, None) == N.PT_EINVAL
