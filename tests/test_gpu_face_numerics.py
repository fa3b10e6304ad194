"""Rounding of the arithmetic that the kernels write themselves, function by function.

Reciprocals and roots against numpy's correctly rounded ones over the exponent
range; the conversions and predicates on bits against the casts and
comparisons that they stand for, at the ends of the ranges too; the Riemann solution near p_K, and its departures from the side states, against
a Newton iteration in long double.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TINY32, TINY64 = np.finfo(np.float32).tiny, np.finfo(np.float64).tiny


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch
    from paper_2207_04252_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "face_probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "face_probe.cu")
    subprocess.check_call([build.nvcc()] + build.COMPILE_FLAGS + build.LINK_FLAGS[2:] + ["-o", so, src])
    lib = ctypes.CDLL(so)

    class Probe:
        @staticmethod
        def _run(fn, *head, x, rows):
            a = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
            n = a.shape[-1]
            out = torch.empty((rows, n) if rows else (n,), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            assert fn(*head, ctypes.c_int(n), ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(out.data_ptr())) == 0
            return out.cpu().numpy()

        def scalar(self, op, x):
            return self._run(lib.probe_scalar, ctypes.c_int(op), x=x, rows=0)

        def near(self, gamma, x):
            return self._run(lib.probe_near, ctypes.c_double(gamma), x=x, rows=6)

    return Probe()


def _sweep(lo, hi, n=200000, seed=0):
    """Random mantissas over the binary exponents lo ... hi, and the powers of two themselves."""
    rng = np.random.default_rng(seed)
    e = rng.integers(lo, hi + 1, n)
    return np.concatenate([np.ldexp(1.0 + rng.random(n), e), np.ldexp(1.0, np.arange(lo, hi + 1))])


def _ulps(got, want):
    return float((np.abs(got - want) / np.spacing(np.abs(want))).max())


def test_double_reciprocals_and_roots(probe):
    # one third-order step leaves 2^-59 of the value (0.03 ulp); its last operation and the one
    # before it round: within 1 ulp of the correctly rounded result, within 2 for the longer x^-1/2
    x = _sweep(-1020, 1020)
    assert _ulps(probe.scalar(0, x), 1.0 / x) <= 1.0
    assert _ulps(probe.scalar(1, x), (1.0 / np.sqrt(x.astype(np.longdouble))).astype(np.float64)) <= 2.0
    assert _ulps(probe.scalar(2, x), np.sqrt(x)) <= 1.0


def test_double_roots_and_reciprocals_at_the_ends(probe):
    x = np.array([0.0, 5e-324, 1e-310, 6e-309, TINY64, np.finfo(np.float64).max, np.inf, np.nan, -1.0])
    with np.errstate(all="ignore"):
        np.testing.assert_allclose(probe.scalar(2, x), np.sqrt(x), rtol=2.3e-16)
        got, want = probe.scalar(0, x), 1.0 / x
    np.testing.assert_allclose(got, want, rtol=2.3e-16)


def test_float_reciprocals_and_roots(probe):
    # the hardware's approximations: 1 ulp for the reciprocal, 2 for x^-1/2 and the root
    x = _sweep(-125, 125).astype(np.float32)
    v = x.astype(np.float64)
    for op, want, bar in ((7, 1.0 / v, 1.0), (8, np.sqrt(v), 2.0), (9, 1.0 / np.sqrt(v), 2.0)):
        err = np.abs(probe.scalar(op, v) - want) / np.spacing(want.astype(np.float32)).astype(np.float64)
        assert err.max() <= bar + 0.5, (op, err.max())
    ends = np.array([0.0, 1e-45, 1e-40, 5e-39, TINY32, np.finfo(np.float32).max, np.inf, np.nan, -1.0], dtype=np.float32)
    with np.errstate(all="ignore"):
        np.testing.assert_allclose(probe.scalar(8, ends.astype(np.float64)), np.sqrt(ends), rtol=3e-7)
        np.testing.assert_allclose(probe.scalar(7, ends.astype(np.float64)), np.float32(1.0) / ends, rtol=3e-7, atol=2e-45)


def test_conversions_and_predicates(probe):
    x = np.concatenate([_sweep(-200, 200), _sweep(-1022, 1022, seed=1)])
    x = np.concatenate([x, -x, [0.0, -0.0, 5e-324, -5e-324, TINY64, np.inf, -np.inf]])
    big, low = np.abs(x) >= 2.0 ** 128, np.abs(x) < TINY32
    cut = (np.ascontiguousarray(x).view(np.int64) & ~np.int64((1 << 29) - 1)).view(np.float64)  # towards zero
    want = np.where(big, np.copysign(np.finfo(np.float32).max, x), np.where(low, np.copysign(0.0, x), cut))
    assert np.array_equal(probe.scalar(3, x), want)
    f = want[~big]
    assert np.array_equal(probe.scalar(4, f), f)
    assert np.array_equal(probe.scalar(4, np.array([1e-45, -1e-40, 0.0])), np.zeros(3))
    y = np.append(x, np.nan)
    with np.errstate(invalid="ignore"):
        bits = (y > 0) * 1 + (y >= 0) * 2 + np.signbit(y) * 4
    assert np.array_equal(probe.scalar(5, y), bits)
    y = x[np.isfinite(x)]
    want = np.where(np.abs(y) >= 8.0 * TINY64, y / 8.0, 0.0)
    assert np.array_equal(probe.scalar(6, y), want)


def _star(g, v):
    """p* - p_L, u* and rho* - rho_K by Newton in long double, from p_R - p_L and u_R - u_L as given."""
    rl, ul, pl, rr, ur, pr, dP, dU = v.astype(np.longdouble)
    g = np.longdouble(g)
    one, half = np.longdouble(1), np.longdouble(0.5)

    def side(r, p, y):
        x, c = y / p, np.sqrt(g * p / r)
        al = (g + one) / (2 * g)
        f = np.where(x > 0, x * c / g / np.sqrt(one + al * x),
                     2 * c / (g - one) * np.expm1((g - one) / (2 * g) * np.log1p(x)))
        fd = np.where(x > 0, (one + half * al * x) / (one + al * x) ** np.longdouble(1.5),
                      np.exp((-(g + one) / (2 * g)) * np.log1p(x))) / (r * c)
        be = (g - one) / (2 * g)
        h = np.where(x > 0, x / g / (one + be * x), np.expm1(np.log1p(x) / g))
        return f, fd, r * h

    d = np.zeros_like(rl)
    for _ in range(8):
        fl, dl, hl = side(rl, pl, d)
        fr, dr, hr = side(rr, pr, d - dP)
        step = (fl + fr + dU) / (dl + dr)
        d = d - step
    fl, dl, hl = side(rl, pl, d)
    fr, dr, hr = side(rr, pr, d - dP)
    us = ul - fl
    left = us >= 0
    return d, us, np.where(left, hl, hr), left, fl, fr


@pytest.mark.parametrize("scale", (0, -66, -400, 300))
@pytest.mark.parametrize("gamma", (1.4, 5.0 / 3.0))
@pytest.mark.parametrize("jump", (1e-30, 1e-17, 1e-12, 1e-9, 1e-6, 1e-4, 1e-3))
def test_star_departures(probe, jump, gamma, scale):
    """p* - p_L, u* and rho* - rho_K of departures `jump` of the state: within 16 roundings of the larger
    jump that they come from, as the perturbation forms hand them on.  A side takes a reciprocal, a
    root, a sum of five terms and three products; the two sides and the last correction add up to about
    ten roundings."""
    rng = np.random.default_rng(9)
    n = 1500
    base = 2.0 ** scale
    c = np.sqrt(gamma * 1.3 / 0.7)
    n_ = lambda: rng.uniform(-1.0, 1.0, n) * 10.0 ** rng.uniform(-3.0, 0.0, n)  # noqa: E731
    dpl, dpr, dul, dur = 1.3 * jump * n_(), 1.3 * jump * n_(), c * jump * n_(), c * jump * n_()
    rl, rr = 0.7 * (1.0 + 0.5 * n_()), 0.7 * (1.0 + 0.5 * n_())
    v = np.stack([rl * base, dul, (1.3 + dpl) * base, rr * base, dur, (1.3 + dpr) * base, (dpr - dpl) * base, dur - dul])
    kind, d, us, drho, fl, fr = probe.near(gamma, v)
    assert (kind >= 3).all(), np.unique(kind)
    D, US, H, left, FL, FR = _star(gamma, v)
    eps = 16 * 2.0 ** -53
    J = np.maximum(np.abs(D), np.abs(D - v[6]))
    V = np.maximum(np.abs(FL), np.abs(FR)) + np.maximum(np.abs(dul), np.abs(dur))
    assert (np.abs(d - D) / J).max() <= eps, float((np.abs(d - D) / J).max())
    clear = np.abs(US) > eps * V  # beside it the side is a matter of rounding
    assert (np.abs(us - US) / V)[clear].max() <= eps, float((np.abs(us - US) / V)[clear].max())
    K = np.where(left, rl, rr) * base * (J / np.where(left, v[2], v[5]))
    assert (np.abs(drho - H) / K)[clear].max() <= eps
