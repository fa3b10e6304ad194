"""Rounding of the arithmetic that the kernels write themselves, function by function.

The Riemann solution near p_K, and its departures from the side states, against
a Newton iteration in long double.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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

        def near(self, gamma, x):
            return self._run(lib.probe_near, ctypes.c_double(gamma), x=x, rows=6)

    return Probe()


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
