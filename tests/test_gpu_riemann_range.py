"""The Riemann solution near p_K against the oracle over its range and past its edges.

Random states on a ragged periodic Box whose jumps are a times the state, so
that |p*/p_K - 1| runs from small through the series' limit (1/32) to strong
waves, at Mach numbers inside, at the edges of and beyond the sonic band, for
two gamma and every form.  One step is compared element-wise; the bar is the
project's own for element-wise parity, 20 times the oracle's response to a
perturbation of the input by its rounding (1e-15 in double, 6e-8 in float),
and at least 1e-13 (1e-5).  The adjoint's bar is the transpose identity at
1e-12, on jumps of 2e-3 and more as the identity needs both sides on the same
limiter branches.
"""
import numpy as np
import pytest

import oracle
import synthetic as syn
from tests.parity import elementwise

pytestmark = pytest.mark.gpu

AMPLITUDES = (1e-5, 2e-3, 0.01, 0.03, 0.1)
MACHS = ((0.0, 0.0, 0.0), (0.97, -1.02, 1.0), (-1.06, 1.12, -0.9), (3.0, -8.0, 0.3))


def _workload(gamma):
    nr, nth, nz = 61, 13, 9
    return syn.Workload(name="range", geometry=syn.GEOM_BOX, nr=nr, nth=nth, nz=nz, x0=(0.0, 0.0, 0.0),
                        x1=(1.0, nth / nr, nz / nr), bc_lo=(0, 0, 0), bc_hi=(0, 0, 0), ic="sod", steps=1, gamma=gamma,
                        omega_frame=0.0)


def _state(w, a, mach, seed):
    rng = np.random.default_rng(seed)
    shape = (w.nz, w.nth, w.nr)
    noise = lambda: rng.uniform(-1.0, 1.0, shape)  # noqa: E731
    rho, p = 0.7 * (1.0 + a * noise()), 1.3 * (1.0 + a * noise())
    c = np.sqrt(w.gamma * 1.3 / 0.7)
    v = [c * (m + a * noise()) for m in mach]
    E = np.zeros((5,) + shape)
    E[:3] = [rho * q for q in v]
    E[3] = p / (w.gamma - 1.0) + 0.5 * rho * sum(q * q for q in v)
    E[4] = rho
    return E


@pytest.mark.parametrize("gamma", (1.4, 5.0 / 3.0))
@pytest.mark.parametrize("a", AMPLITUDES)
def test_step_against_oracle(a, gamma):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = _workload(gamma)
    o = oracle.Oracle(w)
    rng = np.random.default_rng(5)
    for prec, eps, least in ((R.ROSSBI_FP64, 1e-15, 1e-13), (R.ROSSBI_FP64_PERT, 1e-15, 1e-13),
                             (R.ROSSBI_FP32_PERT, 6e-8, 1e-5)):
        g = workloads.Grid(w, precision=prec)
        for k, mach in enumerate(MACHS):
            s = torch.from_numpy(_state(w, a, mach, 7 * k + 1)).to("cuda", g.dtype)
            E = s.cpu().numpy().astype(np.float64)
            dt = 0.8 * o.cfl_dt(E)
            ref = o.step(E, dt)
            moved = o.step(E * (1.0 + eps * rng.uniform(-1.0, 1.0, E.shape)), dt)
            own, _ = zip(*elementwise(moved, ref).values())
            g.step(s, dt=dt)
            assert g.take_status() == 0 and o.take_status() == 0
            err = elementwise(g.full_state(s), ref)
            for (v, at), bar in zip(err.values(), own):
                assert v <= max(least, 20.0 * bar), (prec, mach, v, bar, at)


@pytest.mark.parametrize("gamma", (1.4, 5.0 / 3.0))
@pytest.mark.parametrize("a", AMPLITUDES[1:])
def test_adjoint_against_oracle(a, gamma):
    import torch
    from paper_2207_04252_gb300 import workloads
    w = _workload(gamma)
    o = oracle.Oracle(w)
    g = workloads.Grid(w)
    for k, mach in enumerate(MACHS):
        rng = np.random.default_rng(100 + k)
        E = _state(w, a, mach, 3 * k + 2)
        dt = 0.8 * o.cfl_dt(E)
        scale = np.abs(E).mean(axis=(1, 2, 3), keepdims=True) + 1e-30
        lam, delta = rng.standard_normal(E.shape) / scale, rng.standard_normal(E.shape) * scale
        _, t = o.step_tlm(E, delta, dt)
        out = torch.from_numpy(lam).cuda().contiguous()
        g.adjoint_step(torch.from_numpy(E).cuda().contiguous(), dt, out)
        lhs, rhs = float((lam * t).sum()), float((out.cpu().numpy() * delta).sum())
        assert g.take_status() == 0
        assert abs(lhs - rhs) <= 1e-12 * float(np.abs(lam * t).sum()), (mach, lhs, rhs)
