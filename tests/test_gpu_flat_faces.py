"""Cells whose parabola is not physical: both their faces take the flat state, in every form.

Density and pressure vary by factors of 30 from cell to cell at Mach numbers up
to 4, so that the pressure of the conservative parabola, a difference of
energies, is negative in many cells.  One step against the oracle, at 20 times
the oracle's own response to a rounding of the input and at least 1e-12 (1e-4 in
float, where the pressure is the difference of numbers 30 times its size).
"""
import numpy as np
import pytest

import oracle
import synthetic as syn
from tests.parity import elementwise
from tests.test_gpu_riemann_range import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,eps,least", (("ROSSBI_FP64", 1e-15, 1e-12), ("ROSSBI_FP64_PERT", 1e-15, 1e-12),
                                            ("ROSSBI_FP32_PERT", 6e-8, 1e-4)))
def test_rough_state(form, eps, least):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = _workload(1.4)
    rng = np.random.default_rng(21)
    shape = (w.nz, w.nth, w.nr)
    rho, p = 30.0 ** rng.uniform(-1.0, 0.0, shape), 30.0 ** rng.uniform(-1.0, 0.0, shape)
    v = 4.0 * np.sqrt(1.4 * p / rho) * rng.uniform(-1.0, 1.0, (3,) + shape) / np.sqrt(3.0)
    E = np.zeros((5,) + shape)
    E[:3], E[3], E[4] = rho * v, p / 0.4 + 0.5 * rho * (v * v).sum(0), rho
    g = workloads.Grid(w, precision=getattr(R, form))
    s = torch.from_numpy(E).to("cuda", g.dtype)
    E = s.cpu().numpy().astype(np.float64)
    o = oracle.Oracle(w)
    dt = 0.1 * o.cfl_dt(E)
    ref = o.step(E, dt)
    moved = o.step(E * (1.0 + eps * rng.uniform(-1.0, 1.0, E.shape)), dt)
    g.step(s, dt=dt)
    assert g.take_status() == 0 and o.take_status() == 0
    err, own = elementwise(g.full_state(s), ref), elementwise(moved, ref)
    for name in err:
        assert err[name][0] <= max(least, 20.0 * own[name][0]), (name, err[name], own[name])
    g.close()
