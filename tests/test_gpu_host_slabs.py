"""rossbi_step_host in slabs along z: the same bits as rossbi_step.

200 x 240 x 40 cells are seven layers of 600 tiles, which the library cuts into
six slabs on 152 SMs; the last layer is ragged.
"""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


def _box():
    nr, nth, nz = 200, 240, 40
    return syn.Workload(name="box", geometry=syn.GEOM_BOX, nr=nr, nth=nth, nz=nz, x0=(0.0, 0.0, 0.0),
                        x1=(1.0, nth / nr, nz / nr), bc_lo=(0, 0, syn.BC_OUTFLOW), bc_hi=(0, 0, syn.BC_OUTFLOW),
                        ic="sod", steps=1, omega_frame=0.0)


@pytest.mark.parametrize("pinned", (True, False))
@pytest.mark.parametrize("form", ("ROSSBI_FP64", "ROSSBI_FP32_PERT", "ROSSBI_FP64_PERT"))
@pytest.mark.parametrize("flow", ("vortex", "box"))
def test_same_bits_as_device_steps(flow, form, pinned):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = _box() if flow == "box" else syn.scaled(syn.VORTEX, 200, 240, 40, steps=2)
    g = workloads.Grid(w, precision=getattr(R, form))
    if flow == "box":
        rng = np.random.default_rng(1)
        rho = 1.0 + 0.01 * rng.standard_normal((w.nz, w.nth, w.nr))
        E = np.zeros((5,) + rho.shape)
        E[0:3] = 0.1 * rng.standard_normal(E[0:3].shape)
        E[3] = 2.5 + 0.5 * (E[0:3] ** 2).sum(0) / rho
        E[4] = rho
        s = torch.from_numpy(E).to("cuda", g.dtype)
    else:
        s = g.initial_state()
    h = torch.empty(s.shape, dtype=s.dtype, pin_memory=pinned).copy_(s).numpy()
    dt = dt_h = g.cfl_dt(s)
    for _ in range(2):
        dt_h = R.rossbi_step_host(g.h, h, dt=dt_h, dust=g.dust)
    for _ in range(2):
        dt = g.step(s, dt=dt, want_next_dt=True)
    assert dt == dt_h
    assert np.array_equal(h, s.cpu().numpy())
