"""CFL steps and drag where squares leave the normal range of the state's precision.

A Gaussian velocity pulse in a gas at rest has every speed below its peak in
its tails, among them those whose square is subnormal (10^-23 ... 10^-19 in
float, 10^-162 ... 10^-154 in double).  Such cells do not bound the step: the
gas's sound speed does, as in the oracle.  The bar is the rounding of the step
itself, some ten operations: 1e-12 in double, 1e-5 in float (with the state's
own rounding after a step).  An infinite energy still means a step of zero.

In a deep atmosphere pressure times density of the top is below the normal
range, while the sound speed is an ordinary number: the Epstein stopping time
there is finite (rho c_s underflows only with the density itself).
"""
from dataclasses import replace

import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu

FORMS = (("ROSSBI_FP64", 1e-12), ("ROSSBI_FP64_PERT", 1e-12), ("ROSSBI_FP32_PERT", 1e-5))


def _pulse(n_dust, axis):
    """A resting Box of 250 x 12 x 6 cells with the pulse along x, and dust that carries it alone."""
    nr, nth, nz = 250, 12, 6
    w = syn.Workload(name="pulse", geometry=syn.GEOM_BOX, nr=nr, nth=nth, nz=nz, x0=(0.0, 0.0, 0.0),
                     x1=(1.0, nth / nr, nz / nr), bc_lo=(syn.BC_OUTFLOW, 0, 0), bc_hi=(syn.BC_OUTFLOW, 0, 0),
                     ic="none", steps=1, omega_frame=0.0, n_dust=n_dust, stokes=0.07)
    x = (np.arange(nr) + 0.5) / nr
    u = 0.1 * np.exp(-0.5 * ((x - 0.5) / 0.0165) ** 2)
    E = np.zeros((w.nfields, nz, nth, nr))
    E[4], E[axis], E[3] = 1.0, u, 2.5 + 0.5 * u * u
    if n_dust:
        E[8], E[5 + axis] = 0.01, 0.03 * u
    return w, E


@pytest.mark.parametrize("axis", (0, 1))
@pytest.mark.parametrize("n_dust", (0, 1))
@pytest.mark.parametrize("form,bar", FORMS)
def test_step_of_a_velocity_pulse(form, bar, n_dust, axis):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w, E = _pulse(n_dust, axis)
    g = workloads.Grid(w, precision=getattr(R, form))
    s = torch.from_numpy(E).to("cuda", g.dtype)
    o = oracle.Oracle(w)
    E = g.full_state(s)
    want = o.cfl_dt(E)
    dt = g.cfl_dt(s)
    assert abs(dt - want) <= bar * want, (dt, want)
    E = o.step(E, want)
    nxt = g.step(s, dt=want, want_next_dt=True)
    assert abs(nxt - o.cfl_dt(E)) <= bar * want, (nxt, o.cfl_dt(E))
    g.step(s)  # on the device-resident step
    assert np.abs(g.full_state(s) - o.step(E, o.cfl_dt(E))).max() <= 10 * bar
    g.close()


@pytest.mark.parametrize("form,bar", FORMS)
def test_infinite_energy_stops_the_clock(form, bar):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w, E = _pulse(0, 0)
    E[3, 2, 5, 100] = np.inf
    g = workloads.Grid(w, precision=getattr(R, form))
    assert g.cfl_dt(torch.from_numpy(E).to("cuda", g.dtype)) == 0.0
    g.close()


# Aspect ratio and half-height of the mesh: at its top the density is e^-68 (float: 10^-30) or e^-536 (double:
# 10^-233) of the midplane's, and the pressure 10^-3 (10^-6) times that.
@pytest.mark.parametrize("n_dust", (1, 2))
@pytest.mark.parametrize("form,h,top", (("ROSSBI_FP32_PERT", 0.05, 0.42), ("ROSSBI_FP64_PERT", 0.002, 0.044)))
def test_epstein_drag_in_a_deep_atmosphere(form, h, top, n_dust):
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = replace(syn.scaled(syn.VORTEX, 16, 12, 160, steps=1), x0=(0.95, 0.0, -top), x1=(1.05, 2.0 * np.pi, top),
                disc=(1.0, -0.5, 0.5 * h * h, -1.0), vortex_amp=0.0, drag_law=1, n_dust=n_dust,
                dust_stokes_factors=(1.0, 0.3) if n_dust > 1 else ())
    g = workloads.Grid(w, precision=getattr(R, form))
    s = g.initial_state()
    # where the drag is strong (the midplane) the dust stays with the gas; at the top it falls freely, dw = g_z dt
    dt = 0.25 * g.cfl_dt(s)
    g.step(s, dt=dt)
    E = g.full_state(s)
    assert np.isfinite(E).all()
    r, z = g.centres(0)[None, :], g.centres(2)[[0, -1], None]
    fall = -dt * z / (r * r + z * z) ** 1.5
    for b in range(5, 5 + 4 * n_dust, 4):
        v = E[b + 2][[0, -1]] / E[b + 3][[0, -1]]
        # the free fall's own change over the step is dt^2 Omega^2 ~ 1e-6 of it, the outflow's the CFL number
        assert np.abs(v / fall[:, None, :] - 1.0).max() <= 0.05
    g.close()
