"""The adjoint against central differences of the library's own step, where its limiter's and solver's branches are
decided by rounding: an isobaric state (the primitive option's pressure and velocity departures are rounding only) and
a disc whose cells meet equilibrium ghosts (the limited face state beside one is the equilibrium).

<lambda, (S(E + h d) - S(E - h d)) / 2h> = <J^T lambda, d>.  The differences lose 1e-16 / h of the state, h = 1e-8
(isobaric: along densities at fixed pressure and velocity, where the step is smooth) and 1e-9 (the disc, of noise
1e-3: a limiter branch changes within h in 1e-6 of its decisions).  The oracle's step and its tangent differ by 5e-11
and 2e-9 of the sum of the magnitudes in the same test; the bars are 1e-8 and 1e-6.
"""
from dataclasses import replace

import numpy as np
import pytest

import oracle
import synthetic as syn
from tests.parity import jitter

pytestmark = pytest.mark.gpu

RECONS = pytest.mark.parametrize("recon", (syn.RECON_CONSERVATIVE, syn.RECON_PRIMITIVE), ids=("conservative", "primitive"))


def _check(w, E, d, h, dt, bar, seed):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    g = workloads.Grid(w)
    lam = np.random.default_rng(seed).standard_normal(E.shape) / (np.abs(E).mean(axis=(1, 2, 3), keepdims=True) + 1e-30)

    def step(x):
        s = torch.from_numpy(x).cuda().contiguous()
        g.step(s, dt=dt)
        return s.cpu().numpy()

    t = (step(E + h * d) - step(E - h * d)) / (2.0 * h)
    out = torch.from_numpy(lam).cuda().contiguous()
    g.adjoint_step(torch.from_numpy(E).cuda().contiguous(), dt, out)
    assert g.take_status() == R.ROSSBI_OK
    g.close()
    lhs, rhs = float((lam * t).sum()), float((out.cpu().numpy() * d).sum())
    assert abs(lhs - rhs) <= bar * float(np.abs(lam * t).sum()), (lhs, rhs, float(np.abs(lam * t).sum()))


@RECONS
def test_isobaric_state(recon):
    nr, nth, nz = 40, 13, 9
    w = syn.Workload(name="isobaric", geometry=syn.GEOM_BOX, nr=nr, nth=nth, nz=nz, x0=(0.0, 0.0, 0.0),
                     x1=(1.0, nth / nr, nz / nr), bc_lo=(syn.BC_OUTFLOW, 0, 0), bc_hi=(syn.BC_OUTFLOW, 0, 0), ic="none",
                     steps=1, omega_frame=0.0, recon=recon)
    rng = np.random.default_rng(6)
    v, noise = (0.31, -0.17, 0.23), 1.0 + 0.1 * rng.standard_normal((nz, nth, nr))
    unit = np.array([*v, 0.5 * sum(q * q for q in v), 1.0])[:, None, None, None]
    E = unit * noise
    E[3] += 1.3 / 0.4
    _check(w, E, unit * rng.standard_normal(noise.shape), 1e-8, 5e-3, 1e-8, 8)


@RECONS
def test_disc_with_equilibrium_walls(recon):
    w = replace(syn.scaled(syn.VORTEX, 20, 18, 24, steps=1), recon=recon)
    o = oracle.Oracle(w)
    rng = np.random.default_rng(2)
    E = jitter(oracle.initial_state(o), w.gamma, rng, 1e-3)
    d = (jitter(E, w.gamma, rng, 1e-3) - E) / 1e-3
    _check(w, E, d, 1e-9, 0.5 * o.cfl_dt(E), 1e-6, 5)
