"""Units of the mass: the state times a power of two steps to the result times that power, bit for bit.

Density, pressure and energy scale, velocities and the step do not, and every
operation on them commutes with a power of two while nothing underflows, so
there is no rounding to allow for.  2^-100 brings pressures to 10^-30, 2^100
and 2^-300 beyond float's range.
"""
from dataclasses import replace

import numpy as np
import pytest

import synthetic as syn
from tests.test_gpu_riemann_range import _state, _workload

pytestmark = pytest.mark.gpu

POWERS = (-66, -100, -300, 100)


@pytest.mark.parametrize("a", (1e-9, 1e-5, 0.01))
@pytest.mark.parametrize("form", ("ROSSBI_FP64", "ROSSBI_FP64_PERT"))
def test_box(form, a):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = _workload(1.4)
    g = workloads.Grid(w, precision=getattr(R, form))
    for mach in ((0.0, 0.0, 0.0), (0.6, -0.3, 0.97), (-1.5, 0.4, 0.1)):
        E = torch.from_numpy(_state(w, a, mach, 11)).cuda()
        one, lam = E.clone(), torch.from_numpy(np.random.default_rng(3).standard_normal(E.shape)).cuda()
        nxt = g.step(one, dt=2e-3, want_next_dt=True)
        if form == "ROSSBI_FP64":
            adj = torch.empty_like(E)
            g.adjoint_step(E, 2e-3, lam, adj)
        for k in POWERS:
            s = E * 2.0 ** k
            assert g.step(s, dt=2e-3, want_next_dt=True) == nxt, k
            assert torch.equal(s * 2.0 ** -k, one), k
            if form == "ROSSBI_FP64":
                out = torch.empty_like(E)
                g.adjoint_step(E * 2.0 ** k, 2e-3, lam, out)
                assert torch.equal(out, adj), k
    g.close()


@pytest.mark.parametrize("recon", (syn.RECON_CONSERVATIVE, syn.RECON_PRIMITIVE), ids=("conservative", "primitive"))
def test_disc_departures(recon):
    """The perturbation form's disc, bi-fluid, with departures down to 1e-12 of the equilibrium."""
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = replace(syn.scaled(syn.VORTEX, 30, 24, 26, steps=1), recon=recon, vortex_amp=1e-9)
    s0, bs, t0, bt = w.disc
    one = nxt = None
    for k in (0,) + POWERS:
        g = workloads.Grid(replace(w, disc=(s0 * 2.0 ** k, bs, t0, bt)), precision=R.ROSSBI_FP64_PERT)
        s = g.initial_state()
        dt = g.step(s, dt=1e-3, want_next_dt=True)
        s *= 2.0 ** -k
        if one is None:
            one, nxt = s, dt
        assert dt == nxt and torch.equal(s, one), k
        g.close()
