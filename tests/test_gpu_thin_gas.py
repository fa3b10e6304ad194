"""Gas at rest whose density is a subnormal number, as at the top of a deep atmosphere.

The quotients by it are ordinary numbers as long as 1 / rho is finite (rho above
2.9e-39 in float, 5.6e-309 in double), and an equilibrium stays what it is, to
the bit.  The disc here is hot in its units, so that its pressure stays normal
while the density does not.
"""
from dataclasses import replace

import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


def _disc(rho, recon):
    gm, h = 1e4, 0.05
    w = syn.scaled(syn.VORTEX, 20, 18, 12, steps=1)
    return replace(w, x0=(0.95, 0.0, -0.012), x1=(1.05, 2.0 * np.pi, 0.012), gm=gm, omega_frame=100.0, n_dust=0,
                   vortex_amp=0.0, recon=recon, disc=(rho * np.sqrt(np.pi) * h, -0.5, 0.5 * h * h * gm, -1.0))


RECONS = pytest.mark.parametrize("recon", (syn.RECON_CONSERVATIVE, syn.RECON_PRIMITIVE), ids=("conservative", "primitive"))


@RECONS
@pytest.mark.parametrize("form,rho", (("ROSSBI_FP32_PERT", 7e-39), ("ROSSBI_FP64", 1.2e-308), ("ROSSBI_FP64_PERT", 1.2e-308)))
def test_equilibrium_stays(form, rho, recon):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    g = workloads.Grid(_disc(rho, recon), precision=getattr(R, form))
    tiny = np.finfo(np.float32 if g.dtype == torch.float32 else np.float64).tiny
    assert (g.equilibrium()[4] < tiny).all() and (g.equilibrium()[3] > tiny).all()
    s = g.initial_state()
    E = s.clone()
    dt = g.cfl_dt(s)
    assert 0.0 < dt < 1.0
    g.step(s, dt=dt)
    assert g.take_status() == R.ROSSBI_OK
    assert torch.equal(s, E)
    g.close()
