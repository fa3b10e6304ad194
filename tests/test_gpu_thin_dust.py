"""Dust of zero, subnormal and smallest normal density beside ordinary dust.

The reciprocal of a subnormal density may overflow; a species has mass where
its density is a normal number of the state's precision.  Below that the gas
and the step are those without the species, and everything stays finite.
"""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu

THIN = {"ROSSBI_FP32_PERT": (0.0, 1e-42, 5e-39, 1.1e-38, 2e-38), "ROSSBI_FP64": (0.0, 5e-320, 4e-309, 1.1e-308, 3e-308),
        "ROSSBI_FP64_PERT": (0.0, 5e-320, 4e-309, 1.1e-308, 3e-308)}


@pytest.mark.parametrize("n_dust", (1, 2))
@pytest.mark.parametrize("form", sorted(THIN))
def test_thin_dust(form, n_dust):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    nr, nth, nz = 40, 13, 9
    args = dict(name="thin", geometry=syn.GEOM_BOX, nr=nr, nth=nth, nz=nz, x0=(0.0, 0.0, 0.0),
                x1=(1.0, nth / nr, nz / nr), bc_lo=(0, 0, 0), bc_hi=(0, 0, 0), ic="none", steps=1, omega_frame=0.0,
                stokes=0.07)
    rng = np.random.default_rng(4)
    E = np.zeros((5 + 4 * n_dust, nz, nth, nr))
    v = 0.2 * rng.standard_normal((3, nz, nth, nr))
    E[4] = 1.0 + 0.1 * rng.standard_normal(v[0].shape)
    E[:3] = E[4] * v
    E[3] = 2.5 + 0.5 * E[4] * (v ** 2).sum(0)
    rd = np.array(THIN[form])[rng.integers(0, len(THIN[form]), v[0].shape)]
    for b in range(5, E.shape[0], 4):
        E[b + 3] = rd
        E[b:b + 3] = rd * (v + 0.5)
    alone = workloads.Grid(syn.Workload(**args, n_dust=0), precision=getattr(R, form))
    g = workloads.Grid(syn.Workload(**args, n_dust=n_dust,
                                    dust_stokes_factors=(1.0, 0.3) if n_dust > 1 else ()), precision=getattr(R, form))
    s = torch.from_numpy(E).to("cuda", g.dtype)
    gas = s[:5].clone().contiguous()
    rel = 1e-14 if form == "ROSSBI_FP64" and n_dust > 1 else 0.0
    dt, dt_gas = g.cfl_dt(s), alone.cfl_dt(gas)
    # dust slower than its cell's fastest gas wave does not bound the step: |v_d| <= |v_g| + 0.87 < |v_g| + c
    assert dt == dt_gas
    for _ in range(3):
        dt, dt_gas = g.step(s, dt=dt, want_next_dt=True), alone.step(gas, dt=dt_gas, want_next_dt=True)
        assert abs(dt - dt_gas) <= rel * dt_gas
        assert torch.isfinite(s).all()
        assert float((s[:5] - gas).abs().max()) <= rel * float(gas.abs().max())
    assert g.take_status() == R.ROSSBI_OK and alone.take_status() == R.ROSSBI_OK
    if form == "ROSSBI_FP64" and n_dust == 1:
        lam, lam_gas = torch.ones_like(s), torch.ones_like(gas)
        lam[5:] = 0.0
        g.adjoint_step(s, dt, lam)
        alone.adjoint_step(gas, dt, lam_gas)
        assert torch.isfinite(lam).all()
    g.close()
    alone.close()
