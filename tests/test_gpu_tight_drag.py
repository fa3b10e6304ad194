"""Drag of dust that stops at once: Stokes numbers whose reciprocal leaves the state's range.

Where tau / t_s is beyond 1 / eps, 1 + tau / t_s is tau / t_s and the velocities
become equal whatever St is: the result at any smaller power of two is that at
2^-60 (float) or 2^-100 (double), bit for bit, in a disc of two scale heights
(the Epstein time grows with the gas's thinning).
"""
import math
from dataclasses import replace

import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_dust", (1, 2))
@pytest.mark.parametrize("law", (0, 1))
@pytest.mark.parametrize("form,powers", (("ROSSBI_FP32_PERT", (60, 100, 126, 130, 146)),
                                         ("ROSSBI_FP64", (100, 300, 1018, 1024, 1060))))
def test_small_stokes_numbers(form, powers, law, n_dust):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    w = replace(syn.scaled(syn.VORTEX, 20, 18, 24, steps=1), x0=(0.5, 0.0, -0.05), x1=(2.0, 2.0 * math.pi, 0.05),
                drag_law=law, n_dust=n_dust, dust_stokes_factors=(1.0, 0.25) if n_dust > 1 else ())
    out = []
    for k in powers:
        g = workloads.Grid(replace(w, stokes=2.0 ** -k), precision=getattr(R, form))
        s = g.initial_state()
        s[5:8] *= 1.01
        g.step(s, dt=1e-3)
        assert g.take_status() == R.ROSSBI_OK, k
        out.append(s)
        g.close()
    for k, s in zip(powers[1:], out[1:]):
        assert torch.equal(s, out[0]), k
