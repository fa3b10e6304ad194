"""The adjoint's flux kernel on axes that end at and beside the ends of its
lines: 12 cells a narrow line, 28 a wide one, each axis by itself.

The transpose identity <lambda, J delta> = <J^T lambda, delta> with J from the
oracle, to 1e-12 of the sum of the magnitudes: sums of some 10^4 to 10^5 terms
rounded at 1e-16 each, while one edge cell left out or taken twice is 1e-5 of it.
"""
import numpy as np
import pytest

import oracle
import synthetic as syn
from tests.parity import jitter

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", (syn.BC_OUTFLOW, syn.BC_PERIODIC), ids=("outflow", "periodic"))
@pytest.mark.parametrize("n", ((28, 27, 26), (56, 5, 29), (25, 28, 12), (12, 57, 25), (13, 24, 28)), ids=str)
def test_transpose_identity_at_line_ends(n, bc):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    from tests.test_gpu_parity import _box, _smooth_state
    w = _box(n, n_dust=1, stokes=0.07, bc=bc)
    o = oracle.Oracle(w)
    rng = np.random.default_rng(sum(n))
    E = jitter(_smooth_state(w, 9), w.gamma, rng, 1e-3)
    dt = o.cfl_dt(E)
    scale = np.abs(E).mean(axis=(1, 2, 3), keepdims=True)
    lam = rng.standard_normal(E.shape) / scale
    delta = rng.standard_normal(E.shape) * scale
    _, t = o.step_tlm(E, delta, dt)
    g = workloads.Grid(w, precision=R.ROSSBI_FP64)
    adj = torch.empty(E.shape, dtype=torch.float64, device="cuda")
    g.adjoint_step(torch.from_numpy(E).cuda(), dt, torch.from_numpy(lam).cuda(), adj)
    assert g.take_status() == R.ROSSBI_OK
    lhs, rhs = float((lam * t).sum()), float((adj.cpu().numpy() * delta).sum())
    g.close()
    assert abs(lhs - rhs) <= 1e-12 * float(np.abs(lam * t).sum()), (lhs, rhs)
