"""The FP32 stage kernel's two block shapes: one wide block per SM up to three
tiles per SM, two narrow ones beyond.

A state repeated along the periodic axis steps to the repeated result, bit for
bit: a tile's arithmetic and the order of its sums do not depend on the block.
152 SMs: 228 and 456 tiles take wide blocks, 684 and 912 narrow ones.
"""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_dust", (0, 1))
@pytest.mark.parametrize("recon", (syn.RECON_CONSERVATIVE, syn.RECON_PRIMITIVE), ids=("conservative", "primitive"))
def test_repeated_state_same_bits(recon, n_dust):
    import torch
    from paper_2207_04252_gb300 import rossbi as R
    from paper_2207_04252_gb300 import workloads
    from tests.test_gpu_parity import _smooth_state
    nr, nth, nz = 40, 114, 24
    out = {}
    for times in (1, 2, 3, 4):
        w = syn.Workload(name="box", geometry=syn.GEOM_BOX, nr=nr, nth=nth * times, nz=nz, x0=(0.0, 0.0, 0.0),
                         x1=(nr / 32, nth * times / 32, nz / 32), bc_lo=(syn.BC_OUTFLOW, 0, 0),
                         bc_hi=(syn.BC_OUTFLOW, 0, 0), ic="none", steps=0, omega_frame=0.0, n_dust=n_dust,
                         stokes=0.07, recon=recon)
        g = workloads.Grid(w, precision=R.ROSSBI_FP32_PERT)
        one = _smooth_state(syn.Workload(**{**w.__dict__, "nth": nth}), g.nf)
        one[3] += 2.0 * (np.arange(nr) > 25)  # a strong jump: faces of the general solver
        s = torch.from_numpy(np.tile(one, (1, 1, times, 1))).to("cuda", g.dtype).contiguous()
        nxt = g.step(s, dt=1e-3, want_next_dt=True)
        g.step(s, dt=1e-3)
        assert g.take_status() == R.ROSSBI_OK
        out[times] = nxt, s.cpu().numpy()
        g.close()
    for times in (2, 3, 4):
        assert out[times][0] == out[1][0], times
        assert np.array_equal(out[times][1], np.tile(out[1][1], (1, 1, times, 1))), times
