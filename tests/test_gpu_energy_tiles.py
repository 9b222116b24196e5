"""The energy kernels where their normalisers' references differ inside one
tile, against the FP64 oracle: half of the volume is smooth (every output
changes to the reference 0 after its centre column), half is noise whose best
matches lie about 90 to 180 binary orders down (running references stay), on
sizes that are no multiple of a tile.

Tolerance: a weight's exponent is a sum of 27 or 125 squares whose rounding is
about 1.5 half-ulps rms; at 170 binary orders that is 170 ln 2 * 9e-8 = 1.1e-5
per normalised weight and 1.5e-5 for the two normalisers of a gradient term, so
2e-5 on the gradient in relative L2; the energy sums them with either sign
(1e-5)."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, M, amp", [(1, 1, 0.12), (1, 2, 0.12), (2, 1, 0.06)])
def test_energy_mixed_references(d, M, amp):
    import oracle
    oracle.build()
    geom = synth.make_geometry(nx=45, ny=21, nz=10, dx=1.0, nu=48, nv=14, du=1.2, sad=200, sdd=300, n_phases=2,
                               views_per_phase=[3, 2], angle_offset=0.1)
    G, OG = tnlm.Geometry(geom), oracle.Geometry(geom)
    a = synth.smooth_volume((2, 10, 21, 45), 940)
    a[:, :, :10] += synth.uniform((2, 10, 10, 45), 941, 0.0, amp)
    f = synth.uniform(a.shape, 942, 0.0, 0.04)
    y = synth.uniform(G.proj_shape, 943, 0.0, 0.3)
    E_ref, g_ref = oracle.energy_grad(OG, y, f, a, d, M, 0.02, 1e-12)
    E, g = tnlm.tnlm_energy_grad(G, *(torch.from_numpy(t.astype(np.float32)).cuda() for t in (y, f, a)),
                                 tnlm.Params(d=d, M=M, h=0.02, mu=1e-12))
    assert E == pytest.approx(E_ref, rel=1e-5)
    assert np.linalg.norm(g.cpu().numpy() - g_ref) <= 2e-5 * np.linalg.norm(g_ref)
