"""Infinite and not-a-number voxels in the projector.  A ray with a share in an
infinite voxel is infinite, not NaN, also where it enters or leaves that voxel
through a z plane; a ray without is what it is when the voxel holds 0
(relative L2 <= 1e-5, the FP32 target).  The shares are the FP64 oracle's
chords through the voxels; rays that graze one (chords up to 1e-3 mm) may fall
to either side."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = {
    "cubic": dict(nx=33, ny=35, nz=40, dx=1.0, nu=41, nv=65, du=1.3),
    "one_row_per_lane": dict(nx=31, ny=29, nz=17, dx=1.0, nu=37, nv=32, du=1.1),
    "thin_slices": dict(nx=24, ny=26, nz=90, dx=1.0, dz=0.1, nu=40, nv=70, du=1.2, dv=0.4),
}


@pytest.mark.parametrize("code", [102, 104, 108])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("name", list(CASES))
def test_rays_through_non_finite_voxels(ora, name, value, code):
    desc = synth.make_geometry(sad=300.0, sdd=450.0, angle_offset=0.13, cz=0.3, n_phases=2, views_per_phase=[3, 2], **CASES[name])
    G = tnlm.Geometry(desc)
    x = synth.uniform(G.vol_shape, 830)
    hit = (synth.uniform(G.vol_shape, 831) < 0.005).astype(np.float32)
    x[hit > 0] = 0.0
    chord = ora.project(ora.Geometry(desc), hit)
    tnlm.tnlm_set_launch_shapes(G, code, 8, 4)
    assert tnlm.tnlm_get_launch_shapes(G)["projector_rows"] == code
    plain = tnlm.tnlm_project(G, torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    x[hit > 0] = value
    got = tnlm.tnlm_project(G, torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    through, clear = chord > 1e-3, chord == 0.0
    assert through.sum() > 100 and clear.sum() > 100
    assert np.array_equal(got[through], np.full(through.sum(), value), equal_nan=True)
    assert np.isfinite(got[clear]).all()
    assert np.linalg.norm(got[clear] - plain[clear]) <= 1e-5 * np.linalg.norm(plain[clear])
