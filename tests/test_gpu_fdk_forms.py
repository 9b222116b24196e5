"""The tiles of the FDK filter (64 rows x 256 outputs, 16 x 64) and the runs of
its backprojection (8 voxels per thread, 1) give the same bits: a phase is what
it is alone, however many phases share the call and choose its forms.  The
large call is checked against the FP64 oracle (relative L2 <= 1e-5; without
noise, as pixel coordinates of long rows carry ~nu 2^-24 pixels of rounding)."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,nu,nv,phases", [(20, 7, 510, 80, 50), (20, 7, 395, 90, 100), (60, 9, 90, 24, 40), (64, 31, 65, 24, 9)])
def test_a_phase_alone_equals_a_phase_of_many(ora, nx, nz, nu, nv, phases):
    def desc(n):
        return synth.make_geometry(nx=nx, ny=nx - 2, nz=nz, dx=1.0, nu=nu, nv=nv, du=2.4 * nx / nu, dv=2.0 * nz / nv + 0.1,
                                   sad=300.0, sdd=450.0, n_phases=n, views_per_phase=[5] * n, angle_offset=0.11)

    one, many = desc(1), desc(phases)
    many["angles"] = np.tile(one["angles"], phases)
    y = synth.analytic_projections(one, [[((0.5, -0.5, 0.2), (0.2 * nx, 0.15 * nx, 0.4 * nz), 0.02)]]).numpy().astype(np.float32)
    alone = tnlm.tnlm_fdk(tnlm.Geometry(one), torch.from_numpy(y).cuda())
    got = tnlm.tnlm_fdk(tnlm.Geometry(many), torch.from_numpy(np.tile(y, (phases, 1, 1))).cuda())
    assert all(torch.equal(got[i], alone[0]) for i in range(phases))
    ref = ora.fdk(ora.Geometry(one), y)
    assert np.linalg.norm(alone.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)
