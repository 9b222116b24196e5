"""The table walker takes 4, 8 or 16 rows of several columns per warp on
detectors of few rows and volumes that few rows see: a row's projection is the
same to the bit as among the rows of a taller detector (64 rows per warp), and
agrees with the slab walker (relative L2 <= 1e-5); so do the residuals of a
gradient step, whose block sums follow the same tiles."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


def scan(nx, nz, nu, nv, **kw):
    views = 5000 // nu + 1  # more than one wave of warps, below which there are always 32 or 64 rows
    d = dict(dx=1.0, du=1.3, dv=1.1, sad=300.0, sdd=450.0, angle_offset=0.13, n_phases=2, views_per_phase=[views - 2, 2])
    d.update(kw)
    return tnlm.Geometry(synth.make_geometry(nx=nx, ny=nx - 3, nz=nz, nu=nu, nv=nv, **d))


# narrow and wide blocks against the columns, an empty last warp, rows beyond the volume, a volume off the axis
@pytest.mark.parametrize("nx,nz,nu,kw", [(33, 40, 41, {}), (21, 30, 7, {}), (40, 12, 130, dict(u_off=9.0)),
                                         (25, 60, 65, dict(v_off=0.55, cz=3.0))])
@pytest.mark.parametrize("nv", [1, 2, 3, 5, 8, 9, 13, 16, 17])
def test_rows_equal_those_of_a_taller_detector(nv, nx, nz, nu, kw):
    few, tall = scan(nx, nz, nu, nv, **kw), scan(nx, nz, nu, nv + 64, **kw)
    x = torch.from_numpy(synth.uniform(few.vol_shape, 850)).cuda()
    want = tnlm.tnlm_project(tall, x)[:, 32:32 + nv]
    for code in (102, 104, 108):
        tnlm.tnlm_set_launch_shapes(few, code, 8, 4)
        assert torch.equal(tnlm.tnlm_project(few, x), want)
    tnlm.tnlm_set_launch_shapes(few, 4, 8, 4)
    slab = tnlm.tnlm_project(few, x).double()
    assert float((want.double() - slab).norm()) <= 1e-5 * float(slab.norm())


@pytest.mark.parametrize("nz,cz", [(1, 0.0), (3, 0.0), (6, 9.0), (14, -4.0)])
def test_few_slices_under_many_rows(nz, cz):
    G = scan(50, nz, 70, 150, cz=cz)
    x = torch.from_numpy(synth.uniform(G.vol_shape, 851)).cuda()
    y = torch.from_numpy(synth.uniform(G.proj_shape, 852)).cuda()
    got, p = [], tnlm.Params(d=1, M=1, h=0.02, mu=1.0, tau=1e-4)
    for code in (4, 102, 104, 108):
        tnlm.tnlm_set_launch_shapes(G, code, 8, 4)
        g = torch.empty_like(x)
        report = tnlm.tnlm_p1(G, y, x, g, p, report=True)
        got.append((tnlm.tnlm_project(G, x).double(), g.double(), float(np.asarray(report[-1]).ravel()[0])))
    for proj, g, norm in got[1:]:
        assert float((proj - got[0][0]).norm()) <= 1e-5 * float(got[0][0].norm())
        assert float((g - got[0][1]).norm()) <= 1e-5 * float(got[0][1].norm())
        assert abs(norm - got[0][2]) <= 1e-5 * got[0][2]
