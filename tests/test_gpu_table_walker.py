"""The table walker (32 rows of a detector column per warp) where it can go
wrong, against the slab walker on the same handle (both FP32 walkers of one
exact model: relative L2 <= 1e-5, the FP32 target): ragged rows and columns,
rows that enter or leave through the top and bottom or miss the volume,
several z planes in one xy cell, one slice, one row, a row in a face plane."""
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


def geom(nx, ny, nz, nu, nv, du, views, **kw):
    d = dict(dx=1.0, sad=300.0, sdd=450.0, angle_offset=0.13)
    d.update(kw)
    return synth.make_geometry(nx=nx, ny=ny, nz=nz, nu=nu, nv=nv, du=du, n_phases=len(views), views_per_phase=views, **d)


CASES = {
    "one_row_per_lane": geom(31, 29, 17, 37, 32, 1.3, [3, 2]),
    "ragged_rows_65": geom(33, 35, 40, 41, 65, 1.3, [2, 3]),
    "rows_beyond_the_volume": geom(40, 38, 12, 50, 150, 1.1, [2, 2]),
    "thin_slices": geom(24, 26, 90, 40, 70, 1.2, [2, 2], dz=0.05),  # many planes per xy cell
    "one_slice": geom(20, 24, 1, 33, 40, 1.2, [2, 2], dz=6.0),
    "one_row": geom(20, 24, 9, 33, 1, 1.7, [2, 2]),
    "row_in_a_face_plane": geom(21, 24, 16, 34, 65, 1.2, [2, 2]),  # v = 0 at z plane 8
    "narrow": geom(1, 30, 20, 45, 64, 1.0, [3, 2]),
    "offset_detector": geom(30, 30, 30, 64, 96, 1.0, [2, 2], u_off=11.0, v_off=-17.0, cz=5.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_table_walker_matches_slab_walker(name):
    G = tnlm.Geometry(CASES[name])
    x = torch.from_numpy(synth.uniform(G.vol_shape, 800)).cuda()
    tnlm.tnlm_set_launch_shapes(G, 4, 8, 4)
    ref = tnlm.tnlm_project(G, x).double()
    for code in (102, 104, 108):
        tnlm.tnlm_set_launch_shapes(G, code, 8, 4)
        assert tnlm.tnlm_get_launch_shapes(G)["projector_rows"] == code
        got = tnlm.tnlm_project(G, x).double()
        assert float((got - ref).norm()) <= 1e-5 * float(ref.norm())
