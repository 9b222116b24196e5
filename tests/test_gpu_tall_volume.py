"""Rows in and next to the top face of a volume of more slices than FP32
resolves to 1e-3 (beyond 2^14): the table walker keeps every row that could
round to the slice above the last one under its bounds test.  A row in the
face plane is outside (half-open cells): exactly 0.  Where the rows run the
values do not change along z, so the others equal those of a volume of 1024
slices below the same top face (slab walker; relative L2 <= 1e-5)."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


def top_slices(nz):
    """A handle and a volume of nz slices of 2^-10 mm whose top face is the plane z = 0, to the bit; row 32 of 65 lies in
    it, the others fan out by 0.01 mm."""
    dz = 2.0**-10
    G = tnlm.Geometry(synth.make_geometry(nx=3, ny=2, nz=nz, dx=1.0, dz=dz, cz=-0.5 * nz * dz, nu=9, nv=65, du=0.9, dv=0.01,
                                          sad=300.0, sdd=450.0, n_phases=1, views_per_phase=[3], angle_offset=0.13))
    x = np.broadcast_to(synth.uniform((1, 1, 2, 3), 820), G.vol_shape).copy()
    x[:, 0] = 1e3  # what a read one slice too far finds: the first slice of the next voxel column
    return G, torch.from_numpy(x).cuda()


@pytest.mark.parametrize("nz", [16000, 40000, 262144])
def test_rows_at_the_top_face(nz):
    G, x = top_slices(1024)
    tnlm.tnlm_set_launch_shapes(G, 4, 8, 4)
    ref = tnlm.tnlm_project(G, x).double()
    assert float(ref[:, 32].abs().max()) == 0.0 and float(ref[:, :32].abs().max()) > 0.0
    G, x = top_slices(nz)
    for code in (102, 104, 108):
        tnlm.tnlm_set_launch_shapes(G, code, 8, 4)
        assert tnlm.tnlm_get_launch_shapes(G)["projector_rows"] == code
        got = tnlm.tnlm_project(G, x).double()
        assert float(got[:, 32].abs().max()) == 0.0
        assert float((got - ref).norm()) <= 1e-5 * float(ref.norm())
