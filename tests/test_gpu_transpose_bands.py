"""The band transpose where its forms can go wrong, against the exact per-cell
transpose (what runs without the prefix workspace; relative L2 <= 1e-5, the
FP32 target): chunks of 4, 8 and 16 cells with ragged nz, the views of a patch
split over the warps of a block, bands of several detector rows, boundaries
off the detector, views that miss warps.  The per-cell form is the reference
and not the oracle because rays that lie in or graze a face plane (level_row;
the corners seen by two views only) fall to either side in FP32 in both."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu
RTOL = 1e-5


def geom(nx, ny, nz, nu, nv, du, views, **kw):
    d = dict(dx=1.0, sad=300.0, sdd=450.0, angle_offset=0.13)
    d.update(kw)
    return synth.make_geometry(nx=nx, ny=ny, nz=nz, nu=nu, nv=nv, du=du, n_phases=len(views), views_per_phase=views, **d)


CASES = {
    "split_cells_4": geom(9, 7, 5, 21, 12, 1.5, [3, 1, 6]),             # fewer views than warps in one phase
    "split_cells_8": geom(66, 50, 21, 61, 30, 1.9, [5, 2, 3]),
    "cells_8_odd_chunks": geom(97, 90, 39, 80, 50, 2.2, [3, 2]),
    "cells_16_ragged": geom(97, 90, 61, 80, 76, 2.2, [2, 3]),
    "off_detector": geom(40, 40, 64, 64, 11, 1.3, [3, 4]),              # most boundaries image off the rows
    "one_row_detector": geom(17, 33, 9, 30, 1, 2.0, [2, 2]),
    "bands_of_2_rows": geom(40, 36, 21, 100, 90, 0.9, [3, 3], dx=2.0, dz=2.0),
    "bands_of_rows": geom(24, 20, 21, 100, 130, 0.45, [3, 3], dx=3.0, dz=3.0),
    "bands_of_rows_unsplit": geom(98, 90, 40, 128, 260, 0.5, [2, 2], dx=1.6, dz=1.6),
    "level_row": geom(20, 20, 16, 31, 25, 1.5, [4, 4], angle_offset=0.0),  # v = 0 in the plane of a boundary
}


@pytest.mark.parametrize("name", list(CASES))
def test_band_transpose_matches_per_cell_form(name):
    G = tnlm.Geometry(CASES[name])
    y = synth.normal(G.proj_shape, 700)
    per_cell = tnlm.Geometry(CASES[name])
    tnlm._load().tnlm_test_fail_allocations(1)  # the prefix workspace
    try:
        ref = tnlm.tnlm_backproject(per_cell, torch.from_numpy(y).cuda()).cpu().numpy().astype(np.float64)
    finally:
        tnlm._load().tnlm_test_fail_allocations(0)
    outs = []
    for cells in (8, 4):
        tnlm.tnlm_set_launch_shapes(G, 4, cells, 4)
        outs.append(tnlm.tnlm_backproject(G, torch.from_numpy(y).cuda()))
    assert torch.equal(outs[0], outs[1])
    got = outs[0].cpu().numpy()
    assert np.linalg.norm(got - ref) <= RTOL * np.linalg.norm(ref)

