"""A rank that holds some of a scan's phases gets, bit for bit, what a process
that holds all of them gets from the transpose: the order in which a voxel's
views are summed must not depend on the number of phases in the handle.  The
sizes are those where the whole scan and one rank's share launch different
forms (four warps splitting the views of a patch below 608 blocks, or below 1520 with
10 views a phase or more)."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import shard, synth

pytestmark = pytest.mark.gpu

CASES = {  # nx, ny, nz, views of each phase, ranks
    "64^3_over_2": (64, 64, 64, [6, 3, 5, 7, 2, 4, 5, 3], 2),
    "96x90x40_over_6": (96, 90, 40, [5, 6, 9, 2, 3, 4], 6),
    "80x80x40_over_4": (80, 80, 40, [4, 5, 6, 1, 7, 3, 2, 2], 4),
    "64^3_10_views": (64, 64, 64, [12, 11, 16, 14, 12, 9, 15], 2),
    "ragged_16_cells": (88, 61, 70, [5, 2, 6, 4, 3, 8, 1], 7),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("cells,rows", [(8, 4), (8, 2), (4, 4), (4, 2)])
def test_transpose_of_a_share_equals_the_whole(name, cells, rows):
    nx, ny, nz, views, ranks = CASES[name]
    desc = synth.make_geometry(nx=nx, ny=ny, nz=nz, dx=1.0, nu=70, nv=50, du=2.1, sad=300.0, sdd=450.0,
                               n_phases=len(views), views_per_phase=views, angle_offset=0.13)
    y = synth.normal((int(np.sum(views)), 50, 70), 710)
    whole = tnlm.Geometry(desc)
    tnlm.tnlm_set_launch_shapes(whole, 104, cells, rows)
    ref = tnlm.tnlm_backproject(whole, torch.from_numpy(y).cuda())
    for a, b in shard.phase_blocks(len(views), ranks):
        G = tnlm.Geometry(shard.local_geometry(desc, a, b))
        yl = torch.from_numpy(np.ascontiguousarray(shard.local_projections(desc, y, a, b))).cuda()
        assert torch.equal(tnlm.tnlm_backproject(G, yl), ref[a:b]), (a, b)
