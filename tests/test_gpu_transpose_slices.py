"""Volumes of a few slices take chunks of 4 cells: against the exact per-cell
transpose (what runs without the prefix workspace; relative L2 <= 1e-5), with
the views of a patch split over the warps and without, one candidate row per
boundary and two."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [1, 3, 4, 5])
@pytest.mark.parametrize("nx,phases,du", [(33, 2, 1.5), (260, 3, 1.5), (66, 2, 0.7)])
def test_few_slices_match_per_cell_form(nx, phases, du, nz):
    desc = synth.make_geometry(nx=nx, ny=nx - 4, nz=nz, dx=1.0, nu=int(1.5 * nx / du), nv=9, du=du, sad=600.0, sdd=900.0,
                               n_phases=phases, views_per_phase=[4] * phases, angle_offset=0.13)
    y = torch.from_numpy(synth.normal((4 * phases, desc["nv"], desc["nu"]), 720)).cuda()
    G, per_cell = tnlm.Geometry(desc), tnlm.Geometry(desc)
    got = tnlm.tnlm_backproject(G, y).cpu().numpy().astype(np.float64)
    tnlm._load().tnlm_test_fail_allocations(1)  # the prefix workspace
    try:
        ref = tnlm.tnlm_backproject(per_cell, y).cpu().numpy().astype(np.float64)
    finally:
        tnlm._load().tnlm_test_fail_allocations(0)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
