"""The FDK filter and backprojection at the edges of their tiles (64 rows, 256
outputs of one parity, 64 samples a chunk; 16 x 8 columns, 8 slices), odd and
even row lengths, voxels that image off the detector, against the FP64 oracle
(relative L2 <= 1e-5, the FP32 target)."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


def check(geom, noise):
    import oracle
    oracle.build()
    G = tnlm.Geometry(geom)
    objs = [[((0.5, -0.5, 0.2), (5.0, 4.0, 3.0), 0.02)] for _ in range(2)]
    p = (synth.analytic_projections(geom, objs).numpy() + synth.normal(G.proj_shape, 950, noise)).astype(np.float32)
    ref = oracle.fdk(oracle.Geometry(geom), p)
    got = tnlm.tnlm_fdk(G, torch.from_numpy(p).cuda()).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("nx,ny,nz,nu,nv", [(17, 9, 9, 1, 5), (16, 8, 8, 2, 64), (12, 13, 5, 65, 13), (20, 18, 7, 129, 33),
                                            (24, 20, 40, 90, 11)])
def test_fdk_tile_edges(nx, ny, nz, nu, nv):
    geom = synth.make_geometry(nx=nx, ny=ny, nz=nz, dx=1.0, nu=nu, nv=nv, du=60.0 / nu, dv=1.6, sad=300.0, sdd=450.0,
                               n_phases=2, views_per_phase=[5, 7], angle_offset=0.11)
    check(geom, 1e-3)


@pytest.mark.parametrize("nu", [513])
def test_fdk_long_rows(nu):
    """Several tiles of outputs per row.  Without noise: a pixel coordinate of
    a long row carries ~nu 2^-24 pixels of FP32 rounding, which noise that is
    white from pixel to pixel (and ramp-filtered) would turn into errors of
    that relative size times several."""
    check(synth.make_geometry(nx=24, ny=20, nz=11, dx=1.0, nu=nu, nv=9, du=70.0 / nu, dv=1.6, sad=300.0, sdd=450.0,
                              n_phases=2, views_per_phase=[5, 7], angle_offset=0.11), 0.0)
