"""One infinite detector pixel in the FDK filter and backprojection.  The ramp
has a positive tap at 0, negative taps at odd offsets and none at even ones, so
the filtered row is +inf at the pixel, -inf at the columns of the other parity
and finite elsewhere; a voxel takes two neighbouring columns, one of each
parity, and is -inf wherever neither is the pixel itself: far from it, near
it (the taps that are summed apart), and where one of the two columns lies off
the detector and the voxel takes only the other."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu

NU, NV, ROW = 65, 21, 10


def images(desc):
    """Detector coordinates (column, row) of every voxel centre in the one view, FP64."""
    c, s = np.cos(desc["angles"][0]), np.sin(desc["angles"][0])
    x, y, z = ((np.arange(desc["n" + a]) + 0.5 - 0.5 * desc["n" + a]) * desc["d" + a] for a in "xyz")
    depth = desc["sad"] - (x[None, :] * c + y[:, None] * s)
    u = desc["sdd"] * (-x[None, :] * s + y[:, None] * c) / depth
    fu = u / desc["du"] + 0.5 * (NU - 1)
    fv = desc["sdd"] * z[:, None, None] / depth / desc["dv"] + 0.5 * (NV - 1)
    return np.broadcast_to(fu, fv.shape), fv


@pytest.mark.parametrize("where", ["near", "far", "left_edge", "right_edge"])
@pytest.mark.parametrize("column", [31, 33])
def test_infinite_pixel(column, where):
    desc = synth.make_geometry(nx=70, ny=66, nz=14, dx=1.0, nu=NU, nv=NV, du=1.2, dv=1.2, sad=300.0, sdd=450.0, n_phases=1,
                               views_per_phase=[1], angle_offset=0.13)
    G = tnlm.Geometry(desc)
    y = synth.uniform(G.proj_shape, 840)
    y[0, ROW, column] = np.inf
    vol = tnlm.tnlm_fdk(G, torch.from_numpy(y).cuda()).cpu().numpy()[0]
    fu, fv = images(desc)
    rows = np.abs(fv - ROW) < 0.999  # the infinite row has a share
    clear = np.abs(fv - ROW) > 1.001
    away = np.abs(fu - column)
    sel = {"near": (away > 1.001) & (away < 14) & (fu > 0.001), "far": (away > 16) & (fu > 0.001) & (fu < NU - 1.001),
           "left_edge": (fu > -0.999) & (fu < -0.001), "right_edge": (fu > NU - 0.999) & (fu < NU - 0.001)}[where]
    assert (sel & rows).sum() > 20
    assert np.isneginf(vol[sel & rows]).all()
    assert np.isfinite(vol[clear]).all()
