"""The column walk (32 columns of one row per warp), which the table walker
takes on volumes of thin slices under steep rays, against the slab walker on
the same handle (relative L2 <= 1e-5, the FP32 target): projections, gradient
steps with their residual norms, 16-bit storage, and the host-buffer call,
which copies and projects phase by phase, to the bit."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = {  # half cones of 16 to 30 degrees; slices of a tenth to a third of a pixel of the plane
    "ragged": dict(nx=33, ny=29, nz=200, dx=1.0, dz=0.2, nu=41, nv=67, du=1.3, dv=1.5),
    "narrow": dict(nx=3, ny=30, nz=301, dx=1.0, dz=0.1, nu=31, nv=33, du=0.9, dv=2.1),
    "off_axis": dict(nx=40, ny=38, nz=150, dx=1.0, dz=0.3, cz=9.0, nu=70, nv=50, du=1.1, dv=2.0, u_off=6.0, v_off=11.0),
}


def handle(name):
    return tnlm.Geometry(synth.make_geometry(sad=150.0, sdd=225.0, angle_offset=0.13, n_phases=3, views_per_phase=[3, 1, 2],
                                             **CASES[name]))


@pytest.mark.parametrize("name", list(CASES))
def test_column_walk_matches_slab_walker(name):
    G = handle(name)
    x = torch.from_numpy(synth.uniform(G.vol_shape, 860)).cuda()
    y = torch.from_numpy(synth.uniform(G.proj_shape, 861)).cuda()
    p = tnlm.Params(d=1, M=1, h=0.02, mu=1.0, tau=1e-4)
    got = []
    for code in (4, 102, 104, 108):
        tnlm.tnlm_set_launch_shapes(G, code, 8, 4)
        g = torch.empty_like(x)
        report = tnlm.tnlm_p1(G, y, x, g, p, report=True)
        got.append((tnlm.tnlm_project(G, x).double(), g.double(), float(report[0])))
    for proj, g, norm in got[1:]:
        assert float((proj - got[0][0]).norm()) <= 1e-5 * float(got[0][0].norm())
        assert float((g - got[0][1]).norm()) <= 1e-5 * float(got[0][1].norm())
        assert abs(norm - got[0][2]) <= 1e-5 * got[0][2]


@pytest.mark.parametrize("name", list(CASES))
def test_host_buffers_and_16_bit_storage(name):
    G = handle(name)
    f0, y = synth.uniform(G.vol_shape, 862), synth.uniform(G.proj_shape, 863)
    p = tnlm.Params(d=1, M=1, h=0.02, mu=1.0, tau=1e-4, n_outer=2)
    f = torch.from_numpy(f0.copy()).cuda()
    tnlm.tnlm_reconstruct(G, torch.from_numpy(y).cuda(), f, p)
    host = torch.from_numpy(f0.copy()).pin_memory()
    tnlm.reconstruct_host(G, torch.from_numpy(y).pin_memory(), host, p)
    torch.cuda.synchronize()
    assert np.array_equal(host.numpy(), f.cpu().numpy())
    # 16-bit storage against the slab walker: FP32 rounding flips the stored rounding of ~1e-4 of the elements by an ulp of
    # up to 2^-8, which the weights of noise this strong carry on ~10 times as large: 4e-4
    for dtype, call in ((torch.bfloat16, tnlm.tnlm_reconstruct_bf16), (torch.float16, tnlm.tnlm_reconstruct_fp16)):
        out = []
        for code in (104, 4):
            tnlm.tnlm_set_launch_shapes(G, code, 8, 4)
            out.append(torch.from_numpy(f0).cuda().to(dtype))
            call(G, torch.from_numpy(y).cuda().to(dtype), out[-1], p)
        assert float((out[0].double() - out[1].double()).norm()) <= 1e-3 * float(out[1].double().norm())
