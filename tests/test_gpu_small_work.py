"""Small and thin problems cost less than the ones whose launches they share:
each test compares a call with one that does several times its work.  Minima
of repeated runs; the limits leave a third of the measured difference as room."""
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


def time_us(fn, repeats=7, calls=10):
    fn()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(repeats):
        torch.cuda._sleep(4_000_000)  # ~2 ms: the calls are queued behind it, so that the GPU's time counts and not the host's
        a.record()
        for _ in range(calls):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / calls * 1e3)
    return best


def scan(nx, ny, nz, nu, nv, views, **kw):
    d = dict(dx=2.0, du=1.56, sad=1000.0, sdd=1500.0, angle_offset=0.07)
    d.update(kw)
    return tnlm.Geometry(synth.make_geometry(nx=nx, ny=ny, nz=nz, nu=nu, nv=nv, n_phases=len(views),
                                             views_per_phase=views, **d))


def backproject_us(G):
    y, v = torch.rand(G.proj_shape, device="cuda"), torch.empty(G.vol_shape, device="cuda")
    return time_us(lambda: tnlm.tnlm_backproject(G, y, v))


def test_transpose_of_one_slice():
    """One slice against eight: measured 0.68 (1.0 when both took chunks of 8)."""
    one, eight = (backproject_us(scan(256, 256, nz, 512, 64, [180], du=0.78)) for nz in (1, 8))
    assert one < 0.85 * eight


def fdk_us(nx, nz, nu, nv, views):
    G = scan(nx, nx, nz, nu, nv, views, du=400.0 / nu, dv=300.0 / nv)
    y, v = torch.rand(G.proj_shape, device="cuda"), torch.empty(G.vol_shape, device="cuda")
    return time_us(lambda: tnlm.tnlm_fdk(G, y, v))


def test_fdk_of_few_rows():
    """The filter of one view against four: measured 0.56 (0.89 when 384 rows made 12 tiles)."""
    assert fdk_us(32, 32, 512, 384, [1]) < 0.72 * fdk_us(32, 32, 512, 384, [4])


def test_fdk_of_a_small_volume():
    """32^3 against 64^3: measured 0.37 (1.1 with 8 voxels per thread in both)."""
    assert fdk_us(32, 32, 128, 96, [30] * 4) < 0.6 * fdk_us(64, 64, 128, 96, [30] * 4)


def project_us(G):
    x, p = torch.rand(G.vol_shape, device="cuda"), torch.empty(G.proj_shape, device="cuda")
    return time_us(lambda: tnlm.tnlm_project(G, x, p))


def test_projection_of_few_rows():
    """2 detector rows against 32: measured 0.39 (0.74 when both filled warps with rows)."""
    few, many = (project_us(scan(128, 128, 64, 256, nv, [40] * 4, dv=5.6)) for nv in (2, 32))
    assert few < 0.58 * many


def test_projection_of_few_slices():
    """4 slices under 192 rows against 24: measured 0.59 (0.94 with 64 rows per warp in both)."""
    few, many = (project_us(scan(128, 128, nz, 256, 192, [40] * 4)) for nz in (4, 24))
    assert few < 0.77 * many


def test_projection_of_thin_slices():
    """512 slices of a sixteenth of the pixels under a half cone of 20 degrees against the slab walker: measured
    0.76 (1.19 when the planes were settled row by row)."""
    G = scan(64, 64, 512, 128, 160, [20] * 2, dx=4.0, dz=0.25, du=3.0, dv=2.0, sad=300.0, sdd=450.0)
    table = project_us(G)
    tnlm.tnlm_set_launch_shapes(G, 4, 8, 4)
    slab = project_us(G)
    assert table < 0.95 * slab


def test_weights_gradient_of_one_candidate():
    """A window of one candidate against one of 27: measured 0.28 (0.48 when its box sums were one march in z)."""
    f, a = (torch.rand((4, 64, 64, 64), device="cuda") for _ in range(2))
    one, many = (time_us(lambda M=M: tnlm.tnlm_energy_grad_weights(f, a, 1, M, 0.02)) for M in (0, 1))
    assert one < 0.38 * many
