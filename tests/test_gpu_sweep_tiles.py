"""The tiles of the box-sum sweep where they can go wrong, against the FP64
oracle (relative L2 <= 1e-5, the FP32 target): one output row or column more
or less than a tile (30 or 28 x 8 x 8 outputs and their fractions), volumes
smaller than a window, both sides of the volume rule that picks the block,
values apart from the weights' sources, warps that keep running references."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu
RTOL = 1e-5


@pytest.fixture(scope="module")
def ora():
    import oracle
    oracle.build()
    return oracle


def rel_l2(a, b):
    return float(np.linalg.norm(a.astype(np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("d, M", [(1, 1), (1, 2), (1, 3), (2, 1), (2, 2), (2, 3)])
@pytest.mark.parametrize("shape", [(2, 1, 1, 1), (3, 2, 3, 4), (2, 9, 17, 31), (2, 8, 16, 30), (2, 7, 8, 29), (2, 5, 9, 57)])
def test_sweep_tile_edges(ora, shape, d, M):
    a = synth.smooth_volume(shape, 900) + synth.normal(shape, 901, 0.004)
    v, g = synth.smooth_volume(shape, 902), synth.smooth_volume(shape, 903)
    h = 0.03 if d == 1 else 0.06
    A, V, G = (torch.from_numpy(t.astype(np.float32)).cuda() for t in (a, v, g))
    same = tnlm.tnlm_gauss_jacobi(A, A, G, d, M, h, 0.7, 1)
    apart = tnlm.tnlm_gauss_jacobi(A, V, G, d, M, h, 0.7, 1)
    assert rel_l2(same.cpu().numpy(), ora.gj_sweep(a, a, g, d, M, h, 0.7, 1)) <= RTOL
    assert rel_l2(apart.cpu().numpy(), ora.gj_sweep(a, v, g, d, M, h, 0.7, 1)) <= RTOL
    assert torch.equal(same, tnlm.tnlm_gauss_jacobi(A, A.clone(), G, d, M, h, 0.7, 1))


@pytest.mark.parametrize("d, M, h", [(1, 2, 0.02), (2, 1, 0.02)])
def test_sweep_big_block_samples(ora, d, M, h):
    """A volume beyond sweep_small (the other block) with tiles whose best
    matches are poor (uniform noise: running references stay) beside smooth
    ones, on sampled voxels."""
    shape = (2, 43, 115, 130)
    a = synth.smooth_volume(shape, 910)
    a[:, :, :40] = synth.uniform((2, 43, 40, 130), 911)
    A = torch.from_numpy(a).cuda()
    got = tnlm.tnlm_gauss_jacobi(A, A, A, d, M, h, 1.0, 0).cpu().numpy()
    rng = np.random.default_rng(912)
    ref, out = [], []
    for _ in range(120):
        i, z, y, x = (int(rng.integers(0, n)) for n in shape)
        lo = [max(0, c - M - d) for c in (z, y, x)]
        hi = [min(n, c + M + d + 1) for n, c in zip(shape[1:], (z, y, x))]
        crop = np.ascontiguousarray(a[:, lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]])
        r = ora.gj_sweep(crop, crop, crop, d, M, h, 1.0, 0)
        ref.append(r[i, z - lo[0], y - lo[1], x - lo[2]])
        out.append(got[i, z, y, x])
    assert rel_l2(np.array(out), np.array(ref)) <= RTOL
