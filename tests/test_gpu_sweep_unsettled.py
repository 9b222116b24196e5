"""Noise of the order of h and far above it: warps in which some output's first
matches are poor keep running references.  The sweep of a large volume from
its own weight sources (16 outputs per thread, the rest of such a warp's
columns out of line) against the one with the values in a buffer of their own
(8 outputs per thread), which sums alike: equal to the bit; and both against
the FP64 oracle on a few slices (relative L2 <= 1e-5, the FP32 target)."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2, 3])
@pytest.mark.parametrize("noise,h", [(0.02, 0.02), (0.02, 0.005), (0.05, 0.001)])
def test_large_block_equals_small_block(M, noise, h):
    g = torch.from_numpy(synth.smooth_volume((3, 43, 118, 121), 870) + synth.normal((3, 43, 118, 121), 871, noise)).cuda()
    assert torch.equal(tnlm.tnlm_gauss_jacobi(g, g, g, 1, M, h, 1.0, 1), tnlm.tnlm_gauss_jacobi(g, g.clone(), g, 1, M, h, 1.0, 1))


def test_unsettled_against_the_oracle(ora):
    shape = (2, 3, 450, 452)  # more than 600 000 voxels: the large block
    g = synth.smooth_volume(shape, 872) + synth.normal(shape, 873, 0.02)
    G = torch.from_numpy(g).cuda()
    got = tnlm.tnlm_gauss_jacobi(G, G, G, 1, 2, 0.02, 1.0, 0).cpu().numpy()
    ref = ora.enhance(g, 1, 2, 0.02, 1.0, 1)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
