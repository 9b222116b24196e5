"""The gradient through the weights in every form its kernels are compiled in,
against the FP64 oracle: patch radii 0 to 3, window radii 0 to 4, rows that
cross the box sum's hand-over in x (28 positions at d = 2) and its runs in z,
and volumes smaller than d + M, where both faces fold onto the same voxels.
Relative L2 <= 2e-5: f and a are alike here, and the terms of a voxel cancel."""
import numpy as np
import pytest
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,M,shape", [(0, 1, (3, 9, 10, 35)), (0, 2, (2, 3, 5, 4)), (3, 1, (2, 8, 9, 31)), (3, 2, (2, 2, 3, 4)),
                                       (1, 4, (2, 7, 8, 9)), (2, 4, (2, 2, 1, 2)), (2, 1, (2, 40, 7, 29)), (2, 2, (3, 11, 9, 57)),
                                       (1, 3, (2, 4, 3, 2)), (2, 3, (2, 2, 3, 4)), (1, 1, (3, 70, 17, 33))])
def test_every_form_matches_the_oracle(ora, d, M, shape):
    f = synth.smooth_volume(shape, 880) + synth.normal(shape, 881, 0.002)
    a = synth.smooth_volume(shape, 882) + synth.normal(shape, 883, 0.002)
    got = tnlm.tnlm_energy_grad_weights(torch.from_numpy(f).cuda(), torch.from_numpy(a).cuda(), d, M, 0.03).cpu().numpy()
    ref = ora.energy_grad_a(f, a, d, M, 0.03)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
