"""Batches with more systems than a grid has blocks in y (65,535): the coarsest
factors are launched in parts."""

import numpy as np
import pytest
import torch

from synthetic import uniform01

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys", [65535, 65536, 70001])
def test_systems_beyond_one_launch(amg, nsys):
    # one or two rows each, solved exactly by the one-level hierarchy
    mats = [np.array([[2.0 + k]]) for k in range(3)]
    mats += [np.array([[2.0, -1.0], [-1.0, 3.0 + k]]) for k in range(4)]
    dev = []
    for M in mats:
        m = len(M)
        dev.append(amg.csr_to_device((np.arange(m + 1) * m, np.tile(np.arange(m), m),
                                      M.reshape(-1))))
    kind = (uniform01(61, nsys) * len(mats)).astype(int)
    H = amg.BatchHierarchy([dev[k] for k in kind])
    assert H.levels == 1 and H.nsys == nsys
    b = uniform01(62, H.n)
    z = H.vcycle(torch.as_tensor(b, device="cuda")).cpu().numpy()
    off = np.array(H.offsets[:-1])
    for k, M in enumerate(mats):  # condition numbers below 4: rounding errors only
        at = off[kind == k][:, None] + np.arange(len(M))
        np.testing.assert_allclose(z[at], b[at] @ np.linalg.inv(M), rtol=1e-13)
