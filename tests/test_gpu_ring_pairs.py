"""Two slices a warp in the ring's FP32 pre-smoother against the per-lane kernel:
levels of at least 4,864 slices, an odd number of slices, ragged last slices, pairs
of one coding and width (both rows' gathers together) and mixed pairs.  The order
of a row's operations is the same, so the V-cycles agree bit for bit."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, poisson3d, uniform01
from tests.test_gpu_ring_index import _far_chords

pytestmark = pytest.mark.gpu

CASES = {
    "ragged": lambda: poisson3d(67, 61, 41),        # 5,237 slices, the last of 7 rows
    "two_levels": lambda: poisson3d(90, 91, 92),    # level 1 as well
    "mixed": lambda: _far_chords(160001, 70000),    # codings and widths change
    "diffusion": lambda: diffusion3d(np.exp(gaussian_field((59, 57, 53), 2.0, 4.0, 5))),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("opts", [dict(), dict(smooth_sweeps=2), dict(bf16_from_level=1)])
def test_pairs_bitwise(amg, case, opts):
    Ad = amg.csr_to_device(CASES[case]())
    n = Ad[0].numel() - 1
    assert (n + 31) // 32 >= 2 * 8 * 304
    H1 = amg.Hierarchy(*Ad, precision="f32", stream_ring=1, **opts)
    H0 = amg.Hierarchy(*Ad, precision="f32", stream_ring=0, **opts)
    r = torch.as_tensor(uniform01(61, n + 1), device="cuda")
    assert torch.equal(H1.vcycle(r[:n].clone()), H0.vcycle(r[:n].clone()))
    assert torch.equal(H1.vcycle(r[1:]), H0.vcycle(r[1:].clone()))  # off a 16-byte boundary
