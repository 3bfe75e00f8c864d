"""A set-up in which a device allocation fails: it ends with AMG_ERR_OOM, or, for
what is there for speed only (edge weights of the matching, packed column indices
of the streams), goes on without it to the same hierarchy and the same bits."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, uniform01

pytestmark = pytest.mark.gpu

SHAPE, N = (20, 18, 16), 5760


@pytest.mark.parametrize("opts", [dict(), dict(precision="f32"),
                                  dict(sweeps=3, smooth_sweeps=2, smooth_prolongator=1)],
                         ids=["f64", "f32", "smoothed"])
def test_setup_without_room_for_what_only_speeds_it_up(amg, opts):
    from paper_2406_19754_gb300 import _lib

    A = amg.csr_to_device(diffusion3d(np.exp(gaussian_field(SHAPE, 1.5, 3.0, 13))))
    opts = dict(opts, max_coarse=60)
    ref = amg.Hierarchy(*A, **opts)
    r = torch.as_tensor(uniform01(14, N), device="cuda")
    z_ref = ref.vcycle(r)
    iterations = ref.pcg(r, tol=1e-8)[1]["iterations"]
    lib = _lib.load()
    went_on = failed = k = 0
    while True:
        lib.amg_debug_fail_alloc_after(k)
        H = None
        try:
            H = amg.Hierarchy(*A, **opts)
        except amg.AmgError as e:
            assert e.status == _lib.AMG_ERR_OOM
            failed += 1
        finally:
            # still armed: the set-up made no k-th allocation
            done = H is not None and _armed(amg)
            lib.amg_debug_fail_alloc_after(-1)
        if done:
            break
        if H is not None:
            went_on += 1
            assert H.levels == ref.levels
            assert torch.equal(H.vcycle(r), z_ref)
            info = H.pcg(r, tol=1e-8)[1]  # dot products may be summed over other grids
            assert info["status"] == 0 and info["true_relres"] <= 2e-8
            assert abs(info["iterations"] - iterations) <= 1
        k += 1
    # a weight array a matching sweep, records and indices of every streamed operator
    assert went_on >= 3 * (ref.levels - 1) and failed > went_on


def _armed(amg):
    """Whether the failure is still to come (uses it up)."""
    from paper_2406_19754_gb300 import learned

    try:
        for _ in range(200):
            learned.Mlp(0)  # a handful of allocations, each of which ends the call
    except amg.AmgError:
        return True
    return False
