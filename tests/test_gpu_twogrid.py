"""The two-grid loss for sample counts around its groups of eight (one column is
solved by itself, several by the blocked PCG) and for the hierarchies the blocked
PCG does not serve."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, standard_normal, uniform01

pytestmark = pytest.mark.gpu

SHAPE, N = (12, 11, 10), 1320
# the coarsest PCG solves far below the inner solve's 1e-12, so its V-cycle is the
# linear one that the inner CG expects
PCG_COARSE = dict(coarse_solver=1, coarse_maxit=400, coarse_tol=1e-13)


@pytest.fixture(scope="module")
def lm(amg):
    from paper_2406_19754_gb300 import learned

    return learned


@pytest.fixture(scope="module")
def problem(amg, orc):
    """Matrix on the device, weights, twelve initial errors, and the oracle's
    loss and gradient for the first k of them."""
    A = diffusion3d(np.exp(gaussian_field(SHAPE, 2.0, 3.0, 3)))
    om = (0.2 + 0.8 * uniform01(4, N)).astype(np.float32)
    e0 = standard_normal(9, 12 * N).reshape(12, N)
    Ho = orc.Hierarchy(A, max_coarse=1)
    args = (A, Ho.level_agg(0), Ho.level_csr(1), om.astype(np.float64))
    known = {}

    def expect(k):
        if k not in known:
            known[k] = orc.twogrid_loss(*args, e0[:k], K=2)
        return known[k]

    return amg.csr_to_device(A), om, torch.as_tensor(e0, device="cuda"), expect


def _hierarchy(amg, problem, **opts):
    H = amg.Hierarchy(*problem[0], max_coarse=20, **opts)
    assert H.levels >= 4  # the inner hierarchy has several levels
    H.set_smoother_weights(torch.as_tensor(problem[1], device="cuda"))
    return H


def _check(lm, H, problem, k):
    # inner solves to 1e-12, as in test_twogrid_loss_matches_oracle
    loss, dom = lm.twogrid_loss(H, problem[2][:k], 2)
    loss_o, dom_o = problem[3](k)
    assert abs(loss - loss_o) <= 1e-9 * abs(loss_o)
    np.testing.assert_allclose(dom.cpu().numpy(), dom_o, rtol=2e-6,
                               atol=1e-6 * np.abs(dom_o).max())


@pytest.mark.parametrize("opts", [dict(), PCG_COARSE], ids=["dense", "pcg_coarse"])
def test_sample_counts_match_oracle(amg, lm, problem, opts):
    H = _hierarchy(amg, problem, **opts)
    for k in (2, 1, 8, 9, 12, 3):  # more samples after fewer, and back
        _check(lm, H, problem, k)


def test_blocked_calls_refuse_the_pcg_coarsest_solve(amg):
    # such a hierarchy has no dense coarsest factor for the blocked V-cycle
    from paper_2406_19754_gb300 import _lib

    A = diffusion3d(np.exp(gaussian_field(SHAPE, 2.0, 3.0, 3)))
    H = amg.Hierarchy(*amg.csr_to_device(A), max_coarse=20, coarse_solver=1)
    B = torch.as_tensor(uniform01(1, 2 * N), device="cuda").reshape(N, 2)
    for call in (H.pcg_multi, H.vcycle_multi):
        with pytest.raises(amg.AmgError) as e:
            call(B)
        assert e.value.status == _lib.AMG_ERR_UNSUPPORTED
