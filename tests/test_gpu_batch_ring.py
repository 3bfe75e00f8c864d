"""Batched levels on the shared-memory ring against the per-lane kernels: the
chunks of one system, tiles that start at any slice, systems that start at any
row (off the copies' 16-byte boundaries) and systems that stop early.  The
V-cycle's row sums keep their order, so it agrees bit for bit; the dot products
are summed in another order, so solves get the bounds of the batched solves
against the oracle (iterations +-1, solution to 1e-10)."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, poisson3d, uniform01
from tests.helpers import random_spd_graph

pytestmark = pytest.mark.gpu


def _uneven():
    # wide rows in the middle: the widest window of slices starts between two tiles
    return [poisson3d(3, 2, 1), poisson3d(43, 41, 31), random_spd_graph(301, 0.04, 7),
            diffusion3d(np.exp(gaussian_field((33, 31, 29), 2.0, 4.0, 3))), poisson3d(1, 1, 33)]


CASES = {
    "uneven": _uneven,                                         # level 0 on the ring
    "two_levels": lambda: _uneven() + [poisson3d(97, 91, 83)],  # levels 0 and 1
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("precision,sweeps", [("f64", 1), ("f32", 1), ("f64", 2)])
def test_batched_ring_equals_per_lane(amg, case, precision, sweeps):
    systems = [amg.csr_to_device(S) for S in CASES[case]()]
    opts = dict(precision=precision, smooth_sweeps=sweeps)
    H1 = amg.BatchHierarchy(systems, stream_ring=1, **opts)
    H0 = amg.BatchHierarchy(systems, stream_ring=0, **opts)
    o = H1.offsets
    assert H1.level_info(0)[0] >= 32 * 304 * 8
    b = torch.as_tensor(uniform01(41, o[-1]), device="cuda")
    assert torch.equal(H1.vcycle(b), H0.vcycle(b))
    for graph in (True, False):
        x1, s1 = H1.pcg(b, tol=1e-8, use_graph=graph)
        x0, s0 = H0.pcg(b, tol=1e-8, use_graph=graph)
        for k in range(len(systems)):
            assert s1[k]["status"] == s0[k]["status"] == 0
            assert abs(s1[k]["iterations"] - s0[k]["iterations"]) <= 1
            if s1[k]["iterations"] == s0[k]["iterations"]:
                d = x1[o[k]:o[k + 1]] - x0[o[k]:o[k + 1]]
                assert float(d.norm() / x0[o[k]:o[k + 1]].norm()) <= 1e-10
        assert min(s["iterations"] for s in s1) < max(s["iterations"] for s in s1)


@pytest.mark.parametrize("max_coarse", [40, 130, 600])  # blocks of one CTA, of whole-grid rows
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_coarsest_blocks_by_rows(amg, max_coarse, precision):
    # each system's part of the blocked V-cycle is that of the system alone (its
    # coarsest block solved by one CTA in the small-level launch): the same bits
    systems = [poisson3d(21, 20, 19), poisson3d(21, 20, 19)]
    devs = [amg.csr_to_device(S) for S in systems]
    Hb = amg.BatchHierarchy(devs, max_coarse=max_coarse, precision=precision)
    Hs = amg.Hierarchy(*devs[0], max_coarse=max_coarse, precision=precision)
    assert Hb.levels == Hs.levels
    n = Hs.level_info(0)[0]
    b = torch.as_tensor(uniform01(47, 2 * n), device="cuda")
    z = Hb.vcycle(b)
    for k in range(2):
        assert torch.equal(z[k * n:(k + 1) * n], Hs.vcycle(b[k * n:(k + 1) * n].clone()))
