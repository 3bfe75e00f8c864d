"""The ring's packed column indices and its sweep kernels against the per-lane
kernels: the codings (one offset per ELL column with and without clamped
padding, 16-bit deltas, plain columns) and the tile sizes only change how a
column index is stored, so every V-cycle must agree bit for bit."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, poisson3d, uniform01
from tests.helpers import from_dense, random_spd_graph

pytestmark = pytest.mark.gpu


def _far_chords(n, d):
    """Chain with couplings i <-> i + d on every third row: slices mix columns
    near the row with columns more than 65535 away, so neither offsets nor
    16-bit deltas hold them."""
    far = [(i, i + d) for i in range(0, n - d, 3)]
    rows = [[(i, 4.0)] for i in range(n)]
    for i, j in [(i, i + 1) for i in range(n - 1)] + far:
        rows[i].append((j, -1.0))
        rows[j].append((i, -1.0))
    rows = [sorted(r) for r in rows]
    rp = np.zeros(n + 1, dtype=np.int64)
    rp[1:] = np.cumsum([len(r) for r in rows])
    return (rp, np.array([j for r in rows for j, _ in r], dtype=np.int32),
            np.array([v for r in rows for _, v in r]))


CASES = {
    # every slice on the boundary (clamped offsets), ragged last slice
    "thin": lambda: poisson3d(33, 2, 37),
    "line": lambda: poisson3d(67, 1, 1),
    # several tiles a CTA, irregular coarse levels (deltas)
    "diffusion": lambda: diffusion3d(np.exp(gaussian_field((61, 53, 50), 2.0, 4.0, 5))),
    "plain": lambda: _far_chords(140001, 70000),
    "dense_rows": lambda: random_spd_graph(700, 0.05, 3),  # slices near the width limit
    "diagonal": lambda: from_dense(np.diag(np.arange(1.0, 70.0))),
}


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("opts", [dict(precision="f64"), dict(precision="f32"),
                                  dict(precision="f64", smooth_sweeps=3),
                                  dict(precision="f32", smooth_sweeps=2),
                                  dict(precision="f64", stream_ring=4)])
def test_codings_and_sweeps_bitwise(amg, case, opts):
    A = CASES[case]()
    n = len(A[0]) - 1
    Ad = amg.csr_to_device(A)
    opts = dict(dict(stream_ring=1, max_coarse=30), **opts)
    H1 = amg.Hierarchy(*Ad, **opts)
    H0 = amg.Hierarchy(*Ad, **dict(opts, stream_ring=0))
    r = torch.as_tensor(uniform01(31, n), device="cuda")
    assert torch.equal(H1.vcycle(r), H0.vcycle(r))


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_vectors_off_a_16_byte_boundary(amg, precision):
    # row vectors that no bulk copy can start at are read directly
    A = poisson3d(29, 31, 30)
    n = 29 * 31 * 30
    H = amg.Hierarchy(*amg.csr_to_device(A), precision=precision)
    u = torch.as_tensor(uniform01(33, n + 1), device="cuda")
    r = u[1:]
    assert r.data_ptr() % 16 == 8
    z = torch.empty(n + 1, dtype=torch.float64, device="cuda")[1:]
    assert torch.equal(H.vcycle(r, z), H.vcycle(r.clone()))
