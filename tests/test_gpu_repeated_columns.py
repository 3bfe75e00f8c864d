"""Matrices whose rows store a column twice (sorted ascending, not strictly): the
Galerkin product adds the values."""

import numpy as np
import pytest
import torch

from synthetic import uniform01
from tests.helpers import dense, prolongator, random_spd_graph

pytestmark = pytest.mark.gpu


def _halved(A, seed):
    """A with about half of its off-diagonal pairs stored as two equal halves."""
    rp, ci, v = A
    n = len(rp) - 1
    rows = np.repeat(np.arange(n), np.diff(rp))
    u = uniform01(seed, n * n).reshape(n, n)
    twice = (np.where(rows < ci, u[rows, ci], u[ci, rows]) < 0.5) & (rows != ci)
    reps = np.where(twice, 2, 1)
    counts = np.zeros(n + 1, np.int64)
    np.add.at(counts, rows + 1, reps)
    return np.cumsum(counts), np.repeat(ci, reps), np.repeat(np.where(twice, v / 2, v), reps)


# rows of about 450 p entries: 2 or 4 members below, around and above the 64
# contributions that a warp orders by rank
@pytest.mark.parametrize("p", [0.01, 0.03, 0.05, 0.25])
@pytest.mark.parametrize("sweeps", [1, 2])
def test_galerkin_adds_repeated_entries(amg, p, sweeps):
    n = 300
    A = random_spd_graph(n, p, 71, positive_offdiag=True)
    D = _halved(A, 72)
    assert len(D[1]) > len(A[1])
    H = amg.Hierarchy(*amg.csr_to_device(D), sweeps=sweeps, max_coarse=40)
    assert H.levels >= 2
    nc = H.level_info(1)[0]
    P = prolongator(H.level_export(0)["agg"].cpu().numpy(), nc)
    M = dense(A)  # halving is exact
    ex = {k: t.cpu().numpy() for k, t in H.level_export(1).items()}
    rp, ci = ex["rowptr"], ex["col"]
    pattern = P.T @ (M != 0.0) @ P > 0
    assert np.array_equal(np.diff(rp), pattern.sum(axis=1))
    assert np.array_equal(ci, np.nonzero(pattern)[1])
    got = np.zeros((nc, nc))
    got[np.repeat(np.arange(nc), np.diff(rp)), ci] = ex["val"]
    # at most 2^2 x 300 additions: well under 1e-12 of the absolute sums
    assert (np.abs(got - P.T @ M @ P) <= 1e-12 * (P.T @ np.abs(M) @ P)).all()
    b = uniform01(73, n)
    x, info = H.pcg(torch.as_tensor(b, device="cuda"), tol=1e-12)
    assert info["status"] == 0 and info["true_relres"] <= 1e-11
    # strictly diagonally dominant by at least 0.5: |x| error below 2 |residual|
    err = np.abs(x.cpu().numpy() - np.linalg.solve(M, b)).max()
    assert err <= 2.0 * 1e-11 * np.linalg.norm(b)
