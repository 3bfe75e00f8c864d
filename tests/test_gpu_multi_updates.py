"""The vector-column CG updates of the blocked solve against the per-column ones:
element by element the same operations, so a solution vector that starts off a
16-byte boundary (per-column p and x update) gives the same bits.  Row counts that
leave partial passes, columns that stop early, a column that never starts."""

import pytest
import torch

from synthetic import poisson3d, uniform01

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 6, 10, 34, 64])
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_unaligned_solution_same_bits(amg, K, precision):
    A = poisson3d(13, 11, 9)
    n = 13 * 11 * 9
    H = amg.Hierarchy(*amg.csr_to_device(A), precision=precision, max_coarse=40)
    B = torch.as_tensor(uniform01(51, n * K), device="cuda").reshape(n, K).clone()
    B[:, 0] = 0.0                    # converged before the first step
    B[:, K - 1] *= 1e-3
    B[:, K // 2] = 1.0               # smooth: stops at another iteration
    X = torch.zeros(n, K, dtype=torch.float64, device="cuda")
    U = torch.zeros(n * K + 1, dtype=torch.float64, device="cuda")[1:].view(n, K)
    assert U.data_ptr() % 16 == 8
    _, sx = H.pcg_multi(B, X)
    _, su = H.pcg_multi(B, U)
    assert [s["iterations"] for s in sx] == [s["iterations"] for s in su]
    assert all(s["status"] == 0 for s in sx) and sx[0]["iterations"] == 0
    assert torch.equal(X, U)
    # and the residuals by the definition
    assert all(s["true_relres"] <= 1.05e-8 for s in sx[1:])
