"""Small levels in one cluster's shared memory, and the PCG coarsest solve over
a cluster, against the one-launch-per-step kernels: the same rows in the same
order, so the same bits.  Sizes put the cluster's first level at one slice per
CTA, at ragged last CTAs, and at levels too large for it."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, poisson3d, uniform01

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(17, 13, 11), (23, 21, 19), (40, 40, 40), (70, 61, 53)])
@pytest.mark.parametrize("opts", [
    dict(precision="f64"), dict(precision="f32"), dict(precision="f32", bf16_from_level=1),
    dict(precision="f64", smooth_sweeps=2, variable_cycle=1),
    dict(precision="f32", smooth_sweeps=3, coarse_solver=1),
    dict(precision="f64", sweeps=3, coarse_solver=1, coarse_tol=0.0, coarse_maxit=7),
    dict(precision="f64", sweeps=1), dict(precision="f64", max_coarse=40),
])
def test_cluster_levels_bitwise(amg, shape, opts):
    A = diffusion3d(np.exp(gaussian_field(shape, 1.5, 4.0, 51)))
    n = shape[0] * shape[1] * shape[2]
    Ad = amg.csr_to_device(A)
    H = amg.Hierarchy(*Ad, **opts)
    H0 = amg.Hierarchy(*Ad, **dict(opts, tail_rows=0))
    r = torch.as_tensor(uniform01(6, n), device="cuda")
    assert torch.equal(H.vcycle(r), H0.vcycle(r))


@pytest.mark.parametrize("max_coarse", [20, 33, 64, 150, 400])
@pytest.mark.parametrize("tpr", [1, 4, 16])
def test_cluster_pcg_against_numpy(amg, max_coarse, tpr):
    # one level solved by the PCG alone (one to 16 CTAs): far enough for 1e-12
    # of the residual, compared with a dense solve at cond * 1e-12 <= 1e-9
    shape = {20: (5, 2, 2), 33: (11, 3, 1), 64: (8, 4, 2), 150: (10, 5, 3),
             400: (10, 8, 5)}[max_coarse]
    A = poisson3d(*shape)
    n = shape[0] * shape[1] * shape[2]
    H = amg.Hierarchy(*amg.csr_to_device(A), max_coarse=max_coarse, coarse_solver=1,
                      coarse_maxit=500, coarse_tol=1e-12, threads_per_row=tpr)
    assert H.levels == 1
    M = np.zeros((n, n))
    rp, ci, v = A
    for i in range(n):
        M[i, ci[rp[i]:rp[i + 1]]] = v[rp[i]:rp[i + 1]]
    b = uniform01(9, n)
    z = H.vcycle(torch.as_tensor(b, device="cuda")).cpu().numpy()
    want = np.linalg.solve(M, b)
    assert np.linalg.norm(z - want) <= 1e-9 * np.linalg.norm(want)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n_off", [0, 1, 2, 3])
def test_solves_into_other_vectors(amg, precision, n_off):
    # captured iterations find x through the scalars: another x (here also off a
    # 16-byte boundary), another tolerance and another cap on the same handle
    A = poisson3d(21, 19, 17 + n_off)  # row counts of every remainder by 4
    n = len(A[0]) - 1
    Ad = amg.csr_to_device(A)
    b = torch.as_tensor(uniform01(3, n), device="cuda")
    ref, ri = amg.Hierarchy(*Ad, precision=precision).pcg(b, tol=1e-9, use_graph=0)
    H = amg.Hierarchy(*Ad, precision=precision)
    H.pcg(b, tol=1e-3)
    buf = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    for x in (torch.zeros_like(b), buf[1:], torch.zeros_like(b)):
        got, info = H.pcg(b, x, tol=1e-9)
        assert got.data_ptr() == x.data_ptr() and info["iterations"] == ri["iterations"]
        assert torch.equal(got, ref)
    capped, info = H.pcg(b, tol=1e-9, maxit=3)
    assert info["iterations"] == 3 and info["status"] == 1
