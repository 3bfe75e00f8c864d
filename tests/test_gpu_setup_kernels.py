"""Setup kernels at the sizes where they change path: the panel Cholesky at
its panel edges (32 columns), Galerkin rows around 64 contributions (two per
lane; longer rows are sorted by a whole warp), and the blocks a setup reuses
(two hierarchies in a row, and one built after another was destroyed)."""

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, uniform01
from tests.helpers import dense, random_spd_graph

pytestmark = pytest.mark.gpu


def _np(t):
    return t.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 301])
def test_cholesky_at_panel_edges(amg, n):
    # one level: z = L^-T L^-1 b.  The matrices are strictly diagonally dominant
    # (row sums of |off| plus at least 0.5), condition number below 4 n: the
    # backward error bound n eps cond stays under 1e-10 here
    A = random_spd_graph(n, min(1.0, 8.0 / n), 40 + n)
    H = amg.Hierarchy(*amg.csr_to_device(A), max_coarse=n)
    assert H.levels == 1
    b = uniform01(n, n)
    z = _np(H.vcycle(torch.as_tensor(b, device="cuda")))
    np.testing.assert_allclose(z, np.linalg.solve(dense(A), b), rtol=1e-10, atol=1e-13)


@pytest.mark.parametrize("p", [0.02, 0.04, 0.055, 0.07, 0.3])
@pytest.mark.parametrize("sweeps", [1, 2])
def test_galerkin_row_lengths_bit_exact(amg, orc, p, sweeps):
    # rows of about 300 p entries: 2 or 4 members below, around and above 64
    A = random_spd_graph(300, p, 17, positive_offdiag=True)
    H = amg.Hierarchy(*amg.csr_to_device(A), sweeps=sweeps, max_coarse=40)
    Ho = orc.Hierarchy(A, sweeps=sweeps, max_coarse=40, max_dense=2048)
    assert H.levels == Ho.levels
    for l in range(1, H.levels):
        ex, (rp, ci, v) = H.level_export(l), Ho.level_csr(l)
        assert np.array_equal(_np(ex["rowptr"]), rp) and np.array_equal(_np(ex["col"]), ci)
        assert np.array_equal(_np(ex["val"]), v)


def test_csr_with_an_offset_row_pointer(amg, orc):
    # rowptr[0] > 0: a view into larger arrays; edge weights are stored per entry
    A = diffusion3d(np.exp(gaussian_field((9, 8, 7), 1.0, 2.0, 3)))
    rp, ci, v = A
    pad = 5
    big = (rp + pad, np.concatenate([np.zeros(pad, np.int32), ci]),
           np.concatenate([np.zeros(pad), v]))
    Ad = amg.csr_to_device(big)
    from paper_2406_19754_gb300 import _lib
    import ctypes as C

    mate = torch.empty(len(rp) - 1, dtype=torch.int32, device="cuda")
    a = amg.AmgCsr(len(rp) - 1, len(ci), C.c_void_p(Ad[0].data_ptr()),
                   C.c_void_p(Ad[1].data_ptr()), C.c_void_p(Ad[2].data_ptr()))
    rounds = C.c_int()
    assert _lib.load().amg_pairwise_match(C.byref(a), C.c_void_p(mate.data_ptr()),
                                          C.byref(rounds), None) == 0
    assert np.array_equal(_np(mate), orc.match(A))


def test_hierarchies_do_not_share_blocks(amg):
    A = diffusion3d(np.exp(gaussian_field((30, 28, 26), 1.5, 4.0, 8)))
    n = 30 * 28 * 26
    Ad = amg.csr_to_device(A)
    r = torch.as_tensor(uniform01(2, n), device="cuda")
    H1 = amg.Hierarchy(*Ad)
    z = H1.vcycle(r).clone()
    H2 = amg.Hierarchy(*Ad, precision="f32")
    z2 = H2.vcycle(r).clone()
    assert torch.equal(H1.vcycle(r), z)
    H1.close()
    H3 = amg.Hierarchy(*Ad)
    assert torch.equal(H2.vcycle(r), z2) and torch.equal(H3.vcycle(r), z)
