"""Matrices whose nnz field understates what their row pointers hold (as small as
the checks on entry let it be): matching and set-up go by the row pointers."""

import ctypes as C

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field, uniform01

pytestmark = pytest.mark.gpu

SHAPE, N = (14, 12, 10), 1680


def _understated(amg):
    A = diffusion3d(np.exp(gaussian_field(SHAPE, 1.0, 2.0, 5)))
    Ad = amg.csr_to_device(A)
    a, keep = amg.csr_struct(*Ad)
    assert a.nnz > 5 * a.n
    a.nnz = a.n
    return A, Ad, a, keep


def test_matching_goes_by_the_row_pointers(amg, orc):
    A, _, a, keep = _understated(amg)
    mate = torch.empty(N, dtype=torch.int32, device="cuda")
    lib = amg._lib.load()
    assert lib.amg_pairwise_match(C.byref(a), C.c_void_p(mate.data_ptr()), None, None) == 0
    assert np.array_equal(mate.cpu().numpy(), orc.match(A))


def test_setup_goes_by_the_row_pointers(amg):
    _, Ad, a, keep = _understated(amg)
    H = amg.Hierarchy(*Ad)  # as stated
    lib, h = amg._lib.load(), C.c_void_p()
    o = amg.options()
    assert lib.amg_setup(C.byref(a), C.byref(o), None, C.byref(h)) == 0
    r = torch.as_tensor(uniform01(6, N), device="cuda")
    z = torch.empty_like(r)
    torch.cuda.synchronize()
    assert lib.amg_vcycle_apply(h, C.c_void_p(r.data_ptr()), C.c_void_p(z.data_ptr()), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(z, H.vcycle(r))
    assert lib.amg_destroy(h) == 0
