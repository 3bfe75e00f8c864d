"""Matching when a device allocation fails: its vectors end the call cleanly, the
array of edge weights (8 bytes an entry, there for speed) does not."""

import ctypes as C

import numpy as np
import pytest
import torch

from synthetic import diffusion3d, gaussian_field

pytestmark = pytest.mark.gpu


def test_matching_without_room_for_edge_weights(amg, orc):
    A = diffusion3d(np.exp(gaussian_field((14, 12, 10), 1.0, 2.0, 5)))
    want = orc.match(A)
    a, keep = amg.csr_struct(*amg.csr_to_device(A))
    lib = amg._lib.load()
    rounds, status = [], []
    for k in range(8):  # more than the call allocates
        mate = torch.full((a.n,), 7, dtype=torch.int32, device="cuda")
        r = C.c_int()
        lib.amg_debug_fail_alloc_after(k)
        try:
            rc = lib.amg_pairwise_match(C.byref(a), C.c_void_p(mate.data_ptr()), C.byref(r), None)
        finally:
            lib.amg_debug_fail_alloc_after(-1)
        status.append(rc)
        if rc == 0:
            assert np.array_equal(mate.cpu().numpy(), want)
            rounds.append(r.value)
    # diagonal, candidates, flags, frontiers, counters; then the weights
    assert status == [amg._lib.AMG_ERR_OOM] * 5 + [0] * 3
    assert len(set(rounds)) == 1
