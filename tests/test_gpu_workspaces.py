"""Workspaces that a handle keeps between calls: an allocation that fails while
one grows leaves the handle usable, for fewer columns or samples and for as many."""

import pytest
import torch

from synthetic import poisson3d, uniform01

pytestmark = pytest.mark.gpu


def _fails_at(amg, k, call):
    """The k-th device allocation of `call` fails; whether that ended it."""
    from paper_2406_19754_gb300 import _lib

    lib = _lib.load()
    lib.amg_debug_fail_alloc_after(k)
    try:
        call()
    except amg.AmgError as e:
        assert e.status == _lib.AMG_ERR_OOM
        return True
    finally:
        lib.amg_debug_fail_alloc_after(-1)
    return False


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_multi_workspace_survives_a_failed_allocation(amg, precision):
    n = 13 * 11 * 9
    A = amg.csr_to_device(poisson3d(13, 11, 9))
    H = amg.Hierarchy(*A, precision=precision, max_coarse=40)
    B = torch.as_tensor(uniform01(52, n * 8), device="cuda").reshape(n, 8)
    few, many = B[:, :2].contiguous(), B
    want = [amg.Hierarchy(*A, precision=precision, max_coarse=40).pcg_multi(b)[0]
            for b in (few, many)]
    k = 0
    while _fails_at(amg, k, lambda: H.pcg_multi(many)):
        assert torch.equal(H.pcg_multi(few)[0], want[0])  # grows from nothing to two
        k += 1
    assert k >= 9  # vectors, partial sums, scalars, then three vectors a level
    assert torch.equal(H.pcg_multi(few)[0], want[0])
    assert torch.equal(H.pcg_multi(many)[0], want[1])


def test_multi_workspace_keeps_its_capacity(amg):
    # a call with fewer columns in between: the buffers of the larger one stay
    n = 9 * 8 * 7
    H = amg.Hierarchy(*amg.csr_to_device(poisson3d(9, 8, 7)), max_coarse=40)
    B = torch.as_tensor(uniform01(53, n * 8), device="cuda").reshape(n, 8)
    x = H.pcg_multi(B)[0]
    H.pcg_multi(B[:, :3].contiguous())
    out = []
    assert not _fails_at(amg, 0, lambda: out.append(H.pcg_multi(B)[0]))
    assert torch.equal(out[0], x)
