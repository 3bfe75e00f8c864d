"""Workspaces that a handle keeps between calls: an allocation that fails while
one grows leaves the handle usable, for fewer columns or samples and for as many."""

import pytest
import torch

from synthetic import poisson3d, standard_normal, uniform01

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


def test_twogrid_workspace_survives_a_failed_allocation(amg):
    from paper_2406_19754_gb300 import learned

    n = 12 * 11 * 10
    A = amg.csr_to_device(poisson3d(12, 11, 10))
    e0 = torch.as_tensor(standard_normal(54, 9 * n).reshape(9, n), device="cuda")
    ref = amg.Hierarchy(*A, max_coarse=20)
    want = {k: learned.twogrid_loss(ref, e0[:k], 2)[0] for k in (2, 9)}

    def check(H, k):  # in groups of any size: inner solves to 1e-12
        loss = learned.twogrid_loss(H, e0[:k], 2)[0]
        assert abs(loss - want[k]) <= 1e-9 * abs(want[k])

    # the inner hierarchy's set-up fails: the call ends, a later one starts over
    H = amg.Hierarchy(*A, max_coarse=20)
    for k in (0, 3, 40):
        assert _fails_at(amg, k, lambda: check(H, 9))
    check(H, 2)
    # the growth to groups of eight fails at each of its allocations (ten vectors,
    # two a cycle, the blocked workspace): a smaller group takes over
    for k in range(36):
        H = amg.Hierarchy(*A, max_coarse=20)
        check(H, 2)
        assert not _fails_at(amg, k, lambda: check(H, 9))
        check(H, 2)
        check(H, 9)
