"""The injected barrier time-out on hierarchies whose small levels also fit one
cluster's shared memory (which has no grid barrier): it is reported all the same,
and the handle works again once the hook is off."""

import pytest
import torch

from synthetic import poisson3d, uniform01

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("side", [42, 48])  # level 1: 18,522 and 27,648 rows in BF16
def test_time_out_reported_where_the_cluster_would_run(amg, side, use_graph):
    from paper_2406_19754_gb300 import _lib

    n = side ** 3
    opts = dict(precision="f32", bf16_from_level=1, tail_rows=30000)
    A = amg.csr_to_device(poisson3d(side))
    H = amg.Hierarchy(*A, **opts)
    b = torch.as_tensor(uniform01(3, n), device="cuda")
    x_ref, info_ref = H.pcg(b, tol=1e-8, use_graph=use_graph)
    lib = _lib.load()
    assert lib.amg_debug_tail_timeout(H.h, 1) == 0
    with pytest.raises(amg.AmgError) as e:
        H.pcg(b, tol=1e-8, use_graph=use_graph)
    assert e.value.status == _lib.AMG_ERR_DEVICE_CHECK
    assert lib.amg_debug_tail_timeout(H.h, 0) == 0
    x, info = H.pcg(b, tol=1e-8, use_graph=use_graph)
    assert info["status"] == 0 and info["iterations"] == info_ref["iterations"]
    assert torch.equal(x, x_ref)
