"""The bounded waits of the FP64 slices on the tensor cores."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kbe():
    import torch
    from paper_2405_08737_gb300 import build as B
    B.build()
    import paper_2405_08737_gb300 as K
    torch.cuda.set_device(0)
    return K


@pytest.mark.parametrize("M,n,precision", [(8, 200, "fp64"), (5, 260, "fp64"), (16, 60, "df64"), (13, 60, "fp64")])
@pytest.mark.parametrize("unit", [0, 3])
def test_a_wait_that_runs_out_is_reported(kbe, M, n, precision, unit):
    """Every CTA's producer withholds one unit and the waits give up after a
    fraction of a millisecond: the launch returns, the status reads
    KBE_ETIMEOUT, and the next slice on the same context has the bits of the first."""
    import torch
    t, order = W.grid(n + 1, 0.05, 0.3, 1)
    ctx = kbe.Context(M, n + 1)
    ctx.set_grid(t, order)
    ctx.set_model(W.goe_h(M, 1), np.ones(M), W.site_potential(M), None)
    L, R = (torch.as_tensor(x, device="cuda") for x in W.random_triangles(M, n + 1, 1))
    Sl, Sg = (torch.as_tensor(x, device="cuda") for x in W.random_rows(M, n, 2))
    out = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    ctx.history_slice(n, L, R, Sl, Sg, out, precision=precision)
    assert ctx.last_launch_count == 3
    ctx.sync_status()
    first = out.clone()
    ctx.debug_withhold_split(unit, 4096)
    ctx.history_slice(n, L, R, Sl, Sg, out, precision=precision)
    with pytest.raises(kbe.KBEError) as e:
        ctx.sync_status()
    assert e.value.status == kbe.KBE_ETIMEOUT
    out.fill_(float("nan"))
    ctx.history_slice(n, L, R, Sl, Sg, out, precision=precision)
    ctx.sync_status()
    assert torch.equal(out, first)
    ctx.close()
