"""Dense-interaction self-energy: the result does not depend on how the call
is run (direct, captured in a graph), and calls that need no workspace wait for none."""
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


def _ctx(kbe, M, n_max):
    ctx = kbe.Context(M, n_max)
    t, order = W.grid(n_max, 0.05, 0.3, 1)
    ctx.set_grid(t, order)
    ctx.set_model(W.chain_h(M), np.ones(M), W.site_potential(M), None)
    rng = np.random.default_rng(M)
    ctx.set_interaction(rng.standard_normal((M,) * 4) / M)
    return ctx


def _data(M, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    return (torch.randn(W.tri_size(n + 1), M, M, dtype=torch.complex128, device="cuda", generator=g) for _ in range(2))


# rows whose blocks are split over several units and not (M < 8; all SMs busy)
@pytest.mark.parametrize("M,n", [(5, 9), (8, 3), (8, 40), (11, 17), (16, 12), (16, 60), (8, 150), (24, 4), (32, 2)])
def test_captured_row_is_the_direct_row(kbe, M, n):
    """Bitwise: the slices of a block are summed in the same order."""
    import torch
    ctx = _ctx(kbe, M, n + 1)
    L, R = _data(M, n)
    out = [torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda") for _ in range(2)]
    ctx.selfenergy_slice(n, L, R, out[0][0], out[0][1])
    ctx.sync_status()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.selfenergy_slice(n, L, R, out[1][0], out[1][1])
    g.replay()
    ctx.sync_status()
    assert out[0].abs().max() > 0 and torch.equal(out[0], out[1])
    ctx.close()


def test_balanced_rows_stay_whole(kbe):
    """Rows that fill every SM alike are not split (M = 8: 0.92 of the speed), the
    rows around them are."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 3 * sms // 2 - 1  # three units per SM
    ctx = _ctx(kbe, 8, n + 30)
    L, R = _data(8, n + 29)
    S = torch.zeros((2, n + 30, 8, 8), dtype=torch.complex128, device="cuda")
    launches = []
    for row in (n, n + 10, n // 2):
        ctx.selfenergy_slice(row, L, R, S[0], S[1])
        launches.append(ctx.last_launch_count)
    ctx.sync_status()
    assert launches == [1, 2, 2]
    ctx.close()


def test_whole_rows_wait_for_no_other_stream(kbe):
    """A call that needs no workspace runs beside split rows of another stream:
    it is done before the last of them."""
    import torch
    M, n, rows = 16, 255, 50
    ctx = _ctx(kbe, M, n + 1)
    L, R = _data(M, n)
    S = torch.zeros((2, n + 1, M, M), dtype=torch.complex128, device="cuda")
    T = torch.zeros((2, W.tri_size(rows), M, M), dtype=torch.complex128, device="cuda")
    ctx.selfenergy_all(rows, L, R, T[0], T[1])
    assert ctx.last_launch_count == 1  # not split
    ctx.sync_status()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    done = torch.cuda.Event()
    for _ in range(20):  # about 10 ms each
        ctx.selfenergy_slice(n, L, R, S[0], S[1], stream=a)
        assert ctx.last_launch_count == 2
    done.record(a)
    ctx.selfenergy_all(rows, L, R, T[0], T[1], stream=b)
    b.synchronize()
    assert not done.query()
    torch.cuda.synchronize()
    ctx.sync_status()
    ctx.close()
