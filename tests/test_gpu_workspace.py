"""Device workspace of a context."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kbe():
    import torch
    from paper_2405_08737_gb300 import build as B
    B.build()
    import paper_2405_08737_gb300 as K
    torch.cuda.set_device(0)
    return K


def _held(kbe, M, n_max):
    import torch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = kbe.Context(M, n_max)
    held = before - torch.cuda.mem_get_info()[0]
    ctx.close()
    return held


def test_digit_workspace_only_where_a_row_can_use_it(kbe):
    """M = 16: rows go to the tensor cores from 35 points on ((n + 1)^2 M^3 >= 5e6).
    The workspace of one partial sum of 64 KB per SM is in a context of 35 points
    and not in one of 34, whose other parts are all but the same size."""
    import torch
    torch.zeros(1, device="cuda")
    _held(kbe, 16, 35)  # the library's own modules
    least = torch.cuda.get_device_properties(0).multi_processor_count * 65536
    assert _held(kbe, 16, 35) - _held(kbe, 16, 34) > 0.8 * least
