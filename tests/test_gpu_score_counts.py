"""A profile's record does not depend on how many profiles are scored with it:
calls of a few profiles take more threads a profile than calls that fill the
GPU, at every length where the choice changes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [7, 197, 198, 384, 385, 1200, 1201, 1537, 2048, 2049, 4111, 8192, 8193, 10240, 10241, 16384, 16385, 20479, 20481]


@pytest.mark.parametrize("ints", [False, True], ids=["f32", "i32"])
@pytest.mark.parametrize("p0", SIZES)
def test_records_of_every_count(p0, ints):
    import torch

    from paper_1703_05581_gb300 import ffa

    n = 1000
    g = torch.Generator(device="cuda").manual_seed(p0)
    x = 20 * torch.randn((n, p0), generator=g, device="cuda")
    x[1::3] = torch.round(x[1::3] / 25)             # few distinct values
    x[2::3] += 30 * torch.rand((len(x[2::3]), p0), generator=g, device="cuda").square()
    x = x.round().to(torch.int32) if ints else x
    widths = [1]
    while widths[-1] <= 0.2 * p0:
        widths.append(2 * widths[-1])
    st = ffa.status_word()
    want = ffa.score(x, widths, status=st).cpu().numpy()
    for k in (1, 150, 310, 500, 800):
        part = ffa.score(x[n - k:].contiguous(), widths, status=st).cpu().numpy()
        np.testing.assert_array_equal(part, want[n - k:])
    assert int(st.item()) == 0
