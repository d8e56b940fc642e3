"""Algorithm 1's S/N does not depend on the profile's scale, down to the
smallest numbers FP32 holds: whole numbers times any power of two give the same
records, and as exact ones as in 64 bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p0", [2, 7, 64, 366, 1100, 1101, 2049, 9000, 20001])
def test_scales(p0):
    import torch

    from paper_1703_05581_gb300 import ffa

    n = 40
    g = torch.Generator().manual_seed(p0)
    x = torch.round(60 * torch.randn((n, p0), generator=g))
    x[1::2] += torch.round(40 * torch.rand((n // 2, p0), generator=g)) + 37
    x[2::8] = torch.round(x[2::8] / 50)
    x[:, p0 // 3:p0 // 3 + max(1, p0 // 30)] += 90
    w = [1]
    while w[-1] <= 0.2 * p0:
        w.append(2 * w[-1])
    st = ffa.status_word()
    want = ffa.records_numpy(ffa.score(x.float().cuda(), w, status=st), n)
    d = x.double().numpy()
    med = np.median(d, axis=1)
    mad = np.median(np.abs(d - med[:, None]), axis=1)
    c = np.concatenate([np.zeros((n, 1)), np.cumsum(np.concatenate([d, d[:, :w[-1]]], axis=1), axis=1)], axis=1)
    best = np.full(n, -np.inf)
    with np.errstate(divide="ignore", invalid="ignore"):
        for k in w:
            best = np.maximum(best, ((c[:, k:k + p0] - c[:, :p0]).max(1) - k * med) / (1.4826 * mad * np.sqrt(k)))
    ok = mad > 0
    # the sums are whole numbers below 2^24; four roundings of the quotient
    np.testing.assert_allclose(want["snr"][ok], best[ok], rtol=4 * 2.0 ** -24)
    for e in (-149, -148, -140, -127, -120, -100, -60, 40, 90):
        got = ffa.records_numpy(ffa.score((x.double() * 2.0 ** e).float().cuda(), w, status=st), n)
        assert np.array_equal(got.view(np.uint8), want.view(np.uint8)), e
    assert int(st.item()) == 0
