"""Algorithm 1 on float profiles of few distinct values or with gaps (sums of
a few rows of a one- or two-bit series): the median and the MAD are then far
from any window of the predicted width.  Records against 64-bit arithmetic,
and no more than a few times an ordinary profile's time."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 9, 64, 197, 198, 700, 1100, 1489, 2048, 2049, 6001, 16384, 20479, 30001]
KINDS = ["two", "halves", "four", "sixteen", "thirds", "offset", "outlier", "few_off", "lone_gap"]


def _profiles(rng, n, p0, kind):
    u = rng.random((n, p0))
    if kind == "two":          # a third and two thirds
        x = np.where(u < 0.35, -0.7, 1.9)
    elif kind == "halves":     # the median of an even length lies between the levels
        x = np.where(np.argsort(u, axis=1) < p0 // 2, -1.1, 0.3)
    elif kind == "four":
        x = np.floor(4 * u) * 1.37 - 2.0
    elif kind == "sixteen":
        x = np.floor(16 * u) * 1.37 - 11.0
    elif kind == "thirds":     # levels no float holds exactly, at uneven distances
        x = np.array([-1.0 / 3, 0.1, 0.7, 1.0 / 7])[np.floor(4 * u).astype(int)]
    elif kind == "offset":     # deviations that differ in the last bits only
        x = 4000.0 + np.floor(3 * u) / 3.0
    elif kind == "outlier":
        x = np.floor(5 * u)
        x[:, p0 // 2] = 3e4
    elif kind == "few_off":    # more than half equal: the MAD is 0
        x = np.where(u < 0.3, np.floor(10 * u), 2.5)
    else:                      # one sample between two far groups
        x = np.where(u < 0.5, -50.0, 50.0) + 1e-3 * rng.standard_normal((n, p0))
        x[:, 0] = 1.0
    return x.astype(np.float32)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("p0", SIZES)
def test_levels(p0, kind):
    import torch

    from paper_1703_05581_gb300 import ffa

    n = 6
    x = _profiles(np.random.default_rng([p0, KINDS.index(kind)]), n, p0, kind)
    w = [1]
    while w[-1] <= 0.2 * p0:
        w.append(2 * w[-1])
    st = ffa.status_word()
    got = ffa.records_numpy(ffa.score(torch.from_numpy(x).cuda(), w, status=st), n)
    assert int(st.item()) == 0
    d = x.astype(np.float64)
    med = np.median(d, axis=1)
    mad = np.median(np.abs(d - med[:, None]), axis=1)
    np.testing.assert_array_equal(got["flags"] != 0, mad == 0)
    c = np.concatenate([np.zeros((n, 1)), np.cumsum(np.concatenate([d, d[:, :w[-1]]], axis=1), axis=1)], axis=1)
    for i in np.flatnonzero(mad > 0):
        box = np.array([c[i, k:k + p0] - c[i, :p0] for k in w])
        snr = (box - np.array(w)[:, None] * med[i]) / (1.4826 * mad[i] * np.sqrt(np.array(w))[:, None])
        # box sums are FP32 sums of in-block prefixes: at most 31 samples of
        # rounding 2^-24 of the prefix on each side
        tol = 64 * 2.0 ** -24 * np.abs(d[i]).max() * 32 / (1.4826 * mad[i]) + 2e-6 * np.abs(snr).max()
        best = snr.max()
        assert abs(got["snr"][i] - best) <= tol
        assert snr[w.index(int(got["width"][i])), int(got["phase"][i])] >= best - 2 * tol


def _graph_us(f):
    import torch

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        f()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(10):
                f()
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(s)
            g.replay()
            b.record(s)
            b.synchronize()
            best = min(best, a.elapsed_time(b) * 100.0)
    return best


@pytest.mark.parametrize("p0,n,levels", [(64, 150, 2), (366, 150, 4), (1100, 3000, 16), (3001, 150, 16)])
def test_levels_take_no_selection_over_all_bits(p0, n, levels):
    """At most 2.5 times the time of normal profiles (a radix select over 64
    bits: 3.9 to 7 times)."""
    import torch

    from paper_1703_05581_gb300 import ffa

    g = torch.Generator(device="cuda").manual_seed(p0)
    a = torch.randn((n, p0), generator=g, device="cuda")
    b = (torch.randint(0, levels, (n, p0), generator=g, device="cuda").float() - (levels - 1) / 2) * 1.37
    w = [1, 2, 4, 8, 16]
    st = ffa.status_word()
    t = [_graph_us(lambda x=x: ffa.score(x, w, status=st)) for x in (a, b)]
    assert t[1] <= 2.5 * t[0], t
