"""The running median of series of few distinct values (one- or two-bit
samples, gaps filled with a constant): exact as ever, and without a selection
over the window for every output."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _series(rng, n, kind):
    x = rng.standard_normal(n)
    if kind == "const":
        x = np.full(n, 3.25)
    elif kind == "zeros":         # of both signs
        x = np.where(x > 0, 0.0, -0.0)
    elif kind == "one_bit":       # the median moves between the levels
        x = (x > 0).astype(np.float64)
    elif kind == "skew_bit":
        x = (x > 0.3).astype(np.float64)
    elif kind == "two_bit":
        x = np.clip(np.rint(x + 1.5), 0, 3)
    elif kind == "thirds":
        x = np.rint(1.5 * x) / 3.0
    elif kind == "clipped":       # half of the samples at one value, the rest continuous
        x = np.maximum(x, 0.0)
    elif kind == "blocks":        # constant stretches and noise in turn
        x = np.where(np.arange(n) // 700 % 2, x, 0.5)
    elif kind == "many":          # more samples of every level than a bracket holds, more levels than one pass takes
        x = np.rint(6 * x)
    return x


def _oracle(x, w):
    import oracle
    oracle.build()
    return x - oracle.running_median(x, w)


@pytest.mark.parametrize("kind", ["const", "zeros", "one_bit", "skew_bit", "two_bit", "thirds", "clipped", "blocks", "many"])
@pytest.mark.parametrize("n,w", [(900, 129), (5000, 513), (20000, 4001), (30000, 20001), (12000, 62501), (150000, 62501)])
def test_exact(n, w, kind):
    import torch

    from paper_1703_05581_gb300 import ffa

    x = _series(np.random.default_rng(n + w), n, kind)
    st = ffa.status_word()
    got = ffa.detrend(torch.from_numpy(x).cuda(), w, status=st).cpu().numpy()
    assert int(st.item()) == 0
    np.testing.assert_array_equal(got, _oracle(x, w))


def _us(f):
    import torch

    f()
    torch.cuda.synchronize()
    best = 1e9
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 200.0)
    return best


@pytest.mark.parametrize("kind", ["const", "one_bit", "two_bit"])
def test_levels_take_no_selection_for_each_output(kind):
    """At most 8 times a normal series' time (a selection for each output:
    3000 times)."""
    import torch

    from paper_1703_05581_gb300 import ffa

    n, w = 1 << 16, 20001
    rng = np.random.default_rng(5)
    st = ffa.status_word()
    t = []
    for k in ("normal", kind):
        x = torch.from_numpy(_series(rng, n, k)).cuda()
        t.append(_us(lambda: ffa.detrend(x, w, status=st)))
    assert t[1] <= 8 * t[0], t
