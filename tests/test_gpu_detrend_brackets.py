"""The running median guesses a bracket for each tile from the tile before it:
series whose median jumps, drifts fast, takes few values or is flat, at windows
of every tile size and at lengths around tile and run edges, must come out
exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_1703_05581_gb300 import ffa
    return ffa


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _series(rng, n, kind):
    x = rng.standard_normal(n)
    if kind == "steps":
        x += np.repeat(rng.uniform(-50, 50, n // 3001 + 1), 3001)[:n]
    elif kind == "drift":
        x = 0.01 * x + 1e-3 * np.arange(n)
    elif kind == "levels":
        x = np.rint(16 * x + 128)
    elif kind == "halves":  # the median hops between two far values
        x = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    elif kind == "zeros":   # signed zeros and a flat stretch
        x = np.where(rng.random(n) < 0.7, rng.choice([-0.0, 0.0], n), x)
    elif kind == "spikes":
        x[rng.integers(0, n, n // 50)] *= 1e200
    return x


@pytest.mark.parametrize("n,w", [(128, 129), (4097, 129), (33000, 259), (33000, 515), (66001, 1023),
                                 (200_000, 2047), (700_001, 4101), (900_000, 20_001)])
@pytest.mark.parametrize("kind", ["steps", "drift", "levels", "halves", "zeros", "spikes"])
def test_bracketed_median(F, orc, n, w, kind):
    import torch
    rng = np.random.default_rng(n + w)
    x = _series(rng, n, kind)
    st = F.status_word()
    got = F.detrend(torch.from_numpy(x).cuda(), w, status=st).cpu().numpy()
    assert int(st.item()) == 0
    assert np.array_equal(got, x - orc.running_median(x, w | 1))
