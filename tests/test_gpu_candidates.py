"""The candidate selection on records made up to be hard to select from: many
equal S/N (all digits of the key down to the trial index), counts around the
point where the passes end early, 0 and 4096 candidates, nothing above the
threshold, infinities and NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def search():
    from paper_1703_05581_gb300 import ffa

    ts = 2.048e-3
    plan = ffa.Plan(ffa.Config(tsamp=ts, period_min=256 * ts, period_max=400 * ts, widths=(1, 2, 4)), 65536)
    return ffa, plan, plan.workspace()


def _snr(rng, n, kind):
    s = (4 + rng.random(n)).astype(np.float32)
    if kind == "equal":
        s[:] = 7.25
    elif kind == "two_values":
        s = np.where(rng.random(n) < 0.01, 9.0, 8.0).astype(np.float32)
    elif kind.startswith("ties"):  # that many at the top value, all others lower
        s[rng.permutation(n)[:int(kind[4:])]] = 12.5
    elif kind == "low_bits":       # S/N that differ in the last bits only
        s = (np.float32(8).view(np.int32) + rng.integers(0, 900, n).astype(np.int32)).view(np.float32)
    elif kind == "special":
        s[::7] = np.nan
        s[3::11] = -np.inf
        s[5] = s[9] = np.inf
        s[1::13] = -0.0
    elif kind == "below":
        s -= 6
    return s


@pytest.mark.parametrize("kind", ["plain", "equal", "two_values", "ties511", "ties512", "ties513", "ties4095", "ties4097",
                                  "low_bits", "special", "below"])
def test_selection(search, kind):
    import torch

    ffa, plan, ws = search
    n = plan.n_trials
    snr = _snr(np.random.default_rng(n), n, kind)
    rec = torch.zeros((n, 4), dtype=torch.int32)
    rec[:, 0] = torch.from_numpy(snr.view(np.int32).copy())
    rec[:, 1], rec[:, 2] = 2, torch.arange(n, dtype=torch.int32) % 251
    rec = rec.cuda()
    e = plan.entries
    for e0, e1 in ((0, plan.n_periods), (3, 4), (10, 29)):
        t0 = int(e["first_trial"][e0])
        t1 = int(e["first_trial"][e1 - 1] + e["m_rows"][e1 - 1])
        part = snr[t0:t1]
        order = np.lexsort((np.arange(t0, t1), -part))
        order = order[part[order] >= 3.0]
        for k in (0, 1, 16, 255, 256, 257, 4096):
            got, best = ffa.candidates_entries(plan, e0, e1, rec, ws, snr_min=3.0, top_k=k)
            want = order[:k] + t0
            np.testing.assert_array_equal(got["trial"], want)
            np.testing.assert_array_equal(got["snr"], snr[want])
            np.testing.assert_array_equal(got["phase"], want % 251)
            if not np.isnan(part).any():
                assert best == t0 + int(np.argmax(part))
