"""Algorithm 1's selections on profiles that are hard to predict: the median
and the MAD are looked for in a window placed from the profile's mean and
spread, so skewed, two-humped, quantised and offset profiles, and every CTA
shape's smallest and largest length, must give the oracle's records too."""
import numpy as np
import pytest

from parity import check_records

pytestmark = pytest.mark.gpu

SIZES = [3, 8, 33, 1200, 1201, 2048, 2049, 8193, 16385, 20479, 20481, 31249]
KINDS = ["normal", "levels", "codes", "humps", "skewed", "wave", "offset", "ramp"]


@pytest.fixture(scope="module")
def F():
    from paper_1703_05581_gb300 import ffa
    return ffa


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _profile(rng, p0, kind):
    x = rng.standard_normal(p0)
    if kind == "levels":     # few distinct values: long runs of ties
        x = np.rint(2.0 * x)
    elif kind == "codes":    # a quantised series' sums: clusters of tens of equal values
        x = np.rint(50.0 * x) / 3.0
    elif kind == "humps":    # no samples near the mean
        x = np.where(rng.random(p0) < 0.3, 20.0, 0.0) + 0.1 * x
    elif kind == "skewed":
        x = np.exp(1.5 * x)
    elif kind == "wave":     # red noise: a slow wave above the noise
        x = 0.3 * x + 3.0 * np.sin(2 * np.pi * np.arange(p0) / p0 + rng.random())
    elif kind == "offset":
        x = x + 50.0
    elif kind == "ramp":
        x = np.arange(p0) / 7.0
    return x


def _widths(p0):
    w = [1]
    while w[-1] <= 0.1 * p0:
        w.append(2 * w[-1])
    return tuple(w)


def _run(F, prof, widths):
    import torch
    st = F.status_word()
    rec = F.score(torch.from_numpy(prof).cuda(), widths, status=st)
    got = F.records_numpy(rec, prof.shape[0])
    assert int(st.item()) == 0
    return got


@pytest.mark.parametrize("p0", SIZES)
@pytest.mark.parametrize("integer", [False, True])
def test_selection_windows(F, orc, p0, integer):
    rng = np.random.default_rng(p0 + 7 * integer)
    x = np.stack([_profile(rng, p0, k) for k in KINDS for _ in range(2)]) * 37.0
    prof = np.rint(x).astype(np.int32) if integer else x.astype(np.float32)
    widths = _widths(p0)
    got = _run(F, prof, widths)
    dt = np.int64 if integer else np.float64
    ref = np.array([orc.score_alg1(p.astype(dt), widths) for p in prof])
    # FP32 in-block sums of at most 32 bins of 50 sigma: below 1e-4 of K*MAD
    # per box, and S/N values up to a few hundred carry 2e-7 of themselves
    tol = 1e-3 + 2e-7 * float(np.abs(ref["snr"]).max())
    check_records(got, ref, lambda i: prof[i].astype(np.float64), tol=tol)
    if integer:
        assert np.array_equal(got["snr"], ref["snr"].astype(np.float32))


def test_consecutive_trials_change_shape(F, orc):
    """More trials than resident CTAs, their distributions alternating: a
    CTA's earlier trials mispredict the next one's windows."""
    rng = np.random.default_rng(5)
    p0, n = 96, 9000
    prof = np.stack([_profile(rng, p0, KINDS[i % len(KINDS)]) * (1.0 + i % 5) for i in range(n)]).astype(np.float32)
    widths = (1, 2, 4, 8, 16)
    got = _run(F, prof, widths)
    pick = np.arange(0, n, 17)
    ref = np.array([orc.score_alg1(prof[i].astype(np.float64), widths) for i in pick])
    check_records(got[pick], ref, lambda i: prof[pick[i]].astype(np.float64), tol=1e-3)


def test_wide_integers(F, orc):
    """Integers whose doubled deviations leave int32."""
    rng = np.random.default_rng(6)
    prof = rng.integers(-(1 << 30), 1 << 30, (6, 501)).astype(np.int32)
    got = _run(F, prof, (1,))
    ref = np.array([orc.score_alg1(p.astype(np.int64), (1,)) for p in prof])
    ref["snr"] = ref["snr"].astype(np.float32)  # a record holds the rounded quotient
    check_records(got, ref, lambda i: prof[i].astype(np.float64), tol=0.0)


@pytest.mark.parametrize("p0", [1, 2, 5, 8, 33, 257, 2047, 2049, 4201, 8193, 16385, 31249])
@pytest.mark.parametrize("integer", [False, True])
def test_alg2_block_edges(F, orc, p0, integer):
    """Algorithm 2 at lengths around blocks, chunks and CTA shapes, with a box
    that starts in the last, partial block and a flat profile."""
    import torch
    rng = np.random.default_rng(p0 * 5 + integer)
    x = rng.standard_normal((6, p0)) * 37.0
    x[1, -1] += 900.0
    x[2, np.arange(p0 - min(p0, 9), p0 + min(p0, 9)) % p0] += 300.0
    x[3, :] = 4.0
    prof = np.rint(x).astype(np.int32) if integer else x.astype(np.float32)
    widths = _widths(p0)
    rec = F.score_alg2(torch.from_numpy(prof).cuda(), widths)
    got = F.records_numpy(rec, prof.shape[0])
    ref = np.array([orc.score_alg2(p.astype(np.float64), widths) for p in prof])
    # FP32 sums of the profile and of the window: 1e-4 of the score, as for the
    # other lengths this scorer is compared at
    tol = 1e-3 + 1e-4 * float(np.abs(ref["snr"]).max())
    check_records(got, ref, lambda i: prof[i].astype(np.float64), tol=tol, scorer=2)
