"""The fold's staging takes rows that start on its alignment pattern by 16-byte
copies and every other row element by element: all residues of P0, views that
start off a 16-byte boundary, rows that wrap in every pass, and more tiles than
resident CTAs must give the recursion's sums bit for bit."""
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


# P0 of every residue mod 4 around tile edges; rows for one to three passes
CASES = [(127, 64, 64), (128, 60, 64), (129, 64, 64), (190, 100, 128), (191, 128, 128), (193, 2000, 2048),
         (254, 33, 64), (255, 17, 32), (257, 9, 16), (318, 4000, 4096), (319, 5, 8), (447, 700, 1024), (1026, 513, 1024)]


@pytest.mark.parametrize("p0,m_data,m", CASES)
@pytest.mark.parametrize("integer", [False, True])
@pytest.mark.parametrize("start", [0, 1, 3])
def test_fold_alignments(F, orc, p0, m_data, m, integer, start):
    import torch
    rng = np.random.default_rng(p0 * 7 + m + start)
    n = m_data * p0 + start
    if integer:
        z = rng.integers(-127, 128, n).astype(np.int8)
    else:
        z = rng.standard_normal(n).astype(np.float32)
    got = F.fold(torch.from_numpy(z).cuda()[start:], p0, m_data, m).cpu().numpy()
    rows = np.zeros((m, p0), np.int64 if integer else np.float32)
    rows[:m_data] = z[start:].reshape(m_data, p0)
    assert np.array_equal(got.astype(rows.dtype), orc.fold(rows))


def test_search_plane_many_tiles(F, orc):
    """The search's padded planes, six stages per pass, more tiles than CTAs."""
    import torch
    p0, n = 2503, 2503 * 900 + 77
    rng = np.random.default_rng(11)
    x = rng.standard_normal(n).astype(np.float32)
    cfg = F.Config(tsamp=1.0, period_min=p0, period_max=p0 + 1, detrend_window=-1)
    plan = F.Plan(cfg, n)
    xs = torch.from_numpy(x).cuda()
    z = F.search_series(plan, xs, 0).cpu().numpy()
    got = F.search_plane(plan, xs, 0).cpu().numpy()
    rows = np.zeros((1024, p0), np.float32)
    rows[:900] = z[: 900 * p0].reshape(900, p0)
    assert np.array_equal(got, orc.fold(rows))
