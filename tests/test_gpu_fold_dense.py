"""Folds whose rows start anywhere: dense planes of every p0 mod 4, series and
planes off 16-byte boundaries, every pass depth from the first pass to plane
to plane, and the padded planes of a search of 12 stages.  The fold adds in one
tree, so every value is compared bit for bit with the plain recursion."""
import pytest

pytestmark = pytest.mark.gpu


def _plain(z, p0, m_data, m_rows):
    import torch

    a = torch.zeros((m_rows, p0), dtype=torch.int32 if z.dtype == torch.int8 else z.dtype, device=z.device)
    a[:m_data] = z[: m_data * p0].view(m_data, p0)
    col = torch.arange(p0, device=z.device)
    s = 1
    while s < m_rows:
        a = a.view(-1, 2, s, p0)
        k = torch.arange(2 * s, device=z.device)
        idx = (col[None, :] + ((k + 1) // 2)[:, None]) % p0
        tail = a[:, 1].repeat_interleave(2, dim=1)
        a = a[:, 0].repeat_interleave(2, dim=1) + tail.gather(2, idx.expand(a.shape[0], -1, -1))
        s *= 2
    return a.view(m_rows, p0)


def _series(n, i8, seed):
    import torch

    z = torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
    return (16 * z).round().clamp(-127, 127).to(torch.int8) if i8 else z


def _fold(z, p0, m_data, m_rows, shift):
    """ffa_fold into a plane `shift` elements past a 16-byte boundary; what
    lies around it must stay as it is."""
    import torch

    from paper_1703_05581_gb300 import ffa

    dt = torch.int32 if z.dtype == torch.int8 else torch.float32
    n = m_rows * p0
    buf = torch.full((n + 64,), 77, dtype=dt, device="cuda")
    tmp = torch.empty(n + 64, dtype=dt, device="cuda")
    plane = buf[32 + shift:32 + shift + n]
    ffa._check(ffa._lib.ffa_fold(ffa._ptr(z), ffa.FOLD_I8 if z.dtype == torch.int8 else ffa.FOLD_F32, p0, m_data, m_rows,
                                 ffa._ptr(plane), ffa._ptr(tmp[shift:]), ffa._stream(None)))
    assert bool((buf[:32 + shift] == 77).all()) and bool((buf[32 + shift + n:] == 77).all())
    return plane.view(m_rows, p0)


# rows: single passes of 0..6 stages, 3+3+.. splits of 7..12, six-stage passes
# plane to plane at 17 and 18 stages
SHAPES = [(r, m) for m in (1, 2, 4, 8, 16, 32, 64, 128, 256, 1024, 2048, 4096) for r in (0, 1, 2, 3)] + \
         [(1, 1 << 17), (2, 1 << 18)]


@pytest.mark.parametrize("i8", [False, True], ids=["f32", "i8"])
@pytest.mark.parametrize("residue,m_rows", SHAPES)
def test_dense_rows(residue, m_rows, i8):
    import torch

    sizes = (20 + residue,) if m_rows > 4096 else (4 + residue, 124 + residue, 252 + residue, 764 + residue, 1532 + residue)
    for p0 in sizes:
        if m_rows >= 2048 and p0 > 800:
            continue
        m_data = max(1, m_rows - m_rows // 5)
        z = _series(m_data * p0 + 8, i8, p0 + m_rows)
        want = _plain(z, p0, m_data, m_rows)
        assert torch.equal(_fold(z, p0, m_data, m_rows, 0), want), p0


@pytest.mark.parametrize("i8", [False, True], ids=["f32", "i8"])
@pytest.mark.parametrize("p0,m_rows", [(766, 1), (767, 2), (516, 4), (765, 16), (1532, 64), (1533, 256), (764, 512)])
def test_series_and_plane_off_boundaries(p0, m_rows, i8):
    import torch

    m_data = max(1, m_rows - 1)
    base = _series(m_data * p0 + 8, i8, p0)
    for a in range(4):
        z = base[a:]
        want = _plain(z, p0, m_data, m_rows)
        for shift in range(4):
            assert torch.equal(_fold(z, p0, m_data, m_rows, shift), want), (a, shift)


@pytest.mark.parametrize("i8", [False, True], ids=["f32", "i8"])
@pytest.mark.parametrize("p0", [636, 637, 638, 639])
def test_padded_planes_of_twelve_stages(p0, i8):
    """2049..4096 data rows: two passes of six stages on a search's padded
    planes, the second from plane to plane."""
    import torch

    from paper_1703_05581_gb300 import ffa

    n = p0 * 2500
    ts = 64e-6
    plan = ffa.Plan(ffa.Config(tsamp=ts, period_min=p0 * ts, period_max=(p0 + 1) * ts, detrend_window=-1,
                               precision=ffa.FOLD_I8 if i8 else ffa.FOLD_F32), n)
    assert plan.entries["m_rows"][0] == 4096 and plan.entries["p0"][0] == p0
    x = _series(n, False, p0)
    z = ffa.search_series(plan, x, 0)
    assert torch.equal(ffa.search_plane(plan, x, 0), _plain(z, p0, 2500, 4096))
