"""What the host side chooses for a launch, seen on a CUDA runtime that runs
nothing."""
import fakecuda
import pytest


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.build(tmp_path_factory.mktemp("fake"))


def test_resident_ctas_by_thread_count(fake):
    """The CTAs that fit the GPU depend on the thread count as much as on the
    shared memory, whichever thread count was asked for first."""
    got = fakecuda.run(fake, """
fn = lib._ZN3ffa13resident_ctasEPKvimPl
def ctas(kernel, threads, smem):
    out = C.c_int64()
    assert fn(C.c_void_p(kernel), C.c_int(threads), C.c_size_t(smem), C.byref(out)) == 0
    return out.value
emit([ctas(64, t, 20000) for t in (1024, 256, 1024)] + [ctas(128, t, 20000) for t in (256, 1024)])
""")
    assert got == [2 * 152, 8 * 152, 2 * 152, 8 * 152, 2 * 152]


def test_tuned_shape_of_padded_rows_only(fake):
    """The autotuner times a search's padded planes: a fold of dense rows that
    are not 16-byte aligned keeps the passes it had."""
    got = fakecuda.run(fake, """
def passes(p0):
    fake.fake_reset()
    assert lib.ffa_fold(BUF, 0, C.c_int64(p0), C.c_int64(4000), C.c_int64(4096), BUF, BUF, None) == 0
    return sum("k_fold" in x[0] for x in launches())
before = [passes(9001), passes(9004)]
ts = 64e-6
h = plan(config(tsamp_s=ts, period_min_s=9000 * ts, period_max_s=9010 * ts, detrend_window=-1), 9000 * 8000)
ws, n = C.c_size_t(), C.c_int32()
lib.ffa_plan_info(h, None, None, None, None, C.byref(ws))
assert lib.ffa_autotune(h, BUF, ws, None, C.byref(n)) == 0 and n.value == 1
emit([before, [passes(9001), passes(9004)]])
""")
    before, after = got
    assert after[0] == before[0]
    assert before[1] == 2 and after[1] == 4  # tuned to three stages a pass: every shape takes as long here


def test_few_profiles_get_more_threads(fake):
    """A scoring call that leaves each SM a few profiles takes the latency of
    one: it gets more threads a profile than a call that fills the GPU, and
    no more than the SM holds."""
    got = fakecuda.run(fake, """
out = {}
for prec in (0, 1):
    for p0 in (64, 700, 1100, 1489, 2048, 2049, 3001, 6000, 9001, 16000, 20000, 30001):
        for n in (1, 152, 153, 304, 500, 900, 8000):
            fake.fake_reset()
            w = (C.c_int32 * 3)(1, 2, 4)
            assert lib.ffa_score(BUF, prec, C.c_int64(n), C.c_int64(p0), w, 3, BUF, BUF, None) == 0
            (name, grid, block, smem), = launches()
            out["%d %d %d" % (prec, p0, n)] = (grid, block, smem)
emit(out)
""")
    for key, (grid, block, smem) in got.items():
        prec, p0, n = map(int, key.split())
        full = got[f"{prec} {p0} 8000"][1]
        each = -(-n // 152)
        assert block % 32 == 0 and grid <= n
        assert block >= full or each == 1  # (one profile an SM above 16384 bins takes the lone CTA's shape)
        if each <= 6 and block > full:
            assert grid == n and each * block <= (768 if p0 <= 2048 else 1024)
        if p0 in (700, 1100, 2048, 3001, 9001) and each == 1:
            assert block > full


def test_running_median_threads(fake):
    """A CTA of the running median has at least the threads of its tile's
    outputs: shared memory bounds how many CTAs an SM holds, so a small CTA
    leaves the SM idle."""
    got = fakecuda.run(fake, """
out = []
for n in (1 << 14, 1 << 17, 1 << 22):
    for w in (129, 257, 1025, 4001, 62501):
        fake.fake_reset()
        assert lib.ffa_detrend(BUF, C.c_int64(n), C.c_int32(w), BUF, BUF, None) == 0
        (name, grid, block, smem), = launches()
        out.append([n, w, block])
emit(out)
""")
    for n, w, block in got:
        tile = 32
        while 2 * tile <= min(1024, (w + 1) // 4):
            tile *= 2
        assert block >= min(tile, 512)
        assert block in (256, 512) and (n > 1 << 14 or block == 512)


@pytest.mark.parametrize("n,lo,hi", [(1 << 20, 0.53, 0.7), (1 << 22, 0.512, 0.52)])
def test_autotune_times_the_search_s_groups(fake, n, lo, hi):
    """The launches that are timed are those of a search: base periods that it
    folds together are timed together."""
    got = fakecuda.run(fake, f"""
ts = 512e-6
h = plan(config(tsamp_s=ts, period_min_s={lo}, period_max_s={hi}, duty_max=0.2), {n})
ws, k = C.c_size_t(), C.c_int32()
lib.ffa_plan_info(h, None, None, None, None, C.byref(ws))
fake.fake_reset()
assert lib.ffa_search(h, BUF, BUF, ws, BUF, BUF, None) == 0
folds = [x[:2] for x in launches() if "k_fold" in x[0]]
assert lib.ffa_autotune(h, BUF, ws, None, C.byref(k)) == 0 and k.value == 1
emit([folds, [x[:2] for x in launches()]])
""")
    searched, timed = ({tuple(x) for x in v} for v in got)
    # (one of the search's groups is timed)
    for name in {name for name, _ in searched}:
        assert any(x in timed for x in searched if x[0] == name), name
