"""The bounded wait's limit counts whole milliseconds: work that ends within
the millisecond after it is waited for (so a limit of 0 covers a short one)."""
import fakecuda
import pytest


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.build(tmp_path_factory.mktemp("fake"))


def test_limit_in_whole_milliseconds(fake):
    got = fakecuda.run(fake, """
def wait(busy_us, limit_ms):
    fake.fake_busy_us(busy_us)
    return lib.ffa_wait(None, None, C.c_int32(limit_ms))
# (the best of several: a loaded host may lose the processor in any one)
emit([min(wait(us, ms) for _ in range(20)) for us, ms in ((0, 0), (400, 0), (5400, 5), (3000, -1))] +
     [wait(us, ms) for us, ms in ((20000, 0), (60000, 20))])
""")
    assert got[:4] == [0, 0, 0, 0]   # FFA_OK
    assert got[4:] == [4, 4]         # FFA_ERR_TIMEOUT
