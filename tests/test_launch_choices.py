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
