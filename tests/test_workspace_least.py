"""A search runs in a workspace with planes for its largest base period (and
1024 rows of the shorter ones); the room that ffa_plan_info asks for on top of
that only makes the groups larger.  So an arena that holds the least is enough
for a server's request."""
import fakecuda
import pytest

PRELUDE = """
ts = 512e-6
cfg = config(tsamp_s=ts, period_min_s=0.5, period_max_s=2.0, duty_max=0.2)
n = 1 << 20
h = plan(cfg, n)
ws, ne, nt = C.c_size_t(), C.c_int64(), C.c_int64()
lib.ffa_plan_info(h, C.byref(ne), C.byref(nt), None, None, C.byref(ws))
ent = C.create_string_buffer(104 * ne.value)
lib.ffa_plan_entries(h, ent, ne)
import struct
slot = lambda e: (e[3] * ((e[1] + 3) // 4 * 4) + 63) // 64 * 64
es = [struct.unpack_from("5i", ent.raw, 104 * i) for i in range(ne.value)]
al = lambda x: (x + 255) // 256 * 256
least = max([slot(e) for e in es] + [min(1024 // e[3] * slot(e), 1 << 24) for e in es if e[3] < 1024])
most = max(least, min(64 * max(map(slot, es)), 1 << 24, sum(map(slot, es))))
least = ws.value - 2 * al(4 * most) + 2 * al(4 * least)
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fakecuda.build(tmp_path_factory.mktemp("fake"))


def test_search_in_the_least_workspace(fake):
    got = fakecuda.run(fake, PRELUDE + """
def search(b):
    fake.fake_reset()
    st = lib.ffa_search(h, BUF, BUF, C.c_size_t(b), BUF, BUF, None)
    return [st, sum("k_score1" in x[0] for x in launches())]
emit([search(b) for b in (ws.value, 2 * ws.value, (ws.value + least) // 2, least, least - 256, 1024)] + [ws.value, least])
""")
    full, double, half, low, short, none, ws, least = got
    assert least < ws // 3
    assert full[0] == double[0] == half[0] == low[0] == 0
    assert double[1] == full[1] < half[1] < low[1]  # fewer, larger launches with more room
    assert short == none == [3, 0]                  # FFA_ERR_OOM


def test_request_in_a_small_arena(fake):
    got = fakecuda.run(fake, PRELUDE + """
class Cfg(C.Structure):
    _fields_ = [("d_arena", C.c_void_p), ("arena_bytes", C.c_size_t), ("n_slots", C.c_int32), ("timeout_ms", C.c_int32)]
series = C.create_string_buffer(4 * n)
need = 256 + al(4 * n) + al(16 * nt.value) + al(least)
def request(arena):
    srv, tk, no, best = C.c_void_p(), C.c_int64(), C.c_int32(), C.c_int64()
    c = Cfg(1 << 20, arena, 1, 10000)
    assert lib.ffa_server_create(C.byref(c), C.byref(srv)) == 0
    st = lib.ffa_server_submit(srv, C.byref(cfg), series, C.c_int64(n), C.c_double(6.0), 4, None, C.byref(tk))
    if st == 0:
        out = C.create_string_buffer(4096)
        st = lib.ffa_server_wait(srv, tk, 10000, out, 4, C.byref(no), C.byref(best), None)
    used = C.c_size_t()
    lib.ffa_server_stats(srv, None, None, C.byref(used))
    lib.ffa_server_destroy(srv)
    return [st, used.value]
emit([request(a) for a in (need, need + (1 << 20), 4 * need + 4 * ws.value, need - 256)])
""")
    assert got == [[0, 0], [0, 0], [0, 0], [3, 0]]
