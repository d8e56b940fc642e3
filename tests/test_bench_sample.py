"""The benchmark's roofline figures book the launches that the library timed:
the base periods it takes for them are those that a search launches alone."""
import os
import sys

import fakecuda
import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

ENTRY = np.dtype([("octave", "<i4"), ("p0", "<i4"), ("m_data", "<i4"), ("m_rows", "<i4"), ("n_widths", "<i4"),
                  ("widths", "<i4", (16,)), ("pad", "<i4"), ("n_octave", "<i8"), ("first_trial", "<i8")])

CASES = {  # samples, interval, periods (s), duty, fixed widths
    "survey": (1 << 26, 64e-6, 1.0, 30.0, 0.1, ()),
    "short": (1 << 22, 64e-6, 1.0, 30.0, 0.1, ()),
    "trials": (1 << 20, 512e-6, 0.5, 20.0, 0.2, ()),
    "plain": (65536, 2.048e-3, 256 * 2.048e-3, 512 * 2.048e-3, 0.2, (1, 2, 4, 8, 16)),
}


@pytest.mark.parametrize("name", CASES)
def test_timed_launches(name, tmp_path):
    n, ts, lo, hi, duty, widths = CASES[name]
    path = tmp_path / "entries.bin"
    got = fakecuda.run(fakecuda.build(tmp_path), f"""
cfg = config(tsamp_s={ts}, period_min_s={lo}, period_max_s={hi}, duty_max={duty}, n_widths_fixed={len(widths)})
for i, w in enumerate({widths}):
    cfg.widths_fixed[i] = w
n = {n}
h = plan(cfg, n)
np_, ws = C.c_int64(), C.c_size_t()
lib.ffa_plan_info(h, C.byref(np_), None, None, None, C.byref(ws))
buf = C.create_string_buffer({ENTRY.itemsize} * np_.value)
lib.ffa_plan_entries(h, buf, C.c_int64(np_.value))
open({str(path)!r}, "wb").write(buf.raw)
lib.ffa_timing_enable(1)
fake.fake_reset()
assert lib.ffa_search(h, BUF, BUF, ws, BUF, BUF, None) == 0, lib.ffa_last_error()
scored = sum("k_score1" in x[0] for x in launches())
ms, cnt = (C.c_double * 384)(), (C.c_int32 * 384)()
assert lib.ffa_timing_read(ms, cnt, 384) == 0
emit([scored, list(cnt)[3 * 64:4 * 64]])
""")
    e = np.frombuffer(path.read_bytes(), ENTRY)
    assert got[0] == len(bench.group_starts(e))
    for o in range(int(e["octave"].max()) + 1):
        assert got[1][o] == len(bench.sampled_singles(e, o, 64)), o
