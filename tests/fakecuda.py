"""The library on a CUDA runtime that runs nothing (fake_cudart.c): `run`
executes a script in a process of its own, with these names at hand:
  lib        the library (ctypes), every call's result an int
  fake       the stand-in runtime
  BUF        an address that passes for device memory
  launches() the launches since the last call: (kernel, grid, block, smem)
  config(**) a search configuration; plan(cfg, n) a plan's handle
and returns what the script gives to emit() (JSON)."""
import ctypes
import json
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(ROOT, "paper_1703_05581_gb300", "libffa_gb300.so")


class Launch(ctypes.Structure):
    _fields_ = [("name", ctypes.c_char * 256), ("grid", ctypes.c_uint), ("block", ctypes.c_uint),
                ("smem", ctypes.c_uint64)]


class SearchConfig(ctypes.Structure):
    _fields_ = [("tsamp_s", ctypes.c_double), ("period_min_s", ctypes.c_double), ("period_max_s", ctypes.c_double),
                ("duty_max", ctypes.c_double)] + \
        [(k, ctypes.c_int32) for k in ("downsample0", "detrend_window", "min_rows", "in_type", "precision",
                                       "n_widths_fixed")] + [("widths_fixed", ctypes.c_int32 * 16)] + \
        [("scorer", ctypes.c_int32), ("alg2_window", ctypes.c_float), ("clip_sigma", ctypes.c_float),
         ("persist_cutoff", ctypes.c_float), ("persistence", ctypes.c_int32)]


def build(tmp) -> str:
    so = os.path.join(str(tmp), "libfakecudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "fake_cudart.c")], check=True)
    return so


def run(so: str, script: str, timeout: float = 120):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), so], input=script, capture_output=True, text=True,
                       timeout=timeout)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.splitlines()[-1])


def _main():
    c = ctypes
    fake = c.CDLL(sys.argv[1], mode=c.RTLD_GLOBAL)
    lib = c.CDLL(LIB)
    fake.fake_launch.restype = c.POINTER(Launch)
    fake.fake_busy_us.argtypes = [c.c_double]
    fake.fake_elapsed_ms.argtypes = [c.c_float]
    lib.ffa_last_error.restype = c.c_char_p

    def launches():
        out = [fake.fake_launch(i).contents for i in range(fake.fake_launches())]
        out = [(x.name.decode(), x.grid, x.block, x.smem) for x in out]
        fake.fake_reset()
        return out

    def config(**kw):
        cfg = SearchConfig(downsample0=1, duty_max=0.2)
        for k, v in kw.items():
            setattr(cfg, k, v)
        return cfg

    def plan(cfg, n):
        h = c.c_void_p()
        st = lib.ffa_plan_create(c.byref(cfg), c.c_int64(n), c.byref(h))
        assert st == 0, lib.ffa_last_error()
        return h

    env = dict(lib=lib, fake=fake, BUF=c.c_void_p(1 << 20), launches=launches, config=config, plan=plan, C=c,
               emit=lambda x: print(json.dumps(x)))
    exec(compile(sys.stdin.read(), "script", "exec"), env)


if __name__ == "__main__":
    _main()
