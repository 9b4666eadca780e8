"""The library's host code on the CPU, in a process of its own: the runtime is
fake_cudart.cpp, preloaded.  A driver script has fg, si, lib, fake, log() (the launches since
the last call of log) and problem(n, na, nb, mode)."""
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = r"""
import ctypes, math, sys
import numpy as np
import paper_2405_10197_gb300 as fg
import synth_inputs as si

fake = ctypes.CDLL(FAKE)
fake.fake_log.restype = ctypes.c_char_p
for f in (fake.fake_allocs, fake.fake_live):
    f.restype = ctypes.c_longlong
for f in (fake.fake_fail_at, fake.fake_fail_copy_at):
    f.argtypes = [ctypes.c_longlong]
lib = fg.library()

def log():
    out = fake.fake_log().decode().split("\n")[:-1]
    fake.fake_clear_log()
    return out

def problem(n, na, nb, mode):
    h, eri = si.integrals(n, 2 * n, seed=1)
    ctx = fg.forte_cas_create(n, na, nb, h, eri)
    fg.forte_set_precision(ctx, mode)
    log()
    return ctx
"""


def include_dir():
    from paper_2405_10197_gb300 import build
    return os.path.join(os.path.dirname(build._cuda_lib_dir(build._nvcc())), "include")


def compile_fake(folder):
    from paper_2405_10197_gb300 import build
    build.build()
    out = os.path.join(str(folder), "libfake_cudart.so")
    subprocess.run([shutil.which("g++"), "-shared", "-fPIC", "-std=c++17", "-I", include_dir(),
                    os.path.join(HERE, "fake_cudart.cpp"), "-o", out], check=True)
    return out


def run(fake, driver, *args):
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=os.pathsep.join([ROOT, HERE]))
    r = subprocess.run([sys.executable, "-c", f"FAKE = {fake!r}\n" + PRELUDE + driver + "\nprint('done')", *map(str, args)],
                       env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr[-2000:]
