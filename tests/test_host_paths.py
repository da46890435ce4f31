"""Host code of the library without a device: a stand-in for the CUDA runtime
counts launches and allocations and fails one on request."""
import ctypes as C
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GCC = shutil.which("gcc")

PRELUDE = """
import ctypes as C, sys
import numpy as np
from paper_2602_07452_gb300 import fpic as F, inputs as I
fake = C.CDLL(None)
fake.fake_bytes.restype = fake.fake_launches.restype = C.c_longlong
fake.fake_fail_alloc_of.argtypes = [C.c_size_t]
L = F.lib()

def at(k, T=C.c_double):          # the address of an array the library only passes on
    return C.cast(C.c_void_p(4096 * k), C.POINTER(T))

def ctx_of(N, a=0.9):
    g = I.wald_grid(N, a)
    c = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(c, g)
    return c, g

def particles(n):
    s = F.fpic_particles()
    s.n = n
    for k, (name, T) in enumerate(F.fpic_particles._fields_[1:]):
        setattr(s, name, at(k + 1, T._type_))
    return s

def watch(name):
    fake.fake_watch(name.encode())
"""


def _run(tmp_path, body):
    so = str(tmp_path / "fake.so")
    subprocess.run([GCC, "-shared", "-fPIC", "-O1", "-w", "-o", so, os.path.join(ROOT, "tests", "native", "fake_cudart.c")],
                   check=True)
    env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", PRELUDE + body], env=env, cwd=ROOT, capture_output=True, text=True)
    assert out.returncode == 0, out.stderr[-2000:]
    return out.stdout.split()


needs = pytest.mark.skipif(GCC is None or not os.path.exists(
    os.path.join(ROOT, "paper_2602_07452_gb300", "_build", "libfpic.so")), reason="needs gcc and the built library")


@needs
def test_coefficients_dropped_by_a_failed_batch_are_built_by_the_next_push(tmp_path):
    """A batch whose second run's allocation fails builds nothing for the first:
    with static fields on, the next push of that run builds its coefficients,
    the one after it does not."""
    out = _run(tmp_path, """
c1, g1 = ctx_of(32)
c2, g2 = ctx_of(48)
F.fpic_set_tuning(c1, F.FPIC_TUNE_STATIC_FIELDS, 1)
f1, f2 = [at(40 + k) for k in range(6)], [at(50 + k) for k in range(6)]
runs = (F.fpic_run * 2)()
for k, (c, f) in enumerate(((c1, f1), (c2, f2))):
    runs[k].ctx = c.handle
    for i in range(6): runs[k].fields[i] = f[i]
    runs[k].begin, runs[k].end, runs[k].r_max, runs[k].B0pot = 100 * k, 100 * k + 100, 50.0, 0.0
p, prm = particles(200), F.push_params(1e-3, scheme=F.FPIC_RK4)
watch("k_field_coef")
fake.fake_fail_alloc_of(6 * 4 * 8 * g2.size)
rc = L.fpic_push_batched(runs, 2, C.byref(p), C.byref(prm), None, None)
print(int(rc != 0), fake.fake_launches())
p = particles(100)
arr = (C.POINTER(C.c_double) * 6)(*f1)
for _ in range(2):
    rc = L.fpic_push(c1.handle, C.byref(p), arr, C.byref(prm), None, None)
    print(rc, fake.fake_launches())
""")
    assert out == ["1", "0", "0", "1", "0", "1"], out


@needs
def test_conserving_deposit_scratch_is_bounded(tmp_path):
    """3e8 particles: 28 bytes each for the sort, and records of 6.7e7 of them at
    a time (240 bytes), in as many turns as that takes; a quarter as many at a
    time when those do not fit, also for the next call, which allocates nothing."""
    out = _run(tmp_path, """
n = 300_000_000
size = lambda chunk: sum((b + 255) & ~255 for b in (4*n, 4*n, 4*n, 4*(2*C_+2), 4*(2*C_+2), 4*(2*C_+2), 4*(n//4096 + 2), 4*n,
                                                   4*(n+1), 8*n, 240*(C_ + chunk)))
c, g = ctx_of(256)
C_ = g.Nr * g.Nth
p = particles(n)
out = [at(80 + k) for k in range(4)]
watch("k_cdep_particle")
before = fake.fake_bytes()
rc = L.fpic_deposit_conserving(c.handle, C.byref(p), C.byref(p), 1e-3, *out, None, None)
print(rc, fake.fake_launches(), int(fake.fake_bytes() - before < 1.13 * (28 * n + 240 * 67_000_000) + 5e7))
del c
c, g = ctx_of(256)
asked = size(67_000_000)
fake.fake_fail_alloc_of(asked + asked // 8)
watch("k_cdep_particle")
rc = L.fpic_deposit_conserving(c.handle, C.byref(p), C.byref(p), 1e-3, *out, None, None)
print(rc, fake.fake_launches())
before = fake.fake_bytes()
rc = L.fpic_deposit_conserving(c.handle, C.byref(p), C.byref(p), 1e-3, *out, None, None)
print(rc, fake.fake_launches(), fake.fake_bytes() - before)
""")
    assert out == ["0", "5", "1", "0", "18", "0", "36", "0"], out
