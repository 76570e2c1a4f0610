"""The library's buffers and plans on the host side, with a CUDA runtime that
has two devices and no GPU (fake_cudart.c)."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2604_08250_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))

HEAD = """
import ctypes as C
from paper_2604_08250_gb300 import inputs, smc
fake, L = C.CDLL(None), smc.lib()
def counts():
    return [fake.fake_count(k) for k in range(3)]
def model(kind=smc.PAIR_F32, S=5):
    return smc.Model(kind, 2, inputs.pair_f32_coeffs(7, 2, S))
class Box:
    def __init__(self, *dims, S=5):
        self.lat = smc.Lattice(*dims, S)
        self.raw = C.create_string_buffer(self.lat.nsites + 16)
        self.occ = C.c_void_p((C.addressof(self.raw) + 15) // 16 * 16)
    def sro(self):
        assert L.smc_sro(C.byref(self.lat._c), 2, self.occ, None, None, None) == 0, L.smc_last_error()
    def sweep(self, m, n):
        kT = (C.c_double * n)(*[0.07] * n)
        assert L.smc_sweep(C.byref(self.lat._c), C.byref(m._c), self.occ, 1, 0, 0, n, kT, None, None, None) == 0, \\
            L.smc_last_error()
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not shutil.which("gcc"):
        pytest.skip("no C compiler")
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["gcc", "-O1", "-w", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "fake_cudart.c")], check=True)

    def go(code):
        r = subprocess.run([sys.executable, "-c", HEAD + code], cwd=build.ROOT, env={**os.environ, "LD_PRELOAD": so},
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout
    return go


@pytest.mark.parametrize("nx", [64, 100])  # rows whose planes are words, and others
def test_counts_on_two_devices_in_turn_allocate_once_each(run, nx):
    run(f"""
box = Box({nx}, 64, 64)
for d in (0, 1):
    fake.fake_set_device(d)
    box.sro()
before = counts()
for d in (0, 1) * 4:
    fake.fake_set_device(d)
    box.sro()
assert counts() == before, (before, counts())
""")


def test_lattices_in_turn_keep_their_plans(run):
    """Resident plans (one with columns for wide blocks only): made once for each of a few lattices."""
    run("""
m = model()
boxes = [Box(64, 64, 64), Box(64, 160, 160), Box(48, 48, 48)]
for b in boxes:
    b.sweep(m, 20)
before = counts()
for b in boxes * 3:
    b.sweep(m, 20)
assert counts() == before, (before, counts())
""")


def test_old_plans_are_given_back(run):
    run("""
m = model()
Box(96, 96, 96).sweep(m, 20)  # the largest: the workspace does not grow any more
start = counts()
for e in range(24, 64, 4):
    Box(e, e, e).sweep(m, 20)
made, freed, _ = [b - a for a, b in zip(start, counts())]
assert made == 10 and made - freed <= 3, (made, freed)
""")


def test_a_lattice_that_streams_makes_no_lists(run):
    run("""
import time
m = model()
Box(24, 24, 24).sweep(m, 20)
def first(dims, n):  # host time of the first call, the least of three lattices
    times = []
    for d in dims:
        box = Box(*d)
        t = time.process_time()
        box.sweep(m, n)
        times.append(time.process_time() - t)
    return min(times)
plan = first([(64, 160, 160), (60, 160, 160), (56, 160, 160)], 20)
# rows too long for wide blocks (by the lists, by the rows); one sweep of a lattice that streams faster
for dims, n in (([(160, 160, 160), (160, 160, 144), (160, 144, 160)], 20),
                ([(192, 160, 160), (200, 160, 160), (208, 160, 160)], 20),
                ([(128, 160, 152), (128, 152, 160), (128, 152, 152)], 1)):
    took = first(dims, n)
    assert took < 0.2 * plan, (dims, took, plan)
""")
