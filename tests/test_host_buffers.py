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
