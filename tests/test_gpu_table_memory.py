"""What a tabulated MLP sweep keeps: the table (4 bytes per feature vector) in
a buffer of its own, which is given back when another allocation of the library
finds no room.  In a process of its own, where no other call holds memory."""
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = """
import torch
from paper_2604_08250_gb300 import inputs, smc
lat = smc.Lattice(128, 128, 128, 5)
occ = torch.empty(lat.nsites, dtype=torch.int8, device="cuda")
smc.init_lattice(lat, inputs.dirichlet_counts(lat.nsites, 5, 3), 3, occ)
model = smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3))
ref, got = occ.clone(), occ.clone()
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
for t in range(12):
    smc.sweep(lat, model, ref, 1, t, 1, 0.07)
f0 = free()
smc.sweep(lat, model, got, 1, 0, 12, 0.07)
kept = f0 - free()
table = 5 * 495 * 210 * 1820 * 4
assert torch.equal(got, ref)
assert table <= kept <= table + (64 << 20), kept
big = smc.Lattice(256, 128, 128, 5)
bocc = torch.zeros(big.nsites, dtype=torch.int8, device="cuda")
f1 = free()
smc.debug_set(smc.DBG_ALLOC_ERROR, 2)  # cudaErrorMemoryAllocation, once
smc.sweep(big, model, bocc, 1, 0, 1, 0.07)  # a larger workspace
assert free() - f1 >= table - (1 << 30)
got = occ.clone()
smc.sweep(lat, model, got, 1, 0, 12, 0.07)
smc.check()
assert torch.equal(got, ref)
print("ok")
"""


WORKSPACE = """
import torch
from paper_2604_08250_gb300 import inputs, smc
lat = smc.Lattice(256, 128, 128, 5)
occ = torch.zeros(lat.nsites, dtype=torch.int8, device="cuda")
model = smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3))
smc.debug_set(smc.DBG_MLP_TABLE, 1)
smc.energy(lat, model, occ, torch.zeros(1, dtype=torch.float64, device="cuda"))  # the kernels are loaded
small = smc.Lattice(16, 16, 16, 5)
smc.sweep(small, model, occ[:small.nsites], 1, 0, 1, 0.07)
torch.cuda.synchronize()
f0 = torch.cuda.mem_get_info()[0]
smc.sweep(lat, model, occ, 1, 0, 1, 0.07)
torch.cuda.synchronize()
kept, need = f0 - torch.cuda.mem_get_info()[0], 20 * lat.nsites
assert need <= kept + (4 << 20) and kept <= need + (8 << 20), (kept, need)
print("ok")
"""


def test_large_workspaces_grow_to_what_is_needed():
    """20 bytes per site of an MLP sweep's caches and little more, not the next power of two."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", WORKSPACE], cwd=build.ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


def test_memory_that_a_tabulated_sweep_keeps():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CODE], cwd=build.ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr
