"""What a failed device allocation does: a lack of memory takes the route that
needs none, for this call only; any other error is the call's.  The errors are
injected (SMC_DBG_ALLOC_ERROR), in a process that holds no other buffer of the
library."""
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HEAD = """
import torch
from paper_2604_08250_gb300 import inputs, smc
OOM, OTHER = 2, 46  # cudaErrorMemoryAllocation, cudaErrorDevicesUnavailable
def start(dims, S=5):
    lat = smc.Lattice(*dims, S)
    g = torch.Generator(device="cuda").manual_seed(1)
    return lat, torch.randint(0, S, (lat.nsites,), dtype=torch.int8, device="cuda", generator=g)
def fails(fn):
    try:
        fn()
    except smc.SMCError as err:
        assert err.code == smc.SMC_ERR_CUDA, err
        return True
    return False
smc.philox4x32_10(*[torch.zeros(4, dtype=torch.int32, device="cuda") for _ in range(3)])
smc.check()  # the workspace
pair = smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(5, 2, 5))
"""

RESIDENT = HEAD + """
# 36 x 37 columns of link cells: resident in blocks of up to 16 columns only
lat, occ = start((20, 144, 148))
def sweep(o):
    smc.sweep(lat, pair, o, 1, 0, 40, 0.07)
    smc.check()
want = occ.clone()
smc.debug_set(smc.DBG_RESIDENT, 1)
sweep(want)
# a tile that never publishes ends a streaming sweep in a timeout; the resident sweep has no block of that number
smc.debug_set(smc.DBG_TIMEOUT_MS, 100)
smc.debug_set(smc.DBG_SKIP_PUBLISH, 200)
try:
    sweep(occ.clone())
    raise SystemExit("the streaming sweep has no tile 200")
except smc.SMCError as err:
    assert err.code == smc.SMC_ERR_TIMEOUT, err
smc.debug_set(smc.DBG_RESIDENT, 0)
smc.debug_set(smc.DBG_SKIP_PUBLISH, -1)
smc.debug_set(smc.DBG_ALLOC_ERROR, OTHER)
assert fails(lambda: sweep(occ.clone()))
smc.debug_set(smc.DBG_ALLOC_ERROR, OOM)
got = occ.clone()
sweep(got)
assert torch.equal(got, want)
smc.debug_set(smc.DBG_SKIP_PUBLISH, 200)
got = occ.clone()
sweep(got)  # resident again
assert torch.equal(got, want)
print("ok")
"""

MLP = HEAD + """
lat, occ = start((64, 64, 64), 4)
mlp = smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3))
def sweep(o):
    smc.sweep(lat, mlp, o, 1, 0, 20, 0.07)
    smc.check()
want = occ.clone()
smc.debug_set(smc.DBG_MLP_TABLE, 1)
sweep(want)
smc.debug_set(smc.DBG_MLP_TABLE, 2)
smc.debug_set(smc.DBG_ALLOC_ERROR, OTHER)
assert fails(lambda: sweep(occ.clone()))
for error in (OOM, 0):
    smc.debug_set(smc.DBG_ALLOC_ERROR, error)
    got = occ.clone()
    sweep(got)
    assert torch.equal(got, want)
print("ok")
"""

PLANES = HEAD + """
for dims in ((64, 64, 64), (100, 64, 64)):  # aligned rows and others
    lat, occ = start(dims)
    counts = [torch.zeros(2, 5, 5, dtype=torch.int64, device="cuda") for _ in range(3)]
    smc.debug_set(smc.DBG_ALLOC_ERROR, OTHER)
    assert fails(lambda: smc.sro(lat, 2, occ, counts=counts[0]))
    for error, c in zip((OOM, 0), counts):
        smc.debug_set(smc.DBG_ALLOC_ERROR, error)
        smc.sro(lat, 2, occ, counts=c)
    smc.check()
    assert counts[0].sum() > 0 and torch.equal(counts[0], counts[1])
print("ok")
"""


@pytest.mark.parametrize("code", [RESIDENT, MLP, PLANES], ids=["resident", "mlp", "planes"])
def test_failed_allocation(code):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", code], cwd=build.ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr
