"""The start configuration's threshold selection at its edges, against the
oracle's sort: the smallest box, absent species (equal thresholds, thresholds
before the first and past the last site), species of one site, and a box whose
candidate lists lie in the occupancy itself (more than 13.6e6 sites with eight
species), unaligned too."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def smc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build, smc as s
    build.build()
    s.lib()
    return s


def _n(dims):
    return 2 * dims[0] * dims[1] * dims[2]


@pytest.mark.parametrize("dims,counts,offset", [
    ((2, 2, 2), [16], 0), ((2, 2, 2), [1, 15], 0), ((7, 5, 3), [0, 0, 100, 0, 110, 0, 0, 0], 1),
    ((8, 8, 8), [1, 1, 1020, 1, 1], 0), ((33, 21, 10), [0, 13860, 0], 3),
    ((200, 200, 180), [2000000, 0, 5000000, 1, 3399999, 1500000, 1500000, 1000000], 0),
    ((200, 200, 180), [14399999, 1], 1)])
def test_start_state_is_the_oracles(smc, dims, counts, offset):
    assert sum(counts) == _n(dims)
    buf = torch.empty(_n(dims) + 64, dtype=torch.int8, device="cuda")
    occ = buf[offset:offset + _n(dims)]
    smc.init_lattice(smc.Lattice(*dims, len(counts)), counts, 77, occ, replica=5)
    smc.check()
    want = oracle.init_lattice(oracle.Lattice(*dims, len(counts)), np.array(counts, dtype=np.int64), 77, replica=5)
    assert np.array_equal(occ.cpu().numpy(), want)
