"""The sweeps that run four mini-steps per launch on rows in shared memory (FCC
pair models, qSRO on both lattices) at the row lengths and alignments where
their copies change: rows of one 16-byte copy, of 4-byte copies, the longest
row they take (1024 cells) and the first they leave to the one-mini-step
kernels, and occupancies at 16-, 4- and 1-byte alignment."""
import numpy as np
import pytest

import oracle
from paper_2604_08250_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DE_TOL_EV = 1e-5  # FP32 dE against FP64: the bound of the floating-point paths


@pytest.fixture(scope="module")
def smc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build, smc as s
    build.build()
    s.lib()
    return s


def _device(ref, offset):
    """ref on the device, `offset` bytes past a 256-byte boundary."""
    buf = torch.empty(ref.size + 256, dtype=torch.int8, device="cuda:0")
    buf[offset:offset + ref.size] = torch.from_numpy(ref.copy()).to("cuda:0")
    return buf[offset:offset + ref.size]


@pytest.mark.parametrize("dims,nsh", [((8, 8, 8), 2), ((12, 8, 16), 3), ((16, 8, 8), 1), ((20, 12, 8), 2),
                                      ((32, 8, 8), 3), ((144, 8, 8), 2), ((1024, 8, 8), 2), ((1028, 8, 8), 1)])
@pytest.mark.parametrize("offset", [0, 4, 1])
def test_fcc_integer_sweep_is_the_oracle_bit_for_bit(smc, dims, nsh, offset):
    S = 4
    V = inputs.pair_int_coeffs(3 + nsh, nsh, S)
    lat, olat = smc.Lattice(*dims, S), oracle.Lattice(*dims, S)
    ref = oracle.fcc_init_lattice(olat, inputs.equiatomic_counts(smc.fcc_nsites(lat), S), 5)
    occ = _device(ref, offset)
    n = torch.zeros(1, dtype=torch.int64, device="cuda:0")
    smc.fcc_sweep(lat, smc.Model(smc.PAIR_I32, nsh, V, unit_ev=1e-4), occ, 9, 2, 1, 0.04, n_acc=n)
    smc.check()
    _, on = oracle.fcc_sweep(olat, oracle.Model(oracle.PAIR_I32, nsh, V, unit_ev=1e-4), ref, 9, 2, 1, [0.04])
    assert int(n) == on
    assert np.array_equal(occ.cpu().numpy(), ref)


@pytest.mark.parametrize("lattice", ["bcc", "fcc"])
@pytest.mark.parametrize("dims,nsh,S", [((8, 8, 8), 3, 5), ((16, 8, 8), 2, 8), ((36, 8, 12), 3, 4), ((48, 8, 8), 1, 5),
                                        ((1024, 8, 8), 2, 5), ((1028, 8, 8), 3, 3)])
def test_qsro_ministeps_against_the_oracle(smc, lattice, dims, nsh, S):
    V, W, C = inputs.qsro_coeffs(7, nsh, S)
    lat, olat = smc.Lattice(*dims, S), oracle.Lattice(*dims, S)
    model = smc.Model(smc.QSRO_F32, nsh, V, qsro_w=W, qsro_c=C)
    omodel = oracle.Model(oracle.QSRO, nsh, V, qsro_w=W, qsro_c=C)
    fcc = lattice == "fcc"
    N = smc.fcc_nsites(lat) if fcc else lat.nsites
    nA = 256 if fcc else 128
    init = oracle.fcc_init_lattice if fcc else oracle.init_lattice
    step = oracle.fcc_ministep_trace if fcc else oracle.ministep_trace
    gstep = smc.fcc_ministep_trace if fcc else smc.ministep_trace
    ref = init(olat, inputs.dirichlet_counts(N, S, 3), 4)
    dE = torch.zeros(N // nA, dtype=torch.float32, device="cuda:0")
    acc = torch.zeros(N // nA, dtype=torch.uint8, device="cuda:0")
    differ = 0
    for k in list(range(0, nA, 7)) + [nA - 1]:
        occ = _device(ref, 0)
        gstep(lat, model, occ, 11, 1, k, 0.06, dE=dE, acc=acc)
        smc.check()
        want, wacc, _, _ = step(olat, omodel, ref, 11, 1, k, 0.06)  # ref becomes the state after the mini-step
        assert np.abs(dE.cpu().numpy().astype(np.float64) - want).max() <= DE_TOL_EV
        bad = int((acc.cpu().numpy().astype(bool) != wacc).sum())
        differ += bad
        if bad == 0:
            assert np.array_equal(occ.cpu().numpy(), ref)
    # a decision differs only where exp(-dE / kT) crosses the random number within the 1e-5 eV above: 1.7e-4 of a
    # trial's acceptance range at 0.06 eV, so of about 1e4 trials at most a few
    assert differ <= 5


@pytest.mark.parametrize("lattice", ["bcc", "fcc"])
@pytest.mark.parametrize("dims,nsh", [((8, 8, 8), 2), ((20, 8, 12), 3), ((32, 16, 8), 3), ((64, 8, 8), 2)])
def test_qsro_sweep_does_not_depend_on_alignment_and_equals_its_ministeps(smc, lattice, dims, nsh):
    S = 5
    V, W, C = inputs.qsro_coeffs(5, nsh, S)
    lat = smc.Lattice(*dims, S)
    model = smc.Model(smc.QSRO_F32, nsh, V, qsro_w=W, qsro_c=C)
    fcc = lattice == "fcc"
    N = smc.fcc_nsites(lat) if fcc else lat.nsites
    sweep, step = (smc.fcc_sweep, smc.fcc_ministep_trace) if fcc else (smc.sweep, smc.ministep_trace)
    start = np.random.default_rng(2).integers(0, S, N).astype(np.int8)
    traced = _device(start, 0)
    for k in range(256 if fcc else 128):
        step(lat, model, traced, 3, 5, k, 0.07)
    for offset in (0, 4, 1):
        occ = _device(start, offset)
        sweep(lat, model, occ, 3, 5, 1, 0.07)
        smc.check()
        assert torch.equal(occ, traced), offset
