"""Pair sweeps of small boxes by one CTA (the whole lattice in its shared
memory): integer trajectories bit for bit against the oracle, floating-point
ones against the streaming kernels, from the smallest box it takes (4 cells
per axis, every axis one link cell) through one, two and more trials per
mini-step to the largest, alone and as replicas of one call."""
import numpy as np
import pytest

import oracle
from paper_2604_08250_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOXES = [(4, 4, 4), (5, 6, 7), (9, 8, 12), (8, 8, 8), (4, 16, 9), (12, 12, 12), (16, 8, 20), (64, 16, 8), (20, 5, 4)]


@pytest.fixture(scope="module")
def smc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build, smc as s
    build.build()
    s.lib()
    return s


def _start(dims, S, seed):
    N = 2 * dims[0] * dims[1] * dims[2]
    return oracle.init_lattice(oracle.Lattice(*dims, S), inputs.dirichlet_counts(N, S, seed), seed)


@pytest.mark.parametrize("dims", BOXES)
@pytest.mark.parametrize("S,nsh", [(2, 1), (5, 2), (8, 3)])
def test_integer_trajectory_is_the_oracle(smc, dims, S, nsh):
    V = inputs.pair_int_coeffs(S + nsh, nsh, S)
    ref = _start(dims, S, 3)
    occ = torch.from_numpy(ref.copy()).to("cuda:0")
    kT = [0.03, 0.06, 0.02]
    e = torch.zeros(1, dtype=torch.float64, device="cuda:0")
    n = torch.zeros(1, dtype=torch.int64, device="cuda:0")
    smc.sweep(smc.Lattice(*dims, S), smc.Model(smc.PAIR_I32, nsh, V, unit_ev=1e-4), occ, 5, 7, 3, kT, e_acc=e, n_acc=n)
    smc.check()
    oe, on = oracle.sweep(oracle.Lattice(*dims, S), oracle.Model(oracle.PAIR_I32, nsh, V, unit_ev=1e-4), ref, 5, 7, 3, kT)
    assert np.array_equal(occ.cpu().numpy(), ref)
    assert int(n) == on and float(e) == oe


@pytest.mark.parametrize("dims", BOXES)
@pytest.mark.parametrize("S,nsh,kT", [(3, 2, [0.05, 0.02]), (5, 3, 0.07), (8, 2, float("inf")), (6, 1, 1e-4)])
def test_floating_point_sweep_equals_the_streaming_kernels(smc, dims, S, nsh, kT):
    model = smc.Model(smc.PAIR_F32, nsh, inputs.pair_f32_coeffs(4, nsh, S))
    start = torch.from_numpy(_start(dims, S, 2)).to("cuda:0")
    got = []
    for streaming in (0, 1):
        occ = start.clone()
        e = torch.zeros(1, dtype=torch.float64, device="cuda:0")
        n = torch.zeros(1, dtype=torch.int64, device="cuda:0")
        smc.debug_set(smc.DBG_RESIDENT, streaming)
        try:
            smc.sweep(smc.Lattice(*dims, S), model, occ, 11, 2 ** 33, 2, kT, e_acc=e, n_acc=n, replica=3)
            smc.check()
        finally:
            smc.debug_set(smc.DBG_RESIDENT, 0)
        got.append((occ, float(e), int(n)))
    assert torch.equal(got[0][0], got[1][0])
    assert got[0][2] == got[1][2]
    # both add exact integer dE and scale once
    assert abs(got[0][1] - got[1][1]) <= 1e-12 * max(1.0, abs(got[1][1]))


@pytest.mark.parametrize("edges", [[8] * 16, [8, 12, 16, 20] * 5, [4, 5, 6]])
def test_replicas_equal_single_calls(smc, edges):
    S, R = 4, len(edges)
    if len({e if e < 8 or e % 4 else 4 for e in edges}) > 1:
        pytest.skip("replicas of one call share their link-cell edge")
    model = smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(9, 2, S))
    lats = [smc.Lattice(e, e, e, S) for e in edges]
    occs = [torch.from_numpy(_start((e, e, e), S, r)).to("cuda:0") for r, e in enumerate(edges)]
    single = [o.clone() for o in occs]
    kT = np.repeat(inputs.ladder_kT(R)[:, None], 3, axis=1)
    n = torch.zeros(R, dtype=torch.int64, device="cuda:0")
    smc.sweep_batched(lats, model, occs, 1, 0, 3, kT, replica0=4, n_acc=n)
    for r in range(R):
        n1 = torch.zeros(1, dtype=torch.int64, device="cuda:0")
        smc.sweep(lats[r], model, single[r], 1, 0, 3, kT[r], replica=4 + r, n_acc=n1)
        smc.check()
        assert torch.equal(occs[r], single[r])
        assert int(n1) == int(n[r])


def test_species_outside_the_range_are_reported(smc):
    S = 3
    occ = torch.zeros(1024, dtype=torch.int8, device="cuda:0")
    occ[100] = S
    smc.sweep(smc.Lattice(8, 8, 8, S), smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(1, 2, S)), occ, 1, 0, 1, 0.05)
    with pytest.raises(smc.SMCError) as err:
        smc.check()
    assert err.value.code == smc.SMC_ERR_ARG
