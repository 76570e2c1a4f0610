"""Resident pair sweeps on boxes of other rows and blocks than the headline's,
bit for bit against the streaming kernels."""
import numpy as np
import pytest

from paper_2604_08250_gb300 import inputs

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


def _sweep(smc, lats, model, streaming, nsweeps=3):
    """Occupancies, accepted counts and energies of a call (batched when there are several lattices)."""
    occs = []
    for r, lat in enumerate(lats):
        o = torch.empty(lat.nsites, dtype=torch.int8, device="cuda")
        smc.init_lattice(lat, inputs.equiatomic_counts(lat.nsites, lat.nspecies), 7, o, replica=r)
        occs.append(o)
    e = torch.zeros(len(lats), dtype=torch.float64, device="cuda")
    n = torch.zeros(len(lats), dtype=torch.int64, device="cuda")
    kT = np.repeat(np.linspace(0.12, 0.05, nsweeps)[None, :], len(lats), axis=0)
    smc.debug_set(smc.DBG_RESIDENT, 1 if streaming else 0)
    try:
        if len(lats) == 1:
            smc.sweep(lats[0], model, occs[0], 7, 0, nsweeps, kT[0], e_acc=e, n_acc=n)
        else:
            smc.sweep_batched(lats, model, occs, 7, 0, nsweeps, kT, e_acc=e, n_acc=n)
        smc.check()
    finally:
        smc.debug_set(smc.DBG_RESIDENT, 0)
    return occs, e.tolist(), n.tolist()


def _model(smc, kind, nsh, S):
    if kind == "int":
        return smc.Model(smc.PAIR_I32, nsh, inputs.pair_int_coeffs(3, nsh, S), unit_ev=1e-4)
    return smc.Model(smc.PAIR_F32, nsh, inputs.pair_f32_coeffs(5, nsh, S))


def _same(smc, dims, kind, S, nsh):
    lats = [smc.Lattice(*d, S) for d in dims]
    model = _model(smc, kind, nsh, S)
    a, b = _sweep(smc, lats, model, False), _sweep(smc, lats, model, True)
    assert all(torch.equal(x, y) for x, y in zip(a[0], b[0]))
    assert a[1:] == b[1:]


def test_rows_of_half_chunks_at_the_short_pitch(smc):
    """228 cells: windows too large for a pitch of 128-byte multiples, rows no multiple of 8 bytes."""
    _same(smc, [(228, 128, 136)], "f32", 5, 2)


@pytest.mark.parametrize("dims,kind,S,nsh", [((12, 144, 140), "f32", 5, 2), ((64, 144, 140), "f32", 8, 3),
                                             ((96, 140, 144), "int", 4, 2), ((100, 144, 140), "f32", 5, 2),
                                             ((140, 140, 144), "f32", 3, 1), ((36, 196, 196), "int", 8, 2),
                                             ((128, 144, 140), "f32", 5, 2), ((160, 144, 140), "f32", 5, 2)])
def test_wide_blocks(smc, dims, kind, S, nsh):
    """More columns than 152 blocks of eight hold: blocks of up to sixteen (the last box fits in neither)."""
    _same(smc, [dims], kind, S, nsh)


@pytest.mark.parametrize("edges,kind,nsh", [([64] * 12, "f32", 2), ([96, 84, 64, 52, 36, 32] * 4, "int", 2),
                                            ([80] * 9 + [40], "f32", 3), ([96] * 6 + [100], "f32", 2)])
def test_wide_blocks_of_replicas(smc, edges, kind, nsh):
    """Replicas that take fewer launches in wide blocks, with odd lattices among them; and, last, a row too long."""
    _same(smc, [(e, e, e) for e in edges], kind, 5, nsh)
