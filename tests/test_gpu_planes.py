"""Neighbour counts from species bit planes on rows that do not fill their last
32-cell word, one-word rows and aligned ones, on both lattices: pair counts,
integer energies and qSRO energies against counts made with torch.roll, the
own-species count cache through the sweeps that start from it."""
import itertools

import numpy as np
import pytest

from paper_2604_08250_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FCC_OFF = ((0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))


@pytest.fixture(scope="module")
def smc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build, smc as s
    build.build()
    s.lib()
    return s


def _vectors(fcc, m, sub):
    if fcc:
        out = []
        for v in itertools.product(range(-2, 3), repeat=3):
            if sum(x * x for x in v) == 2 * (m + 1) and sum(v) % 2 == 0:
                at = [o + x for o, x in zip(FCC_OFF[sub], v)]
                out.append((FCC_OFF.index(tuple(x % 2 for x in at)), tuple(x // 2 for x in at)))
        return out
    if m == 0:
        o = (0, 1) if sub else (-1, 0)
        return [(1 - sub, v) for v in itertools.product(o, repeat=3)]
    return [(sub, v) for v in itertools.product((-1, 0, 1), repeat=3) if sum(map(abs, v)) == m]


def _counts(occ, dims, S, nsh, fcc):
    """Ordered pair counts [nsh][S][S] and sums of squared own counts [nsh][S], int64."""
    nx, ny, nz = dims
    o = occ.reshape(-1, nz, ny, nx).long()
    cnt = torch.zeros((nsh, S, S), dtype=torch.int64, device=occ.device)
    sq = torch.zeros((nsh, S), dtype=torch.int64, device=occ.device)
    for m in range(nsh):
        for s in range(o.shape[0]):
            own = torch.zeros_like(o[s])
            for t, v in _vectors(fcc, m, s):
                nb = torch.roll(o[t], shifts=(-v[2], -v[1], -v[0]), dims=(0, 1, 2))
                cnt[m] += torch.bincount((o[s] * S + nb).reshape(-1), minlength=S * S).reshape(S, S)
                own += nb == o[s]
            for p in range(S):
                sq[m, p] += (own[o[s] == p] ** 2).sum()
    return cnt, sq


def _occ(n, S, seed, offset=0):
    buf = torch.empty(n + 64, dtype=torch.int8, device="cuda")
    buf[offset:offset + n] = torch.from_numpy(np.random.default_rng(seed).integers(0, S, n).astype(np.int8)).cuda()
    return buf[offset:offset + n]


@pytest.mark.parametrize("dims,offset", [((33, 40, 50), 0), ((200, 20, 20), 0), ((31, 47, 47), 3), ((2, 190, 190), 0),
                                         ((64, 32, 32), 1), ((96, 20, 20), 0)])
@pytest.mark.parametrize("S,nsh", [(1, 2), (2, 3), (5, 1), (8, 3)])
def test_bcc_pair_counts(smc, dims, offset, S, nsh):
    lat = smc.Lattice(*dims, S)
    occ = _occ(lat.nsites, S, 4, offset)
    got = torch.zeros((nsh, S, S), dtype=torch.int64, device="cuda")
    smc.sro(lat, nsh, occ, counts=got)
    smc.check()
    assert torch.equal(got, _counts(occ, dims, S, nsh, False)[0])


@pytest.mark.parametrize("dims", [(13, 36, 40), (32, 24, 24), (36, 20, 24), (64, 17, 19), (5, 64, 64)])
@pytest.mark.parametrize("S,nsh", [(2, 3), (5, 2), (8, 3), (3, 1)])
def test_fcc_energies(smc, dims, S, nsh):
    lat = smc.Lattice(*dims, S)
    N = smc.fcc_nsites(lat)
    occ = _occ(N, S, 5)
    cnt, sq = _counts(occ, dims, S, nsh, True)
    V = inputs.pair_int_coeffs(2, nsh, S)
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    e_int = torch.zeros(1, dtype=torch.int64, device="cuda")
    smc.fcc_energy(lat, smc.Model(smc.PAIR_I32, nsh, V, unit_ev=1e-4), occ, e, e_int)
    assert int(e_int) == int((torch.from_numpy(V.astype(np.int64)).cuda() * cnt).sum()) // 2
    Vq, W, C = inputs.qsro_coeffs(7, nsh, S)
    smc.fcc_energy(lat, smc.Model(smc.QSRO_F32, nsh, Vq, qsro_w=W, qsro_c=C), occ, e)
    smc.check()
    z = np.array([12.0, 6.0, 24.0])[:nsh]
    terms = [Vq.astype(np.float64) * cnt.cpu().numpy() / z[:, None, None],
             W.astype(np.float64) * sq.cpu().numpy() / z[:, None] ** 2]
    want = sum(t.sum() for t in terms) + N * C
    # FP64 sums of at most 217 terms
    assert abs(float(e) - want) <= 300 * 2.0 ** -53 * (sum(np.abs(t).sum() for t in terms) + N * abs(C))


@pytest.mark.parametrize("dims", [(33, 40, 50), (64, 32, 32)])
@pytest.mark.parametrize("S,nsh", [(5, 2), (8, 3), (2, 1)])
def test_bcc_qsro_energy(smc, dims, S, nsh):
    lat = smc.Lattice(*dims, S)
    occ = _occ(lat.nsites, S, 6)
    cnt, sq = _counts(occ, dims, S, nsh, False)
    Vq, W, C = inputs.qsro_coeffs(3, nsh, S)
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    smc.energy(lat, smc.Model(smc.QSRO_F32, nsh, Vq, qsro_w=W, qsro_c=C), occ, e)
    smc.check()
    z = np.array([8.0, 6.0, 12.0])[:nsh]
    terms = [Vq.astype(np.float64) * cnt.cpu().numpy() / z[:, None, None],
             W.astype(np.float64) * sq.cpu().numpy() / z[:, None] ** 2]
    want = sum(t.sum() for t in terms) + lat.nsites * C
    assert abs(float(e) - want) <= 300 * 2.0 ** -53 * (sum(np.abs(t).sum() for t in terms) + lat.nsites * abs(C))


@pytest.mark.parametrize("lattice", ["bcc", "fcc"])
@pytest.mark.parametrize("dims,nsh", [((36, 40, 24), 3), ((64, 20, 32), 2), ((20, 60, 32), 1)])
def test_count_cache(smc, lattice, dims, nsh):
    """The energy a sweep accumulates from its count cache is the change of the
    total energy (FP32 trial differences summed in FP64)."""
    S, fcc = 5, lattice == "fcc"
    lat = smc.Lattice(*dims, S)
    occ = _occ(smc.fcc_nsites(lat) if fcc else lat.nsites, S, 7)
    Vq, W, C = inputs.qsro_coeffs(4, nsh, S)
    model = smc.Model(smc.QSRO_F32, nsh, Vq, qsro_w=W, qsro_c=C)
    energy, sweep = (smc.fcc_energy, smc.fcc_sweep) if fcc else (smc.energy, smc.sweep)
    e0, e1, acc = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(3))
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    energy(lat, model, occ, e0)
    sweep(lat, model, occ, 3, 0, 1, 0.07, e_acc=acc, n_acc=n)
    energy(lat, model, occ, e1)
    smc.check()
    # each accepted dE is within 1e-5 eV; their errors are unrelated
    assert abs(float(e1 - e0) - float(acc)) <= 1e-5 * 10 * float(n) ** 0.5
