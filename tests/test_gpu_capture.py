"""Sweeps and energies captured into a CUDA graph after a plain call has warmed
the buffers: a call that would copy host tables or hold a buffer that may move
takes the route without, and the replayed graph gives the plain call's results
also after larger calls have made the buffers grow."""
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


def _start(smc, dims, S, seed):
    lat = smc.Lattice(*dims, S)
    g = torch.Generator(device="cuda").manual_seed(seed)
    return lat, torch.randint(0, S, (lat.nsites,), dtype=torch.int8, device="cuda", generator=g)


def _captured(fn):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fn()
    return g


@pytest.mark.parametrize("S", [2, 3])
def test_mlp_sweep(smc, S):
    lat, occ = _start(smc, (16, 12, 20), S, 3)
    model = smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3))
    plain, again = occ.clone(), occ.clone()
    smc.sweep(lat, model, plain, 5, 0, 2, [0.07, 0.06])
    g = _captured(lambda: smc.sweep(lat, model, again, 5, 0, 2, [0.07, 0.06]))
    assert torch.equal(again, occ)
    g.replay()
    torch.cuda.synchronize()
    smc.check()
    assert torch.equal(again, plain)


@pytest.mark.parametrize("dims", [(64, 32, 32), (40, 32, 32)])
def test_energy(smc, dims):
    lat, occ = _start(smc, dims, 5, 4)
    model = smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(7, 2, 5))
    e, plain = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    smc.energy(lat, model, occ, plain)
    g = _captured(lambda: smc.energy(lat, model, occ, e))
    big, bocc = _start(smc, (68, 60, 64), 5, 5)  # other rows: their planes have a buffer of their own
    for _ in range(2):
        smc.energy(big, model, bocc, torch.zeros(1, dtype=torch.float64, device="cuda"))
    g.replay()
    torch.cuda.synchronize()
    smc.check()
    assert e.item() == plain.item()


@pytest.mark.parametrize("warm", [False, True])
def test_pair_sweep_of_many_short_rows(smc, warm):
    """A lattice that only wide resident blocks hold: captured without a plan it streams, with one it stays resident."""
    lat, occ = _start(smc, (16, 144, 140), 5, 6)
    model = smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(9, 2, 5))
    kT = [0.08, 0.07]
    plain, again = occ.clone(), occ.clone()
    smc.sweep(lat, model, plain, 5, 0, 2, kT)
    if not warm:  # another lattice's plan takes the place of this one's
        other, oocc = _start(smc, (64, 64, 64), 5, 7)
        smc.sweep(other, model, oocc, 5, 0, 1, 0.07)
    g = _captured(lambda: smc.sweep(lat, model, again, 5, 0, 2, kT))
    g.replay()
    torch.cuda.synchronize()
    smc.check()
    assert torch.equal(again, plain)
