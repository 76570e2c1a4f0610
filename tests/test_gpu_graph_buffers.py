"""A graph stays valid when later plain calls need larger library buffers or
another lattice's plan: what a captured call was given is not freed.  (Where it
were, the replay would read and write freed memory.)"""
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


def _overwrite():
    """Memory that the library gave back would be handed out here, and filled."""
    torch.cuda.empty_cache()
    for _ in range(3):
        torch.full((1 << 26,), 0x5A, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()


@pytest.mark.parametrize("kind", ["mlp", "net"])
def test_longer_mlp_call_on_the_same_lattice(smc, kind):
    lat, occ = _start(smc, (64, 32, 16), 4, 3)
    model = smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3)) if kind == "mlp" else \
        smc.Model(smc.MLPNET_BF16, net=inputs.mlpnet_weights(3))
    plain, again, long = occ.clone(), occ.clone(), occ.clone()
    smc.sweep(lat, model, plain, 5, 0, 1, 0.07)
    g = _captured(lambda: smc.sweep(lat, model, again, 5, 0, 1, 0.07))
    smc.sweep(lat, model, long, 5, 0, 400, 0.07)
    torch.cuda.synchronize()
    _overwrite()
    g.replay()
    torch.cuda.synchronize()
    smc.check()
    assert torch.equal(again, plain)


# resident blocks of 8 and of 16 columns, one CTA, rows of 8 cells that stream
@pytest.mark.parametrize("dims", [(48, 48, 48), (16, 144, 140), (12, 8, 16), (64, 200, 200)])
@pytest.mark.parametrize("warm", [True, False])
def test_pair_sweep(smc, dims, warm):
    """Captured with the plan of a plain call or without one; then this lattice's plan (if any) and larger lattices'."""
    model = smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(9, 2, 5))
    lat, occ = _start(smc, dims, 5, 6)
    plain, again, last = occ.clone(), occ.clone(), occ.clone()
    other, oocc = _start(smc, (64, 64, 64), 5, 7)
    if warm:
        smc.sweep(lat, model, plain, 5, 0, 3, 0.08)
    else:
        smc.sweep(other, model, oocc, 5, 0, 1, 0.08)
    g = _captured(lambda: smc.sweep(lat, model, again, 5, 0, 3, 0.08))
    smc.sweep(lat, model, last, 5, 0, 3, 0.08)
    for big in ((64, 64, 64), (128, 128, 128)):
        blat, bocc = _start(smc, big, 5, 8)
        smc.sweep(blat, model, bocc, 5, 0, 2, 0.08)
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    smc.energy(blat, smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3)), bocc, e)
    torch.cuda.synchronize()
    _overwrite()
    g.replay()
    torch.cuda.synchronize()
    smc.check()
    assert torch.equal(again, last)
    assert not warm or torch.equal(plain, last)


def test_counts_of_a_larger_lattice(smc):
    lat, occ = _start(smc, (64, 32, 32), 5, 4)
    want, got = (torch.zeros(2, 5, 5, dtype=torch.int64, device="cuda") for _ in range(2))
    smc.sro(lat, 2, occ, counts=want)
    g = _captured(lambda: smc.sro(lat, 2, occ, counts=got))
    big, bocc = _start(smc, (256, 128, 128), 5, 5)
    smc.sro(big, 2, bocc, counts=torch.zeros(2, 5, 5, dtype=torch.int64, device="cuda"))
    torch.cuda.synchronize()
    _overwrite()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, want)
