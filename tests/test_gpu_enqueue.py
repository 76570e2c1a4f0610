"""Sweeps enqueue their work and return: with work ahead on the stream, the call
comes back before that work is done (after a first call has made its buffers)."""
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


def _model(smc, kind):
    if kind == "mlp":
        return smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3))
    if kind == "net":
        return smc.Model(smc.MLPNET_BF16, net=inputs.mlpnet_weights(3))
    if kind == "pair+mlp":
        return smc.Model(smc.PAIR_F32_MLP_BF16, 2, inputs.pair_f32_coeffs(5, 2, 5), mlp=inputs.mlp_weights(3))
    return smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(5, 2, 5))


@pytest.mark.parametrize("kind,edge,n", [("mlp", 96, 1), ("mlp", 96, 24), ("pair+mlp", 96, 24), ("net", 96, 24),
                                         ("pair", 8, 3), ("pair", 64, 3), ("pair", 160, 3)])
def test_call_returns_before_the_work_ahead_is_done(smc, kind, edge, n):
    lat = smc.Lattice(edge, edge, edge, 5)
    g = torch.Generator(device="cuda").manual_seed(1)
    occ = torch.randint(0, 5, (lat.nsites,), dtype=torch.int8, device="cuda", generator=g)
    ref, model = occ.clone(), _model(smc, kind)
    smc.sweep(lat, model, ref, 1, 0, n, 0.07)
    torch.cuda.synchronize()
    torch.cuda._sleep(1 << 30)  # half a second and more
    ahead = torch.cuda.Event()
    ahead.record()
    smc.sweep(lat, model, occ, 1, 0, n, 0.07)
    assert not ahead.query()
    smc.check()
    assert torch.equal(occ, ref)
