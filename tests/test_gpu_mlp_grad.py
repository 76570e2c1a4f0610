"""MLP gradient where its tiles and flushes can go wrong: less than a tile for
every warpgroup, exactly three tiles, a ragged last tile in a second round, two
flush epochs with warpgroups that have different numbers of tiles; against FP64
back-propagation."""
import numpy as np
import pytest

from paper_2604_08250_gb300 import inputs
from tests import helpers

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# Each term carries two BF16 roundings (activation and derivative, 2^-8 of it each at most) and, far below
# those, FP32 sums and the hardware tanh: within 2^-7 + 2^-9 of the sum of the magnitudes of its factors.
REL = 2.0 ** -7 + 2.0 ** -9


@pytest.fixture(scope="module")
def smc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_08250_gb300 import build, smc as s
    build.build()
    s.lib()
    return s


def _reference(X, w):
    def silu(z):
        s = 1.0 / (1.0 + np.exp(-z))
        return z * s, s * (1.0 + z * (1.0 - s))

    h1, g1 = silu(X @ w["w1"].T + w["b1"])
    h2, g2 = silu(h1 @ w["w2"].T + w["b2"])
    d2 = w["w3"] * g2
    d1 = (d2 @ w["w2"]) * g1
    return np.concatenate([(d1.T @ X).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.sum(0),
                           [float(X.shape[0])]])


@pytest.mark.parametrize("dims,S", [((3, 5, 7), 4), ((8, 6, 4), 5), ((33, 31, 35), 5), ((64, 60, 62), 3)])
def test_gradient_at_tile_edges(smc, dims, S):
    bits = inputs.mlp_weights(11)
    rng = np.random.default_rng(5)
    bits["b1"], bits["b2"] = (rng.uniform(-0.3, 0.3, 64).astype(np.float32) for _ in range(2))
    w = {k: inputs.bf16_bits_to_f32(bits[k]).astype(np.float64) for k in ("w1", "w2", "w3")}
    w["w1"], w["w2"], w["w3"] = w["w1"].reshape(64, 20), w["w2"].reshape(64, 64), w["w3"].reshape(64)
    w["b1"], w["b2"] = bits["b1"].astype(np.float64), bits["b2"].astype(np.float64)
    lat = smc.Lattice(*dims, S)
    occ_h = rng.integers(0, S, lat.nsites).astype(np.int8)
    model = smc.Model(smc.MLP_BF16, mlp=bits)
    g = torch.full((smc.grad_size(lat, model),), float("nan"), dtype=torch.float32, device="cuda")
    smc.energy_grad(lat, model, torch.from_numpy(occ_h).cuda(), g)
    smc.check()
    got = g.cpu().numpy().astype(np.float64)
    X = helpers.mlp_features(occ_h, dims, np.arange(lat.nsites))
    want, scale = _reference(X, w), helpers.mlp_grad_abs_terms(X, w)
    err = np.abs(got - want)
    assert np.all(err <= REL * scale + 1e-7), (np.flatnonzero(~(err <= REL * scale + 1e-7))[:5], np.nanmax(err / (scale + 1e-30)))
    assert got[-1] == lat.nsites
