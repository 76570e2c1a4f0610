"""The tabulated MLP sweeps (f looked up by feature vector) against the
evaluating kernels: the same occupancy and accepted count, bit for bit.

Two and three species have so few feature vectors that every sweep is
tabulated; the reference is the traced mini-steps, which evaluate every row.
With four and five species a call of one sweep evaluates its rows and a call
of many looks them up; the same sweeps in one call and one by one must agree."""
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


def _model(smc, kind, S):
    if kind == "mlp":
        return smc.Model(smc.MLP_BF16, mlp=inputs.mlp_weights(3))
    if kind == "net":
        return smc.Model(smc.MLPNET_BF16, net=inputs.mlpnet_weights(3))
    return smc.Model(smc.PAIR_F32_MLP_BF16, 3, inputs.pair_f32_coeffs(5, 3, S), mlp=inputs.mlp_weights(3))


def _start(smc, dims, S, seed):
    lat = smc.Lattice(*dims, S)
    occ = torch.empty(lat.nsites, dtype=torch.int8, device="cuda")
    smc.init_lattice(lat, inputs.dirichlet_counts(lat.nsites, S, seed), seed, occ)
    return lat, occ


def _run(smc, lat, model, occ, seed, sweep0, n, kT):
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    a = torch.zeros(1, dtype=torch.int64, device="cuda")
    smc.sweep(lat, model, occ, seed, sweep0, n, kT, e_acc=e, n_acc=a)
    return e, a


# rows of two link cells, of a number that does not fill whole warps, of one warp and of the longest row
@pytest.mark.parametrize("dims", [(8, 8, 8), (36, 12, 8), (32, 8, 20), (512, 8, 8)])
@pytest.mark.parametrize("kind,S", [("mlp", 2), ("pair+mlp", 3), ("net", 3)])
def test_tabulated_sweep_equals_traced_ministeps(smc, dims, kind, S):
    kT, seed = inputs.K_B_EV * 300.0, 11
    lat, occ = _start(smc, dims, S, seed)
    model = _model(smc, kind, S)
    ref = occ.clone()
    e, a = _run(smc, lat, model, occ, seed, 4, 1, kT)
    dE = torch.zeros(lat.nsites // 128, dtype=torch.float32, device="cuda")
    acc = torch.zeros(lat.nsites // 128, dtype=torch.uint8, device="cuda")
    n, tot = 0, 0.0
    for k in range(128):
        smc.ministep_trace(lat, model, ref, seed, 4, k, kT, dE=dE, acc=acc)
        n += int(acc.sum())
        tot += float(dE.double()[acc.bool()].sum())
    smc.check()
    assert torch.equal(occ, ref)
    assert int(a) == n
    # the same FP32 dE values summed in FP64 in another order
    assert abs(float(e) - tot) <= 1e-12 * lat.nsites


@pytest.mark.parametrize("dims,kind,S,n", [((64, 32, 16), "mlp", 4, 20), ((40, 32, 24), "pair+mlp", 4, 20),
                                           ((128, 128, 128), "mlp", 5, 12), ((200, 104, 100), "net", 5, 12),
                                           ((512, 64, 64), "pair+mlp", 5, 12)])
def test_one_call_of_many_sweeps_equals_calls_of_one(smc, dims, kind, S, n):
    kT, seed = inputs.K_B_EV * np.linspace(900.0, 500.0, n), 7
    lat, occ = _start(smc, dims, S, seed)
    model = _model(smc, kind, S)
    ref = occ.clone()
    e, a = _run(smc, lat, model, occ, seed, 0, n, kT)
    tot, cnt = 0.0, 0
    for t in range(n):
        et, at = _run(smc, lat, model, ref, seed, t, 1, float(kT[t]))
        tot += float(et)
        cnt += int(at)
    smc.check()
    assert torch.equal(occ, ref)
    assert int(a) == cnt
    assert abs(float(e) - tot) <= 1e-12 * lat.nsites * n
