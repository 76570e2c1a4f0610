"""Replicas of small boxes: one CTA each, or resident blocks that share launches.
One replica more than a launch holds must not cost much more, on either side of
the line between the two."""
import time

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


def _call(smc, edge, R, n):
    lats = [smc.Lattice(edge, edge, edge, 5) for _ in range(R)]
    g = torch.Generator(device="cuda").manual_seed(R)
    occs = [torch.randint(0, 5, (l.nsites,), dtype=torch.int8, device="cuda", generator=g) for l in lats]
    model = smc.Model(smc.PAIR_F32, 2, inputs.pair_f32_coeffs(7, 2, 5))
    kT = np.repeat(inputs.ladder_kT(R)[:, None], n, axis=1)
    return lats, occs, lambda: smc.sweep_batched(lats, model, occs, 1, 0, n, kT), model, kT


def _ms(fn):
    fn()
    best = float("inf")
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        fn()
        torch.cuda.synchronize()
        best = min(best, 1e3 * (time.perf_counter() - t))
    return best


# 152 SMs hold sixteen replicas of 20^3 (nine blocks each) or nine of 16^3 (sixteen blocks) at a time
@pytest.mark.parametrize("edge,few,more,most", [(20, 15, 16, 1.15), (20, 16, 17, 1.45), (16, 9, 10, 1.15), (16, 15, 16, 1.15)])
def test_one_replica_more(smc, edge, few, more, most):
    a, b = (_ms(_call(smc, edge, R, 100)[2]) for R in (few, more))
    assert b <= most * a, (a, b)


@pytest.mark.parametrize("edge,R", [(16, 2), (16, 10), (20, 16), (20, 17)])
def test_replicas_equal_single_calls(smc, edge, R):
    lats, occs, fn, model, kT = _call(smc, edge, R, 3)
    single = [o.clone() for o in occs]
    fn()
    for r in range(R):
        smc.sweep(lats[r], model, single[r], 1, 0, 3, kT[r], replica=r)
        assert torch.equal(occs[r], single[r])
    smc.check()


def test_replicas_of_odd_boxes_equal_single_calls(smc):
    lats, occs, fn, model, kT = _call(smc, 5, 6, 4)
    single = [o.clone() for o in occs]
    fn()
    for r in range(6):
        smc.sweep(lats[r], model, single[r], 1, 0, 4, kT[r], replica=r)
        assert torch.equal(occs[r], single[r])
    smc.check()
