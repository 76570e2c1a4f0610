"""Models from parameter vectors: the layout entry by entry, and BF16 rounding
against integer arithmetic on single values (ties, overflow into infinity, NaN
and negative patterns included)."""
import numpy as np
import pytest

from paper_2604_08250_gb300 import smc


def _bits(x):
    u = int(np.float32(x).view(np.uint32))
    return ((u + 0x7FFF + ((u >> 16) & 1)) >> 16) & 0xFFFF


def test_bf16_bits():
    rng = np.random.default_rng(1)
    u = np.concatenate([rng.integers(0, 2 ** 32, 4000, dtype=np.uint32),
                        np.array([0, 0x80000000, 0x3F808000, 0x3F818000, 0x7F7FFFFF, 0x7F800000, 0xFF800000,
                                  0x7FC00000, 0x7FFFFFFF, 0xFFFFFFFF, 0xFFFF8000, 1], dtype=np.uint32)])
    a = u.view(np.float32)
    got = smc._bf16_bits(a)
    assert got.dtype == np.uint16
    assert [int(g) for g in got] == [((int(x) + 0x7FFF + ((int(x) >> 16) & 1)) >> 16) & 0xFFFF for x in u]


@pytest.mark.parametrize("kind", [smc.PAIR_F32, smc.MLP_BF16, smc.PAIR_F32_MLP_BF16])
@pytest.mark.parametrize("nshells,S", [(1, 1), (2, 5), (3, 2), (3, 8)])
def test_layout(kind, nshells, S):
    pair, mlp = kind != smc.MLP_BF16, kind != smc.PAIR_F32
    n = (smc.n_pair_params(nshells, S) if pair else 0) + (smc.MLP_NPARAM if mlp else 0)
    th = np.random.default_rng(2).normal(size=n)
    m = smc.model_from_theta(kind, nshells, S, th)
    k = 0
    if pair:
        flat = [float(m._c.v_f32[i]) for i in range(nshells * S * S)]
        for a in range(nshells):
            for p in range(S):
                for q in range(p, S):
                    assert flat[(a * S + p) * S + q] == flat[(a * S + q) * S + p] == np.float32(th[k])
                    k += 1
    if mlp:
        for name, size in (("w1", 1280), ("b1", 64), ("w2", 4096), ("b2", 64), ("w3", 64)):
            ptr = getattr(m._c, "mlp_" + name)
            for i in range(size):
                assert ptr[i] == (_bits(th[k]) if name[0] == "w" else np.float32(th[k]))
                k += 1
        assert m._c.mlp_b3 == np.float32(th[k])
        k += 1
    assert k == n
    for bad in (th[:-1], np.append(th, 0.0), th[:0]):
        with pytest.raises((ValueError, IndexError)):
            smc.model_from_theta(kind, nshells, S, bad)
