"""The accepted count of a small box swept by one CTA needs 64 bits: a call may
have more trials than a 32-bit counter holds, with one lane counting them all.
Showing it on the device takes minutes (the trials of such a box follow one
another), so the kernel's counters are looked at here, and the long run is made
only when SMC_LONG_TESTS is set."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_08250_gb300", "csrc")


def test_counters_that_live_for_a_launch_are_64_bits():
    # 41^3 cells: one link cell, 2 * 41^3 trials per sweep, all by one lane
    assert (2 ** 31 // (2 * 41 * 41) - 1) * 2 * 41 ** 3 > 2 ** 31
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "sweep_cta.cu")).read())
    flushed = set(re.findall(r"atomicAdd\(&s_[en], \(unsigned long long\)(\w+)\)", text))
    assert flushed == {"accE", "accN"}
    for name in flushed:
        kinds = re.findall(r"((?:unsigned |long )*(?:int|long|uint32_t))\s*&?\s*" + name + r"\b", text)
        assert kinds and all(k == "long long" for k in kinds), (name, kinds)
        assert re.search(r"long long[^;()]*\b" + name + r" = 0", text), name  # accE, accN of the kernel


@pytest.mark.gpu
@pytest.mark.skipif(not os.environ.get("SMC_LONG_TESTS"), reason="minutes of sweeps: set SMC_LONG_TESTS")
def test_more_than_two_to_the_31_accepted():
    torch = pytest.importorskip("torch")
    from paper_2604_08250_gb300 import smc
    lat, n = smc.Lattice(4, 4, 4, 2), 2 ** 24 + 5  # one trial per mini-step, 128 per sweep, every one accepted
    occ = torch.zeros(lat.nsites, dtype=torch.int8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    smc.sweep(lat, smc.Model(smc.PAIR_F32, 2, np.zeros((2, 2, 2), np.float32)), occ, 1, 0, n, float("inf"), n_acc=cnt)
    smc.check()
    assert int(cnt) == 128 * n
