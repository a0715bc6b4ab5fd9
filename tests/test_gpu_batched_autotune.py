"""What a batched context does depends neither on the contexts before it nor on its layout.

The default layout of a chain length follows the number of chains (32 x 1 for one
wave of warps, 16 x 2 above; 16 x 1 and 8 x 2), and a chunk is one kernel launch per
layout in use: two lengths of the same size class share one, also when a small
context has tuned one of the two lengths before.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu


def _launches(els):
    g = SlipSpring(els, precision="fp32", seed=2)
    g.set_params(**synth.PAPER, corr_levels=-1, chunk_steps=50)
    g.set_batched(True)
    g.run(0)
    before = g.counters()["launches"]
    g.run(50)
    n = g.counters()["launches"] - before
    g.close()
    return n


# lengths that no other test uses in batched mode: the cache is the process's
@pytest.mark.parametrize("M,before,after", [(16384, 29, 28), (9001, 10, 9), (16384, 19, 18)])
def test_small_context_first(cuda_ok, M, before, after):
    assert _launches([(500, before)]) == 1
    assert _launches([(M, before), (M, after)]) == 1


def _first_logs(els):
    g = SlipSpring(els, precision="fp32", seed=6)
    g.set_params(**dict(synth.PAPER, N0=2.0), corr_levels=-1, groups=1, log_every=7, max_logs=10, recenter_every=20)
    g.set_batched(True)
    g.set_flow(synth.shear_kappa(0.1), 0)
    g.run(70)
    assert g.status() == 0
    out = g.get_state(0), g.log_sums(0)[1]
    g.close()
    return out


# 16 x 1 alone and 8 x 2 beside many chains of the length; 32 x 1, 16 x 2 and 8 x 3
@pytest.mark.parametrize("N,others", [(9, (21000,)), (13, (21000, 9000)), (16, (21000,)), (17, (5000, 9000)),
                                      (24, (5000, 9000)), (26, (5000,)), (32, (5000,))])
def test_stress_logs_are_the_same_in_every_layout(cuda_ok, N, others):
    st, ref = _first_logs([(64, N)])
    for M in others:
        s, log = _first_logs([(64, N), (M, N)])
        for k in st:
            assert np.array_equal(s[k], st[k]), k
        # FP64 additions of the same FP32 stresses in any order; another order of a
        # chain's sum over beads would show at 1e-8
        assert np.allclose(log, ref, rtol=1e-12, atol=1e-12 * np.abs(ref).max())
