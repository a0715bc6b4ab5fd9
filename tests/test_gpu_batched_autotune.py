"""The layout of a batched context does not depend on the contexts before it.

The default layout of a chain length follows the number of chains (32 x 1 for one
wave of warps, 16 x 2 above; 16 x 1 and 8 x 2), and a chunk is one kernel launch per
layout in use: two lengths of the same size class share one, also when a small
context has tuned one of the two lengths before.
"""
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
