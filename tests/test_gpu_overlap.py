"""Work that runs side by side inside one ss_run, against the same work in one stream.

A run of 256 steps or more of an ensemble larger than the chip holds at once is
split into parts on several streams, and several elements run beside one another
(32 steps or more); runs of fewer steps use one stream.  The same steps taken
either way give the same bits: states, correlator sums (same launches) and event
counts.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu


def _run(els, timed, steps, precision="fp32", **kw):
    g = SlipSpring(els, precision=precision, seed=31)
    g.set_params(**synth.PAPER, corr_levels=6, groups=8, chunk_steps=130, **kw)
    g.kernel_timing(timed)  # timed launches stay on one stream
    g.run(7)
    g.run(steps)
    g.kernel_timing(False)
    assert g.status() == 0
    out = [(g.get_state(e), g.corr_sums(e)[0]) for e in range(len(els))]
    cnt = g.counters()
    g.close()
    return out, {k: cnt[k] for k in ("hops_up", "hops_down", "created", "destroyed")}


@pytest.mark.parametrize("els,precision,kw", [
    ([(7500, 32)], "fp32", {}),                      # 1.2 waves, a ragged last slice
    ([(65, 16), (130, 40), (1, 8), (700, 24)], "fp32", {}),  # elements beside one another
    ([(3900, 80)], "fp32", {"corr_tt": 1}),
    ([(3800, 24)], "fp64", {}),
])
def test_parts_and_elements_side_by_side_equal_one_stream(cuda_ok, els, precision, kw):
    a, ca = _run(els, False, 300, precision, **kw)
    b, cb = _run(els, True, 300, precision, **kw)
    assert ca == cb
    for (sa, ra), (sb, rb) in zip(a, b):
        for k in ("Z", "S", "R", "A"):
            assert np.array_equal(sa[k], sb[k]), k
        assert np.array_equal(ra, rb)


def test_one_step_calls_sum_the_same_products(cuda_ok):
    """The correlator of one-step launches against one launch of the same steps: the
    same products, summed in FP64 instead of FP32 along a launch."""
    out = []
    for steps in ([1] * 45, [45]):
        g = SlipSpring([(200, 20)], precision="fp64", seed=4)
        g.set_params(**synth.PAPER, corr_levels=6, groups=2, corr_tt=1)
        for n in steps:
            g.run(n)
        out.append((g.get_state(), g.corr_sums()[0], g.corr_sums_tt()[0]))
        g.close()
    (sa, ra, ta), (sb, rb, tb) = out
    assert np.array_equal(sa["S"], sb["S"]) and np.array_equal(sa["R"], sb["R"])
    # FP64 products and sums of at most 45 x 200 terms in another order
    for x, y in ((ra, rb), (ta, tb)):
        assert np.max(np.abs(x - y)) <= 1e-12 * np.max(np.abs(y))
