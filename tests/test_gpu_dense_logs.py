"""Stress logs at any density.

A launch keeps the sums of its log steps in shared memory, so a chunk with many of
them is split into launches of a bounded number: any log_every goes with any
chunk_steps, the sums do not depend on where launches end, and logs at every step hold
those at every tenth.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu

STEPS = 61


def _logs(els, precision, every, chunk, batched=False, levels=-1):
    g = SlipSpring(els, precision=precision, seed=29)
    g.set_params(**synth.PAPER, corr_levels=levels, groups=3, log_every=every, max_logs=STEPS // every,
                 chunk_steps=chunk)
    g.set_flow(synth.shear_kappa(0.1), 0)
    if batched:
        g.set_batched(True)
    g.run(7)
    g.run(STEPS - 7)
    assert g.status() == 0
    out = [g.log_sums(e) for e in range(len(els))]
    g.close()
    return out


def _same(a, b):
    """The sums are FP64 additions of the same numbers in any order."""
    for (ta, la), (tb, lb) in zip(a, b):
        assert np.array_equal(ta, tb)
        assert np.allclose(la, lb, rtol=1e-12, atol=1e-12 * np.abs(lb).max())


@pytest.mark.parametrize("precision,levels,batched", [("fp32", -1, False), ("fp32", 3, False), ("fp32", -1, True),
                                                      ("fp64", 3, False), ("fp64", -1, True)])
def test_sums_do_not_depend_on_launches(cuda_ok, precision, levels, batched):
    els = [(201, 32), (70, 8), (130, 40), (65, 90), (64, 60)]
    every_step = _logs(els, precision, 1, 1000, batched, levels)
    assert all(len(t) == STEPS and np.all(s[:, :, 12].sum(1) > 0) for t, s in every_step)
    for chunk in (1, 2, 5):
        _same(_logs(els, precision, 1, chunk, batched, levels), every_step)
    for every in (2, 3, 10):
        _same(_logs(els, precision, every, 1000, batched, levels),
              [(t[every - 1::every], s[every - 1::every]) for t, s in every_step])


@pytest.mark.parametrize("batched", [False, True])
def test_a_long_launch_with_a_log_every_step(cuda_ok, batched):
    g = SlipSpring([(130, 32)], precision="fp32", seed=1)
    g.set_params(**synth.PAPER, corr_levels=-1, groups=2, log_every=1, max_logs=3000, chunk_steps=3000)
    if batched:
        g.set_batched(True)
    g.run(3000)
    t, s = g.log_sums()
    assert g.status() == 0 and len(t) == 3000 and np.all(s[:, :, 12].sum(1) > 0)
    g.close()
