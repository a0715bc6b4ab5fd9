"""The batched launch against the per-element path, in every lane layout it chooses.

Both paths draw the same numbers and round every operation on a state alike, whatever
their layouts, so states and event counts are equal bit for bit, also under flows that
recentre the chains, whose centre of mass is a sum over beads.  The stress of a chain is
a sum over its beads in an order of the layout.  The layout of a chain length follows
the number of chains the context has of it.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu

# chains and length of one element, and the layout the batched launch takes on 152 SMs
ELEMENTS = {"8x1": (901, 8), "16x1": (3001, 16), "8x2 one wave": (9001, 16), "16x1 again": (15001, 13),
            "8x2": (20001, 11), "32x1": (1001, 32), "16x2": (5001, 32), "16x2 short": (5001, 20), "8x3": (8195, 23),
            "16x3": (1001, 41), "16x4": (1001, 57), "32x3": (501, 90), "32x4": (501, 101)}


def _run(els, precision, batched):
    g = SlipSpring(els, precision=precision, seed=23)
    g.set_params(**dict(synth.PAPER, N0=2.0), corr_levels=-1, groups=4, log_every=25, max_logs=8, chunk_steps=80,
                 recenter_every=20)
    if batched:
        g.set_batched(True)
    kap = np.random.default_rng(5).normal(0.0, 0.05, (len(els), 2, 3, 3))
    kap -= np.trace(kap, axis1=2, axis2=3)[:, :, None, None] / 3.0 * np.eye(3)
    for e in range(len(els)):
        g.set_flow(kap[e, 0], 0, elem=e)
        g.set_flow(kap[e, 1], 70, elem=e)
    g.run(150)
    assert g.status() == 0
    cnt = g.counters()
    out = [(g.get_state(e), g.log_sums(e)) for e in range(len(els))]
    g.close()
    return out, {k: cnt[k] for k in ("hops_up", "hops_down", "created", "destroyed")}


def _compare(els, precision):
    (a, ca), (b, cb) = (_run(els, precision, batched) for batched in (False, True))
    assert ca == cb
    for (sa, (ta, la)), (sb, (tb, lb)) in zip(a, b):
        for k in ("Z", "S", "R", "A"):
            assert np.array_equal(sa[k], sb[k]), k
        assert np.array_equal(ta, tb) and len(ta) == 6
        # up to 64 terms in another order, summed over chains in FP64
        eps = np.finfo(np.float64 if precision == "fp64" else np.float32).eps
        assert np.allclose(la, lb, rtol=64 * eps, atol=64 * eps * np.abs(la).max())


@pytest.mark.parametrize("name", ELEMENTS)
def test_one_length(cuda_ok, name):
    _compare([ELEMENTS[name]], "fp32")


def test_all_layouts_in_one_launch(cuda_ok):
    els = [ELEMENTS[k] for k in ("16x3", "8x2", "32x4", "8x1", "8x3", "32x1", "16x4", "32x3")]
    _compare(els + [(700, 41), (9, 8)], "fp32")


@pytest.mark.parametrize("M,N", [(9001, 16), (8195, 23), (301, 8), (301, 32), (5001, 30), (301, 90)])
def test_one_length_fp64(cuda_ok, M, N):
    _compare([(M, N)], "fp64")
