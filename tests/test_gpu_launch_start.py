"""The first step of a launch.

A launch lays the chains' positions, bond vectors, spring records and slot masks out
in shared memory before its first step, whose forces read entries that other lanes
wrote.  Runs of one launch per step take that first step every time: their states,
spring lists and event counts are those of one launch over all steps bit for bit, in
every lane layout, with both integrators and with a flow, and the gradient of a window
does not depend on where its replayed segments start.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu

STEPS = 41


def _run(M, N, precision, chunk, flow, **kw):
    g = SlipSpring([(M, N)], precision=precision, seed=17)
    g.set_params(**dict(synth.PAPER, **kw), corr_levels=-1, chunk_steps=chunk, recenter_every=10)
    if flow:
        # (the Heun corrector sums in another order in launches without a flow)
        g.set_flow(synth.shear_kappa(0.2), 0 if kw.get("integrator") else 3)
    g.run(STEPS)
    assert g.status() == 0
    out, cnt = g.get_state(), g.counters()
    g.close()
    return out, {k: cnt[k] for k in ("hops_up", "hops_down", "created", "destroyed")}


# lane layouts 8 x 1, 16 x 1, 8 x 2, 16 x 2, 8 x 3, 16 x 3, 16 x 4, 32 x 3, 32 x 4;
# N0 = 1 puts three and more springs on many beads
@pytest.mark.parametrize("M,N,precision", [(67, 8, "fp32"), (301, 13, "fp32"), (40001, 16, "fp32"), (301, 32, "fp32"),
                                           (8195, 23, "fp32"), (301, 40, "fp32"), (301, 62, "fp32"),
                                           (301, 80, "fp32"), (301, 128, "fp32"), (301, 16, "fp64"),
                                           (301, 50, "fp64")])
@pytest.mark.parametrize("flow,kw", [(False, {}), (True, dict(N0=1.0)), (True, dict(integrator=1)),
                                     (False, dict(integrator=1, N0=1.0))])
def test_one_step_launches_equal_one_launch(cuda_ok, M, N, precision, flow, kw):
    (a, ca), (b, cb) = (_run(M, N, precision, chunk, flow, **kw) for chunk in (1, STEPS))
    assert ca == cb
    for k in ("Z", "S", "R", "A"):
        assert np.array_equal(a[k], b[k]), k


# reverse sweeps 8 x 1, 16 x 1 (recorded in 8 x 2), 8 x 3 and 16 x 2
@pytest.mark.parametrize("M,N,precision", [(100, 7, "fp64"), (100, 16, "fp64"), (100, 30, "fp64"),
                                           (40003, 11, "fp32"), (8195, 24, "fp32"), (67, 8, "fp32")])
def test_gradient_does_not_depend_on_the_segments(cuda_ok, M, N, precision):
    out = []
    for every in (1, 6, 40):
        g = SlipSpring([(M, N)], precision=precision, seed=18)
        g.set_params(**dict(synth.PAPER, N0=2.0), corr_levels=4, chunk_steps=64)
        g.run(20)
        g.window_forward(40, every)
        dG = np.linspace(0.5, 1.5, 64).reshape(4, 16)
        dG[1:, :8] = 0.0
        out.append((g.get_state(), g.window_backward(dG)))
        g.close()
    # A chain's sums are folded into FP64 at every segment start and every 32 steps
    # and added up in FP64: up to 40 terms of rounding eps regrouped.  The sums cancel
    # between chains and steps, hence the factor on the largest component.
    eps = np.finfo(np.float64 if precision == "fp64" else np.float32).eps
    for st, grad in out[:-1]:
        for k in ("Z", "S", "R", "A"):
            assert np.array_equal(st[k], out[-1][0][k]), k
        assert np.all(np.isfinite(grad)) and np.max(np.abs(grad)) > 0
        assert np.max(np.abs(grad - out[-1][1])) <= 1e3 * eps * np.max(np.abs(out[-1][1])), (grad, out[-1][1])
