"""Parts of one ensemble and elements beside one another: that work is split, and that
the split changes nothing, with logs, flows and both integrators.

Ensembles are sized by the SM count to a little more than the chip holds at once.
Timed launches stay whole and on one stream; a split run has more launches.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _run(els, timed, precision, flow, **kw):
    g = SlipSpring(els, precision=precision, seed=51)
    g.set_params(**synth.PAPER, groups=8, chunk_steps=130, recenter_every=50, **kw)
    if flow:
        for e in range(len(els)):
            g.set_flow(synth.shear_kappa(0.1 / (e + 1)), 0, elem=e)
            g.set_flow(synth.shear_kappa(0.05), 200, elem=e)
    g.kernel_timing(timed)
    g.run(9)
    before = g.counters()["launches"]
    g.run(300)
    g.kernel_timing(False)
    assert g.status() == 0
    cnt = g.counters()
    out = []
    for e in range(len(els)):
        corr = g.corr_sums(e)[0] if kw["corr_levels"] > 0 else np.zeros(1)
        out.append((g.get_state(e), corr, g.log_sums(e)))
    g.close()
    return out, {k: cnt[k] for k in ("hops_up", "hops_down", "created", "destroyed")}, cnt["launches"] - before


# chains per SM, length, precision, flow, parameters: one and a fifth to one and a half
# waves of 20, 16, 12 and 24 warps per SM
@pytest.mark.parametrize("per_sm,N,precision,flow,kw", [
    (52, 32, "fp32", True, dict(corr_levels=-1, log_every=7, max_logs=60)),
    (52, 32, "fp32", False, dict(corr_levels=5, log_every=50, max_logs=10)),
    (52, 30, "fp32", False, dict(corr_levels=5, integrator=1)),
    (42, 25, "fp32", True, dict(corr_levels=3, integrator=1, log_every=50, max_logs=10)),
    (36, 60, "fp32", True, dict(corr_levels=-1, log_every=20, max_logs=20)),
    (30, 24, "fp64", True, dict(corr_levels=4, log_every=50, max_logs=10)),
])
def test_parts(cuda_ok, per_sm, N, precision, flow, kw):
    els = [(per_sm * _sms() + 1, N)]
    (a, ca, na), (b, cb, nb) = (_run(els, timed, precision, flow, **kw) for timed in (False, True))
    assert na > nb, (na, nb)
    _same(a, b, ca, cb)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_elements(cuda_ok, precision):
    els = [(300, 16), (130, 40), (1, 8), (700, 24), (65, 90), (64, 50), (200, 2), (90, 128), (33, 32)]
    kw = dict(corr_levels=4, log_every=10, max_logs=40)
    (a, ca, na), (b, cb, nb) = (_run(els, timed, precision, True, **kw) for timed in (False, True))
    assert na == nb  # whole elements, on eight streams
    _same(a, b, ca, cb)


def _same(a, b, ca, cb):
    assert ca == cb
    for (sa, ra, (ta, la)), (sb, rb, (tb, lb)) in zip(a, b):
        for k in ("Z", "S", "R", "A"):
            assert np.array_equal(sa[k], sb[k]), k
        assert np.array_equal(ra, rb) and np.array_equal(ta, tb)
        # FP64 additions of the same numbers in any order
        assert np.allclose(la, lb, rtol=1e-12, atol=1e-12 * (np.abs(lb).max() if lb.size else 1.0))
