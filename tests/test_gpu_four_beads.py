"""The two forms of the chain kernel for N = 49..64, bit for bit.

Which form runs follows the number of chains: the first up to 12 warps per SM (13 with
Heun, eight of the second with Heun and a flow), the second where that saves a wave.
Chains of one seed and global id draw the same numbers in any ensemble, and both forms
round alike, so the first 64 chains are equal in states and correlator sums whatever
ensemble they are part of.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu

STEPS = 123  # odd: ends inside a reduction batch of either form


def _run(M, N, flow, integrator, levels):
    g = SlipSpring([(M, N)], precision="fp32", seed=41)
    g.set_params(**dict(synth.PAPER, N0=2.0), corr_levels=levels, groups=-(-M // 64), integrator=integrator,
                 log_every=40, max_logs=3, recenter_every=30, chunk_steps=70)
    if flow:
        g.set_flow(synth.shear_kappa(0.1), 0)
    g.run(STEPS)
    assert g.status() == 0
    acc = g.corr_sums()[0][0] if levels > 0 else None
    out = g.get_state(), acc, g.log_sums()[1][:, 0]
    g.close()
    return out


@pytest.mark.parametrize("N", [49, 62])
@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("integrator", [0, 1])
@pytest.mark.parametrize("levels", [-1, 4])
def test_first_chains_are_the_same_in_any_ensemble(cuda_ok, N, flow, integrator, levels):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ref, acc, log = _run(64, N, flow, integrator, levels)
    # two chains per warp: 9, 14 and 29 warps per SM
    for M in (18 * sms + 1, 28 * sms, 58 * sms):
        st, a, lg = _run(M, N, flow, integrator, levels)
        for k in ("Z", "S", "R", "A"):
            assert np.array_equal(st[k][:64], ref[k]), (M, k)
        if levels > 0:  # FP64 sums of a slice's parts, 16 or 32 chains each
            assert np.allclose(a, acc, rtol=1e-13, atol=1e-13 * np.abs(acc).max())
        assert np.allclose(lg, log, rtol=1e-12, atol=1e-9)
