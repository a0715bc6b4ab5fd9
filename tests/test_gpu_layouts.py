"""Lane layouts of the chain kernel against one another, bit for bit.

A large ensemble of short chains runs eight lanes per chain (N = 9..16 from
40000 chains on, N = 17..24 from 8192), a small one sixteen.  Chains of one seed
and global id draw the same numbers in any ensemble, and every layout rounds each
operation and each sum over beads alike, so the first 64 chains of both, their
spring lists and the correlator sums of their slice are equal bitwise.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu

STEPS = 130  # ends inside a batch of reduced stress samples; crosses a recentring step


def _run(M, N, flow, N0):
    g = SlipSpring([(M, N)], precision="fp32", seed=21)
    kw = dict(synth.PAPER, N0=N0)
    g.set_params(**kw, corr_levels=4, groups=-(-M // 64), log_every=50, max_logs=4, recenter_every=60, chunk_steps=70)
    if flow:
        g.set_flow(synth.shear_kappa(0.1), 20)
    g.run(STEPS)
    assert g.status() == 0
    acc, _ = g.corr_sums()
    out = g.get_state(), acc[0], g.log_sums()[1][:, 0]
    g.close()
    return out


@pytest.mark.parametrize("N,M", [(9, 40001), (16, 40000), (17, 8192), (23, 8195), (24, 8192)])
@pytest.mark.parametrize("flow,N0", [(False, 4.0), (True, 4.0), (True, 1.0)])
def test_eight_lanes_per_chain_equal_sixteen(cuda_ok, N, M, flow, N0):
    big, acc_b, log_b = _run(M, N, flow, N0)
    small, acc_s, log_s = _run(64, N, flow, N0)
    for k in ("Z", "S", "R", "A"):
        assert np.array_equal(big[k][:64], small[k]), k
    assert np.array_equal(acc_b, acc_s)
    # the log sums of a group are FP64 atomics, equal up to their order
    assert np.allclose(log_b, log_s, rtol=1e-12, atol=1e-9)
