"""Reverse sweeps of short chains: eight lanes per chain, and windows recorded in a layout
of eight lanes and two beads, whose sweep runs sixteen lanes.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring
from test_gpu_adjoint import test_fp64_adjoint_matches_replayed_finite_differences as _check_fd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,every", [(8, 100), (5, 256)])
def test_eight_lanes_match_finite_differences(cuda_ok, N, every):
    _check_fd(N, every)


def _gradient(M, N, offset):
    g = SlipSpring([(M, N)], precision="fp32", seed=44, chain_offset=offset)
    g.set_params(**dict(synth.PAPER, N0=2.0), corr_levels=4, chunk_steps=64)
    g.run(20)
    g.window_forward(45, 16)
    dG = np.linspace(0.5, 1.5, 64).reshape(4, 16)
    dG[1:, :8] = 0.0
    out = M * g.window_backward(dG)  # a sum over chains
    assert g.status() == 0
    g.close()
    return out


# 40960 chains of 9..16 beads are recorded in 8 x 2, half of them in 16 x 1; 8192 chains
# of 17..24 beads in 8 x 3, half of them in 16 x 2
@pytest.mark.parametrize("M,N", [(40960, 16), (40960, 11), (8192, 24), (8192, 18)])
def test_gradient_is_the_sum_over_halves(cuda_ok, M, N):
    whole = _gradient(M, N, 0)
    halves = _gradient(M // 2, N, 0) + _gradient(M // 2, N, M // 2)
    # the weights of a half are exactly twice the whole's; a chain's FP32 sums of up to
    # 16 steps and 3 beads may be grouped otherwise
    eps = np.finfo(np.float32).eps
    assert np.max(np.abs(whole)) > 0
    assert np.max(np.abs(whole - halves)) <= 48 * eps * np.max(np.abs(whole)), (whole, halves)
