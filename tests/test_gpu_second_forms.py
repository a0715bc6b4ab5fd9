"""The two forms of the chain kernel in layouts that have them, bit for bit.

Which form runs follows the number of chains: the second where that saves a wave of
warps (at N = 49..64 with Heun and a flow in small ensembles, too).
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


def _check(N, flow, integrator, levels, per_sm):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ref, acc, log = _run(64, N, flow, integrator, levels)
    for chains in per_sm:
        M = chains * sms + 1
        st, a, lg = _run(M, N, flow, integrator, levels)
        for k in ("Z", "S", "R", "A"):
            assert np.array_equal(st[k][:64], ref[k]), (M, k)
        if levels > 0:  # FP64 sums of a slice's parts, 16 or 32 chains each
            assert np.allclose(a, acc, rtol=1e-13, atol=1e-13 * np.abs(acc).max())
        assert np.allclose(lg, log, rtol=1e-12, atol=1e-9)


# two chains per warp: 9, 14 and 29 warps per SM
@pytest.mark.parametrize("N", [49, 62])
@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("integrator", [0, 1])
@pytest.mark.parametrize("levels", [-1, 4])
def test_four_beads_per_lane(cuda_ok, N, flow, integrator, levels):
    _check(N, flow, integrator, levels, (18, 28, 58))


# with a flow: 18 warps per SM of sixteen lanes (14 with Heun at three beads) and, from
# 8192 chains on, of eight
@pytest.mark.parametrize("N,integrator,per_sm", [(33, 0, 36), (48, 0, 36), (24, 0, 72), (17, 0, 72), (18, 1, 36),
                                                 (32, 1, 36), (35, 1, 28), (48, 1, 28)])
@pytest.mark.parametrize("levels", [-1, 4])
def test_flow_at_two_and_three_beads(cuda_ok, N, integrator, per_sm, levels):
    _check(N, True, integrator, levels, (per_sm,))


@pytest.mark.parametrize("flow", [False, True])
@pytest.mark.parametrize("levels", [-1, 2])
def test_allocation_free_call(cuda_ok, flow, levels):
    import ctypes

    import torch
    from paper_1106_2899_gb300 import _native as nat
    from test_zz_no_alloc import _from_device_layout, _to_device_layout
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    M, N, n = 28 * sms, 61, 33
    zm = N
    st0 = synth.random_state(M, N, zm, seed=3, z_mean=N / 4)
    kappa = np.ascontiguousarray(synth.shear_kappa(0.05 if flow else 0.0))
    g = SlipSpring([(M, N)], precision="fp32", seed=8)
    g.set_params(**synth.PAPER, corr_levels=levels)
    g.set_state(st0)
    if flow:
        g.set_flow(kappa, 0)
    g.run(n)
    ref = g.get_state()
    g.close()
    p = nat.ss_params()
    for k, v in synth.PAPER.items():
        setattr(p, k, v)
    p.corr_levels = levels
    dev = [torch.from_numpy(x).cuda() for x in _to_device_layout(st0, N, zm, np.float32)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ptr = [ctypes.c_void_p(x.data_ptr()) for x in dev]
    rc = nat.load().ss_run_noalloc(ctypes.byref(p), nat.SS_FP32, 8, M, N, 0, 0, n,
                                   kappa.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), *ptr, None,
                                   ctypes.c_void_p(status.data_ptr()),
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0 and int(status.item()) == 0
    got = _from_device_layout(*[x.cpu().numpy() for x in dev], N, zm)
    for k in ("Z", "S", "R", "A"):
        assert np.array_equal(got[k], ref[k]), k
