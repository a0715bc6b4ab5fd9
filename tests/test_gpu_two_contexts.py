"""Contexts of one process that need different amounts of shared memory.

The shared memory a kernel may be launched with belongs to the function, not to a
context: a context without stress logs, prepared or run in between, must not take away
what another one's launches and graphs need.
"""
import threading

import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu


def _ctx(els, every, batched):
    g = SlipSpring(els, precision="fp32", seed=12)
    logs = dict(log_every=every, max_logs=3000 // every) if every else {}
    g.set_params(**synth.PAPER, corr_levels=-1, groups=2, chunk_steps=1000, **logs)
    g.set_batched(batched)
    return g


# shared memory of a CTA: 118 KB and 60 KB of log sums; 8 KB and 7 KB
@pytest.mark.parametrize("batched", [True, False])
@pytest.mark.parametrize("every", [(1, 2), (100, 0), (1, 0)])
def test_contexts_in_turn(cuda_ok, batched, every):
    els = [(130, 32), (65, 16), (40, 48)]
    first, second = (_ctx(els, e, batched) for e in every)
    for g in (first, second, first, second, first):
        g.run(600)
    ref = _ctx(els, every[0], batched)
    ref.run(1800)
    for e in range(len(els)):
        a, b = first.get_state(e), ref.get_state(e)
        for k in a:
            assert np.array_equal(a[k], b[k]), k
        (ta, la), (tb, lb) = first.log_sums(e), ref.log_sums(e)
        assert np.array_equal(ta, tb) and len(ta) == 1800 // every[0]
        assert np.allclose(la, lb, rtol=1e-12, atol=1e-12 * np.abs(lb).max())
    for g in (first, second, ref):
        assert g.status() == 0
        g.close()


def test_contexts_in_threads(cuda_ok):
    """Each thread's runs alternate launches of one kernel with 60 to 230 KB of it."""
    errors = []

    def work(every):
        try:
            g = _ctx([(64, 32)], every, False)
            for _ in range(40):
                g.run(1000 // 20)
                g.reset_observables()
            for _ in range(3):
                g.run(900)
                g.reset_observables()
            assert g.status() == 0
            g.close()
        except Exception as ex:  # noqa: BLE001
            errors.append(ex)

    threads = [threading.Thread(target=work, args=(e,)) for e in (1, 2, 3, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_an_error_is_reported_once(cuda_ok):
    """A context too large for the device fails, and the next one does not."""
    big = SlipSpring([(1 << 30, 128)], precision="fp32", seed=1)
    with pytest.raises(Exception, match="ENOMEM"):
        big.set_params(**synth.PAPER, corr_levels=-1)
    big.close()
    g = _ctx([(64, 16)], 0, False)
    g.run(5)
    assert g.status() == 0 and g.step == 5
    g.close()
