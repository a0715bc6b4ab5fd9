"""ss_run captured into a CUDA graph by the caller.

The graph holds every launch of the run, also those on streams beside the context's,
and its replays advance the device state and the logs without a call of the library:
what is read afterwards is what the device holds, also if it was read before.
"""
import numpy as np
import pytest

import synth
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu


def _ctx(stream, els, levels):
    g = SlipSpring(els, precision="fp32", seed=3, stream=stream.cuda_stream)
    g.set_params(**synth.PAPER, corr_levels=levels, groups=8, log_every=7, max_logs=100)
    g.run(0)
    return g


@pytest.mark.parametrize("many", [True, False])
def test_replay_is_the_run(cuda_ok, many):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # several elements on streams of their own, or one in parts
    els, levels = ([(300, 16), (130, 40), (64, 60)], -1) if many else ([(52 * sms, 32)], 4)
    ref = _ctx(torch.cuda.Stream(), els, levels)
    ref.run(300)
    stream = torch.cuda.Stream()
    g = _ctx(stream, els, levels)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        g.run(300)
    for e in range(len(els)):
        assert not np.any(g.log_sums(e)[1])  # nothing has run
    with torch.cuda.stream(stream):
        graph.replay()
    torch.cuda.synchronize()
    for e in range(len(els)):
        a, b = ref.get_state(e), g.get_state(e)
        for k in a:
            assert np.array_equal(a[k], b[k]), k
        if levels > 0:
            assert np.array_equal(ref.corr_sums(e)[0], g.corr_sums(e)[0])
        (ta, la), (tb, lb) = ref.log_sums(e), g.log_sums(e)
        assert np.array_equal(ta, tb) and len(ta) == 42
        # FP64 additions of the same numbers in any order
        assert np.allclose(la, lb, rtol=1e-12, atol=1e-12 * np.abs(la).max())
        assert np.allclose(ref.stress(e)[1], g.stress(e)[1], rtol=1e-9, atol=1e-12)
    del graph
    ref.close()
    g.close()
