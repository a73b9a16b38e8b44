"""An analysis on a stream that is being captured is refused, with any number of earlier
calls on that stream or another, and leaves the capture and the batch as they were."""
from __future__ import annotations

import pytest

import paam_gen as g
from gpu_util import ctx
from test_gpu_analysis_order import _equal, _outputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("calls_before", [0, 1, 2])
@pytest.mark.parametrize("same_stream", [True, False])
@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_a_capturing_stream_is_refused(calls_before, same_stream, mode):
    import torch

    import paper_2404_06452_gb300 as pkg

    sy = g.generate("cfg3", n_sys=300, seed=8)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    want, got = _outputs(sy), _outputs(sy)
    pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(), *want)
    torch.cuda.synchronize()
    b.free()
    b = pkg.paam_rta_load_systems(ctx(), sy)  # no call yet
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    for _ in range(calls_before):
        pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(), *got, stream=first)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=first if same_stream else second, capture_error_mode=mode):
        x.add_(1)
        for _ in range(2):
            with pytest.raises(pkg.PaamError) as e:
                pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(), *got, stream=torch.cuda.current_stream())
            assert e.value.code == -4
        x.add_(1)
    graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 8
    for t in got:
        t.fill_(9)
    torch.cuda.synchronize()
    for _ in range(3):  # afterwards the batch is analysed as ever
        pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(), *got, stream=second)
        second.synchronize()
        assert _equal(got, want)
    graph.reset()
    b.free()
