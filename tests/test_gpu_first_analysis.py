"""A batch's first analysis is launched as it is, later ones replay its graph: both under
the caller's own capture, on the first call's stream and on another one."""
from __future__ import annotations

import numpy as np
import pytest

import paam_gen as g
from gpu_util import ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("calls_before", [0, 1, 2])
@pytest.mark.parametrize("same_stream", [True, False])
def test_analysis_under_capture(calls_before, same_stream):
    import torch

    import paper_2404_06452_gb300 as pkg

    sy = g.generate("cfg3", n_sys=300, seed=8)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    R = torch.zeros(sy.n_chain, dtype=torch.int64, device="cuda")
    status = torch.zeros(sy.n_chain, dtype=torch.uint8, device="cuda")
    verdict = torch.zeros(sy.n_sys, dtype=torch.uint8, device="cuda")
    want = [t.cpu().numpy() for t in pkg.analyze(ctx(), b)]
    other = pkg.paam_rta_load_systems(ctx(), sy)  # no call yet
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(calls_before):
        pkg.paam_rta_analyze_batch(ctx(), other, pkg.analysis_opts(), R, status, verdict, stream=first)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=first if same_stream else second):
        pkg.paam_rta_analyze_batch(ctx(), other, pkg.analysis_opts(), R, status, verdict,
                                   stream=torch.cuda.current_stream())
    torch.cuda.synchronize()
    for t in (R, status, verdict):
        t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for t, w in zip((R, status, verdict), want):
        assert np.array_equal(t.cpu().numpy(), w)
    graph.reset()
    other.free()
    b.free()
