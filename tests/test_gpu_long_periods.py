"""Batches with periods of seconds, whose range test takes the pass over single
chains (none, some or all of the systems), through the calls that validate on
their own: the pipelined analysis of host arrays and the allocation-free one,
against the CPU oracle; and systems past the limits, refused from any chunk."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paam_gen
from gpu_util import assert_same, ctx, gpu_analyze

pytestmark = pytest.mark.gpu

LIMIT = 1 << 40
N = 1_200
PERIODS = {"some": (1e9, 6e9), "all": (4.5e9, 2e10)}  # 2^32 ns = 4.3 s


def _batch(kind, acc=1):
    cfg = dict(paam_gen.CONFIGS["cfg3"], n_geom_p=1.0 / 9.0, util_lo=0.05, util_hi=0.5)
    t_min, t_max = PERIODS[kind]
    sy = paam_gen.generate(cfg, n_sys=N, p_spin=0.2, t_min=t_min, t_max=t_max)
    return paam_gen.assign_accelerators(sy, acc) if acc > 1 else sy


def _host(sy, chunk, **p):
    import paper_2404_06452_gb300 as pkg

    R = np.full(sy.n_chain, -7, np.int64)
    st = np.full(sy.n_chain, 0xEE, np.uint8)
    v = np.full(sy.n_sys, 0xEE, np.uint8)
    pkg.paam_rta_analyze_host(ctx(), sy, pkg.analysis_opts(**p), R, st, v, launch_config=-1, chunk_systems=chunk)
    return dict(R=R, status=st, verdict=v)


def _noalloc(sy, **p):
    import torch

    import paper_2404_06452_gb300 as pkg

    R = torch.full((sy.n_chain,), -7, dtype=torch.int64, device="cuda")
    st = torch.full((sy.n_chain,), 0xEE, dtype=torch.uint8, device="cuda")
    v = torch.full((sy.n_sys,), 0xEE, dtype=torch.uint8, device="cuda")
    pkg.paam_rta_analyze_noalloc(pkg.to_device(sy), pkg.analysis_opts(**p), R, st, v)
    torch.cuda.synchronize()
    return dict(R=R.cpu().numpy(), status=st.cpu().numpy(), verdict=v.cpu().numpy())


@pytest.mark.parametrize("kind", list(PERIODS))
@pytest.mark.parametrize("acc,mode", [(1, 0), (1, 1), (3, 0)])
def test_long_periods(kind, acc, mode):
    sy = _batch(kind, acc)
    p = dict(n_buckets=2, eps=300_000, kappa=20_000, blocking_mode=mode)
    ref = oracle.analyze(sy, threads=8, **p)
    assert set(np.unique(ref["status"])) >= {0, 1}
    assert_same(gpu_analyze(sy, **p), ref)
    assert_same(_noalloc(sy, **p), ref)
    for chunk in (0, 1, 250, 1_199):
        assert_same(_host(sy, chunk, **p), ref)


@pytest.mark.parametrize("at", [3, 600, N - 1])
def test_system_past_the_range_is_refused(at):
    """One system whose magnitude bound is not met, and one invalid one, among long periods."""
    import paper_2404_06452_gb300 as pkg

    for what, code in (("range", -2), ("inval", -1)):
        sy = _batch("some").subset(np.arange(N))
        c, d = sy.sys_chain_off[[at, at + 1]]
        if what == "range":
            sy.T[c:d] = sy.D[c:d] = LIMIT
            sy.T[c] = sy.D[c] = 1 << 19
            sy.E[sy.chain_cb_off[c]:sy.chain_cb_off[d]] = LIMIT
        else:
            sy.D[c] = sy.T[c] + 1
        for call in (lambda: _host(sy, 250), lambda: _host(sy, 0), lambda: _noalloc(sy), lambda: gpu_analyze(sy)):
            with pytest.raises(pkg.PaamError) as e:
                call()
            assert e.value.code == code
