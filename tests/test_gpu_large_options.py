"""GPU parity of the larger systems (17 to 64 chains) with several accelerators
and under the safe blocking reading, at the edges of the kernels' widths: chain
counts around 16, 32 and 64, priorities past the slot tables, more segments than
a table holds, deadlines past the narrow bound, analysis and search, against the
CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paam_gen
from gpu_util import assert_same, ctx, gpu_analyze

pytestmark = pytest.mark.gpu

PARAMS = [dict(n_buckets=1, eps=0, kappa=0), dict(n_buckets=3, eps=391_000, kappa=129_180)]
SIZES = {"n16": (15, 18), "n32": (31, 34), "n64": (60, 64), "mixed": (1, 64)}


def _batch(lo, hi, acc=1, n_sys=150, **kw):
    cfg = dict(paam_gen.CONFIGS["cfg3"], n_geom_p=0.0, n_min=lo, n_max=hi, util_lo=0.03, util_hi=0.4, a_min=2_000,
               a_max=100_000, cb_max=5)
    cfg.update(kw)
    sy = paam_gen.generate(cfg, n_sys=n_sys, p_spin=0.3)
    return paam_gen.assign_accelerators(sy, acc) if acc > 1 else sy


@pytest.mark.parametrize("size", list(SIZES))
@pytest.mark.parametrize("acc", [1, 2, 3, 4])
def test_large_systems(size, acc):
    sy = _batch(*SIZES[size], acc=acc)
    far = paam_gen.Systems(**{**sy.__dict__, "prio": sy.prio * 1000 - 7, "exec_prio": None})
    seen = set()
    for p in PARAMS:
        for s in (sy, far):
            ref = oracle.analyze(s, threads=8, blocking_mode=1 if acc == 1 else 0, **p)
            assert_same(gpu_analyze(s, blocking_mode=1 if acc == 1 else 0, **p), ref)
            seen |= set(np.unique(ref["status"]))
    assert {0, 1} <= seen


def test_safe_reading_with_many_segments():
    """More segments than the 16-lane table (128) and the warp's (512) hold."""
    for lo, hi, cbs, per in ((8, 16, 12, 1), (14, 16, 30, 1), (40, 64, 12, 1), (60, 64, 20, 1)):
        sy = _batch(lo, hi, n_sys=60, cb_min=cbs, cb_max=cbs, p_acc=0.9, a_min=200, a_max=4_000, seg_per_cb=per)
        for p in PARAMS:
            assert_same(gpu_analyze(sy, blocking_mode=1, **p), oracle.analyze(sy, blocking_mode=1, threads=8, **p))


@pytest.mark.parametrize("acc", [1, 3])
def test_deadlines_past_the_narrow_bound(acc):
    sy = _batch(10, 40, acc=acc, t_min=5e7, t_max=4e8)
    mode = 1 if acc == 1 else 0
    for p in PARAMS:
        assert_same(gpu_analyze(sy, blocking_mode=mode, **p), oracle.analyze(sy, blocking_mode=mode, threads=8, **p))


@pytest.mark.parametrize("acc", [1, 2])
def test_search(acc):
    import torch

    import paper_2404_06452_gb300 as pkg

    sy = _batch(10, 40, acc=acc, n_sys=60)
    mode = 1 if acc == 1 else 0
    ranks = paam_gen.candidate_ranks(sy, 12, 3)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    for p in PARAMS:
        ref = oracle.search(sy, ranks, threads=8, blocking_mode=mode, **p)
        first, ok = pkg.search(ctx(), b, torch.from_numpy(ranks).cuda(), blocking_mode=mode, **p)
        assert np.array_equal(ok.cpu().numpy(), ref["cand_ok"])
        assert np.array_equal(first.cpu().numpy(), ref["first_ok"])
