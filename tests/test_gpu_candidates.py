"""GPU parity of the candidate verdicts (the search) and of the Audsley-style
seed at the edges of their group widths, with shared and unshared executors and
cores, busy-waiting chains, several buckets and both blocking readings' options
left to the other kernels, against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paam_gen
from gpu_util import ctx

pytestmark = pytest.mark.gpu

PARAMS = [dict(n_buckets=1, eps=0, kappa=0), dict(n_buckets=2, eps=391_000, kappa=129_180),
          dict(n_buckets=5, eps=3, kappa=1), dict(n_buckets=100, eps=50_000, kappa=0)]
# chains (both sides of 16, 32), executors, executors per core, total utilisation, segments
SHAPES = {
    "one": dict(n_min=1, n_max=2, x_min=1, x_max=2),
    "apart16": dict(n_min=13, n_max=16, x_min=16, x_max=16, exec_per_core=1),
    "paired16": dict(n_min=15, n_max=17, x_min=8, x_max=16, exec_per_core=3),
    "few17": dict(n_min=16, n_max=18, x_min=2, x_max=4, exec_per_core=4, a_min=2_000, a_max=40_000),
    "apart32": dict(n_min=29, n_max=33, x_min=32, x_max=32, exec_per_core=1, a_min=10_000, a_max=300_000),
    "paired32": dict(n_min=31, n_max=33, x_min=10, x_max=20, exec_per_core=2, a_min=2_000, a_max=40_000),
}


def _batch(shape, n_sys, util, seed=5):
    cfg = dict(paam_gen.CONFIGS["cfg4s"], n_geom_p=0.0, util_lo=util, util_hi=util, seed=seed)
    cfg.update(SHAPES[shape])
    return paam_gen.generate(cfg, n_sys=n_sys, p_spin=0.4, cb_min=1, cb_max=5, p_acc=0.5)


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("util", [0.04, 0.4])
def test_search_verdicts(shape, util):
    import torch

    import paper_2404_06452_gb300 as pkg

    sy = _batch(shape, 60, util)
    ranks = paam_gen.candidate_ranks(sy, 24, 11)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    dev = torch.from_numpy(ranks).cuda()
    seen = set()
    for p in PARAMS:
        ref = oracle.search(sy, ranks, threads=8, **p)
        first, ok = pkg.search(ctx(), b, dev, **p)
        assert np.array_equal(ok.cpu().numpy(), ref["cand_ok"]), p
        assert np.array_equal(first.cpu().numpy(), ref["first_ok"]), p
        first, _ = pkg.search(ctx(), b, dev, stop_at_first=True, want_cand_ok=False, **p)
        assert np.array_equal(first.cpu().numpy(), ref["first_ok"]), p
        seen |= set(np.unique(ref["cand_ok"]))
    if util < 0.1:
        assert seen == {0, 1}  # both verdicts occur


@pytest.mark.parametrize("shape", list(SHAPES))
def test_seed_order(shape):
    import paper_2404_06452_gb300 as pkg

    for p in PARAMS[:3]:
        sy = _batch(shape, 40, 0.3)
        nmax = int(sy.chains_per_system().max()) + 1
        b = pkg.paam_rta_load_systems(ctx(), sy)
        got = pkg.audsley_order(ctx(), b, nmax, **p).cpu().numpy()
        assert np.array_equal(got, oracle.audsley(sy, nmax=nmax, threads=8, **p)), p


@pytest.mark.parametrize("n_sys", [608, 609, 4865])
def test_seed_order_batch_sizes(n_sys):
    """Each number of groups per system."""
    import paper_2404_06452_gb300 as pkg

    cfg = dict(paam_gen.CONFIGS["cfg4s"], n_min=2, n_max=9, x_min=2, x_max=9, exec_per_core=2)
    sy = paam_gen.generate(cfg, n_sys=n_sys)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    got = pkg.audsley_order(ctx(), b, 9, n_buckets=2).cpu().numpy()
    assert np.array_equal(got, oracle.audsley(sy, nmax=9, n_buckets=2, threads=8))


def test_short_periods_take_the_joint_evaluation_past_its_limit():
    """Recurrences of thousands of steps (one short period): more than the joint
    evaluation takes, so the chains are taken one by one from where it stopped."""
    import torch

    import paper_2404_06452_gb300 as pkg

    cfg = dict(paam_gen.CONFIGS["cfg4s"], n_min=4, n_max=6, x_min=3, x_max=6, exec_per_core=2, util_lo=0.3, util_hi=0.3)
    sy = paam_gen.generate(cfg, n_sys=40, p_acc=0.0)
    first = sy.sys_chain_off[:-1]
    sy.T[first] = sy.D[first] = 10_000
    for c in first:
        sy.E[sy.chain_cb_off[c]:sy.chain_cb_off[c + 1]] = 0
        sy.E[sy.chain_cb_off[c]] = 9_950
    ranks = paam_gen.candidate_ranks(sy, 16, 3)
    ref = oracle.search(sy, ranks, threads=8)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    _, ok = pkg.search(ctx(), b, torch.from_numpy(ranks).cuda())
    assert np.array_equal(ok.cpu().numpy(), ref["cand_ok"])
