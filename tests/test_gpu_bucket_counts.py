"""More worker buckets than a system has accelerator users, up to the largest
number the options hold: every user then has a bucket of its own (R2), in the
analysis of every size of system, option and launch configuration, in the search
and in the seed, against the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paam_gen

# around the largest system, where rank * buckets passes 2^32 for 64 chains, and the largest
BUCKETS = [63, 64, 65, 68_174_085, (1 << 31) - 1]


def test_partition_by_as_many_buckets_as_a_system_can_hold():
    """rank * n / |U| puts the same users together for n and min(n, 64)."""
    r = np.arange(64, dtype=np.int64)
    for users in range(1, 65):
        for n in [*range(1, 131), *BUCKETS]:
            a, b = r[:users] * n // users, r[:users] * min(n, 64) // users
            assert np.array_equal(a[:, None] == a, b[:, None] == b), (users, n)


def _batch(lo, hi, acc=1, mode=0, n_sys=120):
    # light chains with long segments, so that the same bucket's blocking decides; the safe
    # reading counts segments into the CPU blocking too and needs them shorter
    cfg = dict(paam_gen.CONFIGS["cfg3"], n_geom_p=0.0, n_min=lo, n_max=hi, util_lo=0.02, util_hi=0.2, cb_max=2,
               a_min=50_000 if mode == 0 else 20_000, a_max=1_500_000 if mode == 0 else 300_000, p_acc=0.8, x_min=8, x_max=8)
    sy = paam_gen.generate(cfg, n_sys=n_sys, p_spin=0.2)
    return paam_gen.assign_accelerators(sy, acc) if acc > 1 else sy


SIZES = [(3, 16), (17, 32), (33, 64)]


@pytest.mark.gpu
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("acc,mode", [(1, 0), (1, 1), (2, 0), (4, 0), (2, 1)])
def test_analysis(size, acc, mode):
    from gpu_util import assert_same, gpu_analyze

    sy = _batch(*size, acc=acc, mode=mode)
    for n in BUCKETS:
        assert_same(gpu_analyze(sy, n_buckets=n, blocking_mode=mode),
                    oracle.analyze(sy, n_buckets=n, blocking_mode=mode, threads=8))


@pytest.mark.gpu
def test_every_launch_configuration():
    import paper_2404_06452_gb300 as pkg
    from gpu_util import analyze_poisoned, assert_same, ctx

    sy = _batch(2, 64)
    n = BUCKETS[-1]
    ref = oracle.analyze(sy, n_buckets=n, threads=8)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    for cfg in range(pkg.paam_rta_num_launch_configs()):
        pkg.paam_rta_set_launch_config(b, cfg)
        assert_same(analyze_poisoned(ctx(), b, n_buckets=n), ref)
    b.free()


@pytest.mark.gpu
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("acc,mode", [(1, 0), (1, 1), (3, 0)])
def test_search_and_seed(size, acc, mode):
    import torch

    import paper_2404_06452_gb300 as pkg
    from gpu_util import ctx

    sy = _batch(*size, acc=acc, mode=mode, n_sys=40)
    ranks = paam_gen.candidate_ranks(sy, 10, 5)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    for n in BUCKETS[-2:]:
        ref = oracle.search(sy, ranks, n_buckets=n, blocking_mode=mode, threads=8)
        first, ok = pkg.search(ctx(), b, torch.from_numpy(ranks).cuda(), n_buckets=n, blocking_mode=mode)
        assert np.array_equal(ok.cpu().numpy(), ref["cand_ok"])
        assert np.array_equal(first.cpu().numpy(), ref["first_ok"])
    nmax = int(sy.chains_per_system().max())
    seed = pkg.audsley_order(ctx(), b, nmax, n_buckets=BUCKETS[-1], blocking_mode=mode)
    assert np.array_equal(seed.cpu().numpy(), oracle.audsley(sy, nmax, n_buckets=BUCKETS[-1], blocking_mode=mode))
    b.free()
