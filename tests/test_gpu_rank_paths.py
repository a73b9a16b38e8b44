"""The candidate ranking's variants: the pick of the best scores with the scores in
registers (up to 256 candidates) and in memory, and candidate features under one bucket
and several, for 16- and 32-lane segments; scores of systems of up to 16 chains, whose layers run
in one kernel, against the kernels per layer."""
from __future__ import annotations

import numpy as np
import pytest

import paam_gen as g
from gpu_util import ctx
from test_gpu_surrogate import _features, _random_params, ofeat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 31, 33, 255, 256, 257, 300])
@pytest.mark.parametrize("pinned", [0, 3])
def test_picks_are_a_stable_sort(K, pinned):
    """Duplicated orders give equal scores, which go by index."""
    import torch

    import paper_2404_06452_gb300 as pkg

    m = pkg.Model.create(ctx(), 1)
    m.set_params(_random_params(2))
    sy = g.generate("cfg4s", n_sys=9, seed=K)
    ranks = g.candidate_ranks(sy, K, 5)
    ranks[:, K // 2:] = ranks[:, :K - K // 2]
    pinned, top = min(pinned, K), min(K, 40)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    ranked = torch.empty((sy.n_sys, top), dtype=torch.int32, device="cuda")
    scores = torch.empty((sy.n_sys, K), dtype=torch.float32, device="cuda")
    pkg.paam_surrogate_infer(ctx(), m, b, torch.from_numpy(ranks).cuda(), top, ranked, scores, n_pinned=pinned)
    torch.cuda.synchronize()
    key = scores.cpu().numpy()
    key[:, :pinned] = -np.inf
    assert np.array_equal(ranked.cpu().numpy(), np.argsort(key, axis=1, kind="stable")[:, :top])
    b.free()
    m.free()


@pytest.mark.parametrize("n_buckets,kappa", [(1, 0), (1, 20_000), (4, 0)])
@pytest.mark.parametrize("n_max", [1, 2, 16, 17, 32])
def test_candidate_features_by_buckets(n_buckets, kappa, n_max):
    sy = g.generate("cfg3", n_sys=30, seed=7, n_min=1, n_max=n_max)
    ranks = g.candidate_ranks(sy, 9, 5)
    got = _features(sy, ranks, n_buckets=n_buckets, kappa=kappa)
    ref = ofeat.features(sy, ranks, n_buckets=n_buckets, kappa=kappa)
    assert np.all(np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 2e-3)
    assert np.all(got[ref == 0] == 0)


@pytest.mark.parametrize("K", [1, 7, 300])
@pytest.mark.parametrize("n_max", [1, 4, 5, 9, 16])
def test_scores_of_small_systems(n_max, K):
    """One system of more than 16 chains in the batch takes all of it to the kernels per
    layer; the sums and their order are the same, so are the bits."""
    import torch

    import paper_2404_06452_gb300 as pkg

    m = pkg.Model.create(ctx(), 1)
    m.set_params(_random_params(n_max))
    sy = g.generate("cfg3", n_sys=600, seed=11, n_min=1, n_max=24)
    n = sy.chains_per_system()
    small, big = np.nonzero(n <= n_max)[0], np.nonzero(n > 16)[0]
    assert len(small) > 5 and n[small].max() == n_max
    both = sy.subset(np.r_[small, big[:1]])
    ranks = g.candidate_ranks(both, K, 3)
    got = []
    for part, r in ((sy.subset(small), ranks[:-1, :, :n_max].copy()), (both, ranks)):
        b = pkg.paam_rta_load_systems(ctx(), part)
        scores = torch.empty((part.n_sys, K), dtype=torch.float32, device="cuda")
        ranked = torch.empty((part.n_sys, 1), dtype=torch.int32, device="cuda")
        pkg.paam_surrogate_infer(ctx(), m, b, torch.from_numpy(r).cuda(), 1, ranked, scores)
        torch.cuda.synchronize()
        got.append(scores.cpu().numpy())
        b.free()
    assert np.array_equal(got[0], got[1][:-1]) and np.all(np.isfinite(got[0]))
    assert n_max == 1 or got[0].any()  # one chain: the only output may be negative throughout, its score 0
    m.free()
