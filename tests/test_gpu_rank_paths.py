"""The candidate ranking's variants: the pick of the best scores with the scores in
registers (up to 256 candidates) and in memory, and candidate features under one bucket
and several, for 16- and 32-lane segments."""
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
