"""The training's minibatch order and labels on the GPU: with a vanishing learning
rate the loss of each epoch is the mean over its minibatches of their masked mean
squared errors, and a last minibatch of few systems shows which systems it holds."""
from __future__ import annotations

import numpy as np
import pytest

import paam_gen
from gpu_util import ctx

pytestmark = pytest.mark.gpu

MASK = (1 << 64) - 1


def _shuffles(n, seed, epochs):
    """Fisher-Yates from n - 1 down to 1 on one splitmix64 stream."""
    x = seed ^ 0x5DEECE66D
    out = []
    for _ in range(epochs):
        p = list(range(n))
        for i in range(n - 1, 0, -1):
            x = (x + 0x9E3779B97F4A7C15) & MASK
            z = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & MASK
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK
            z ^= z >> 31
            j = int((((z >> 11) * 2.0 ** -52 - 1.0) * 0.5 + 0.5) * float(i + 1)) % (i + 1)
            p[i], p[j] = p[j], p[i]
        out.append(np.array(p))
    return out


@pytest.mark.parametrize("shape", ["cfg2", "cfg3"])
@pytest.mark.parametrize("n", [1, 2, 129, 131, 1025, 5000])
def test_epoch_losses_follow_the_seeded_order(shape, n):
    import torch

    import paper_2404_06452_gb300 as pkg

    epochs, rows, seed = 3, 128, 77 + n
    sy = paam_gen.generate(shape, n_sys=n)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    R, st, _ = pkg.analyze(ctx(), b)
    from paper_2404_06452_gb300 import _binding as B

    model = B.Model.create(ctx(), 3)
    pred = torch.empty((n, 64), dtype=torch.float32, device="cuda")
    B.paam_surrogate_predict(ctx(), model, b, pred)
    loss = np.zeros(epochs, np.float32)
    B.paam_surrogate_train(ctx(), b, R, st, B.train_opts(epochs=epochs, batch_rows=rows, lr=1e-30, weight_decay=0.0,
                                                         seed=seed, epoch_loss=loss), model)
    torch.cuda.synchronize()
    R, st, P = R.cpu().numpy(), st.cpu().numpy(), pred.cpu().numpy().astype(np.float64)
    cnt = sy.chains_per_system()
    err = np.zeros(n)
    for s in range(n):
        c0, c1 = sy.sys_chain_off[s], sy.sys_chain_off[s + 1]
        y = np.where(st[c0:c1] == 0, np.minimum(R[c0:c1] / sy.D[c0:c1], 2.0), 2.0)
        err[s] = ((P[s, :c1 - c0] - y) ** 2).sum()
    for e, p in enumerate(_shuffles(n, seed, epochs)):
        ref = np.mean([err[p[k:k + rows]].sum() / cnt[p[k:k + rows]].sum() for k in range(0, n, rows)])
        # the same network in another tile shape: fp32 sums of bf16 products, below 1e-3
        assert abs(loss[e] - ref) <= 1e-3 * ref, (e, loss[e], ref)
