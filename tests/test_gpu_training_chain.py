"""Gradients of minibatches of few tiles, of an odd number of them, and with whole
tiles that no label reaches, element by element against the network with its storage
in bf16 and exact sums.  A kernel's value and the reference differ by fp32
accumulation (at most 2^-11 of the sum of the products' magnitudes, as their number is
below 8,192) and by roundings to bf16 that fall the other way, in either operand of a
product: 2^-8 of it each, so 2^-7 of that sum even if all of them did.  (That bound needs many
rows: for a single row one rounding of a hidden activation shifts every product of a
unit alike, so a single row is compared bit for bit between positions instead.)"""
from __future__ import annotations

import numpy as np
import pytest

from gpu_util import ctx
from test_gpu_surrogate import _random_params, mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,labelled", [(128, 128), (384, 384), (640, 257), (2432, 2432)])
def test_gradients_of_few_tiles(rows, labelled):
    import torch

    import paper_2404_06452_gb300 as pkg

    p = _random_params(rows + labelled)
    m = pkg.Model.create(ctx(), 1)
    m.set_params(p)
    rng = np.random.default_rng(rows)
    X = torch.from_numpy(rng.uniform(0, 1.5, (rows, 1024)).astype(np.float32)).to(torch.bfloat16)
    L = rng.uniform(0, 2, (rows, 64)).astype(np.float32)
    L[rng.uniform(size=L.shape) < 0.3] = -1.0
    L[labelled:] = -1.0
    grads, loss = pkg.paam_surrogate_grad(ctx(), m, X.cuda(), torch.from_numpy(L).cuda())
    again, loss2 = pkg.paam_surrogate_grad(ctx(), m, X.cuda(), torch.from_numpy(L).cuda())
    assert np.array_equal(grads, again) and loss == loss2
    Xd = X.to(torch.float32).numpy().astype(np.float64)
    ref_loss, ref, scale = mlp.loss_and_grad_bf16(p.astype(np.float64), Xd, L)
    assert abs(loss - ref_loss) <= 1e-2 * ref_loss
    tol = (2.0 ** -11 + 2.0 ** -7) * scale + 1e-12
    bad = np.nonzero(np.abs(grads.astype(np.float64) - ref) > tol)[0]
    assert len(bad) == 0, (len(bad), bad[:5], grads[bad[:5]], ref[bad[:5]], tol[bad[:5]])
    m.free()


@pytest.mark.parametrize("row", [31, 127, 128, 300, 639])
def test_one_labelled_row_anywhere(row):
    """All other rows contribute exact zeros, so the place in the tile, the tile and the
    split of the rows change no bit of the gradients or of the loss."""
    import torch

    import paper_2404_06452_gb300 as pkg

    m = pkg.Model.create(ctx(), 1)
    m.set_params(_random_params(3))
    rng = np.random.default_rng(4)
    x = rng.uniform(0, 1.5, 1024).astype(np.float32)
    y = rng.uniform(0, 2, 64).astype(np.float32)

    def grad(rows, at):
        X = rng.uniform(0, 1.5, (rows, 1024)).astype(np.float32)
        L = np.full((rows, 64), -1.0, np.float32)
        X[at], L[at] = x, y
        return pkg.paam_surrogate_grad(ctx(), m, torch.from_numpy(X).to(torch.bfloat16).cuda(), torch.from_numpy(L).cuda())

    want, got = grad(128, 0), grad(640, row)
    assert np.count_nonzero(want[0]) > 400_000
    assert np.array_equal(want[0], got[0]) and want[1] == got[1]
    m.free()
