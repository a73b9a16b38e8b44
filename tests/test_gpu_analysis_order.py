"""Analyses of one batch on several streams share its lists and counters: each runs
after the one before it, whichever streams, outputs and options they were given."""
from __future__ import annotations

import pytest

import paam_gen as g
from gpu_util import ctx

pytestmark = pytest.mark.gpu

OPTS = [dict(n_buckets=1), dict(n_buckets=3, eps=1_000, kappa=500), dict(blocking_mode=1)]


def _outputs(sy):
    import torch

    return (torch.full((sy.n_chain,), -7, dtype=torch.int64, device="cuda"),
            torch.full((sy.n_chain,), 0xEE, dtype=torch.uint8, device="cuda"),
            torch.full((sy.n_sys,), 0xEE, dtype=torch.uint8, device="cuda"))


def _equal(got, want):
    import torch

    return all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("pattern", ["one key", "keys in turn", "each key twice", "each key three times"])
def test_streams_in_turn(pattern):
    import torch

    import paper_2404_06452_gb300 as pkg

    sy = g.generate("cfg3", n_sys=20_000, seed=11)  # systems of every width: all passes have work
    b = pkg.paam_rta_load_systems(ctx(), sy)
    want = []
    for o in OPTS:
        want.append(_outputs(sy))
        pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(**o), *want[-1])
    torch.cuda.synchronize()
    b.free()
    streams = [torch.cuda.Stream() for _ in range(3)]
    repeat = {"one key": 24, "keys in turn": 1, "each key twice": 2, "each key three times": 3}[pattern]
    for _ in range(3):
        b = pkg.paam_rta_load_systems(ctx(), sy)
        outs = [_outputs(sy) for _ in range(4)]
        torch.cuda.synchronize()
        last = {}
        for i in range(24):  # nothing waits on the host
            k = i // repeat
            last[k % 4] = k % 3
            pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(**OPTS[k % 3]), *outs[k % 4], stream=streams[i % 3])
        torch.cuda.synchronize()
        for at, o in last.items():
            assert _equal(outs[at], want[o]), (at, o)
        b.free()


def test_autotuning_follows_an_analysis_on_another_stream():
    import torch

    import paper_2404_06452_gb300 as pkg

    sy = g.generate("cfg3", n_sys=20_000, seed=12)
    b = pkg.paam_rta_load_systems(ctx(), sy)
    want, got = _outputs(sy), _outputs(sy)
    pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(), *want)
    torch.cuda.synchronize()
    for _ in range(3):
        pkg.paam_rta_analyze_batch(ctx(), b, pkg.analysis_opts(), *got, stream=torch.cuda.Stream())
        pkg.paam_rta_autotune(ctx(), b, pkg.analysis_opts(), stream=torch.cuda.Stream())
        assert _equal(got, want)
    b.free()
