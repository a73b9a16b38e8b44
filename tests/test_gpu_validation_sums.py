"""GPU validation of systems so large that 64-bit sums of their execution times
could wrap: the sums are decided as in the documented bound."""
from __future__ import annotations

import types

import pytest

from gpu_util import ctx

pytestmark = pytest.mark.gpu

LIMIT = 1 << 40
PERIOD = 1 << 31  # below 2^32 ns: nothing else takes these systems to the test per chain


def _load(per_chain, chains, wcet):
    import torch

    import paper_2404_06452_gb300 as pkg

    def i64(v):
        return torch.tensor(v, dtype=torch.int64, device="cuda")

    n_cb = per_chain * chains
    sy = types.SimpleNamespace(
        sys_chain_off=i64([0, chains]), chain_cb_off=i64([per_chain * c for c in range(chains + 1)]),
        cb_seg_off=torch.zeros(n_cb + 1, dtype=torch.int64, device="cuda"), T=i64([PERIOD] * chains),
        D=i64([PERIOD] * chains), prio=torch.arange(chains, dtype=torch.int32, device="cuda"),
        exec=torch.zeros(chains, dtype=torch.int32, device="cuda"),
        spin=torch.zeros(chains, dtype=torch.uint8, device="cuda"),
        E=torch.full((n_cb,), wcet, dtype=torch.int64, device="cuda"), A=i64([]), acc=None, sys_exec_off=i64([0, 1]),
        exec_core=torch.zeros(1, dtype=torch.int32, device="cuda"),
        exec_prio=torch.zeros(1, dtype=torch.int32, device="cuda"))
    try:
        pkg.paam_rta_load_systems(ctx(), sy).free()
    except pkg.PaamError as e:
        return e.code
    return 0


def test_sums_of_execution_times_that_wrap():
    """2^26 callbacks of 2^40 ns are 2^66: each of four partial sums is 2^64, zero in 64 bits."""
    assert _load(1 << 21, 32, LIMIT) == -2
    assert _load(1 << 15, 64, LIMIT) == -2  # 2^59 per partial sum; 64 chains x 2 arrivals x 2^55: past the bound
    assert _load(1 << 15, 64, 1 << 8) == 0  # as many callbacks inside the bound
