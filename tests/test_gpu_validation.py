"""GPU parity of the input validation: batches with one entry made invalid are
refused with the documented code wherever the entry lies (systems smaller and
larger than a validation group, the first, a middle and the last one), values
on the limits are accepted, and the untouched batches load."""
from __future__ import annotations

import dataclasses

import numpy as np
import pytest

import paam_gen
from gpu_util import analyze_poisoned, assert_same, ctx

pytestmark = pytest.mark.gpu

INVAL, RANGE = -1, -2
LIMIT = 1 << 40

# mean chain counts on each side of the group widths' lines, and sizes around the widths
SHAPES = {
    "n1": dict(n_min=1, n_max=1, cb_min=1, cb_max=1),
    "n4": dict(n_min=3, n_max=5, cb_min=1, cb_max=4),
    "n8": dict(n_min=5, n_max=9, cb_min=1, cb_max=4, x_min=9, x_max=9),
    "n16": dict(n_min=8, n_max=17, cb_min=1, cb_max=3, x_min=1, x_max=5),
    "n64": dict(n_min=2, n_max=64, n_geom_p=1.0 / 9.0, cb_min=1, cb_max=12, x_min=2, x_max=40),
}


def _batch(shape, n_sys=67):
    cfg = dict(paam_gen.CONFIGS["cfg3"], n_geom_p=0.0)
    cfg.update(SHAPES[shape])
    return paam_gen.generate(cfg, n_sys=n_sys, p_acc=0.9, p_spin=0.3)


def _copy(sy):
    return dataclasses.replace(sy, **{f.name: getattr(sy, f.name).copy() for f in dataclasses.fields(sy)
                                      if isinstance(getattr(sy, f.name), np.ndarray)})


def _code(sy):
    import paper_2404_06452_gb300 as pkg

    try:
        pkg.paam_rta_load_systems(ctx(), sy).free()
    except pkg.PaamError as e:
        return e.code
    return 0


def _put(field, value):
    def f(sy, s, rng):
        a = getattr(sy, field)
        if field in ("E", "A", "acc"):
            c = sy.chain_cb_off[sy.sys_chain_off[[s, s + 1]]]
            lo, hi = (c if field == "E" else sy.cb_seg_off[c])
        elif field == "exec_core":
            lo, hi = sy.sys_exec_off[[s, s + 1]]
        else:
            lo, hi = sy.sys_chain_off[[s, s + 1]]
        if hi <= lo:
            return False
        a[rng.integers(lo, hi)] = value
        return True

    return f


def _deadline_past_period(sy, s, rng):
    c = int(rng.integers(*sy.sys_chain_off[[s, s + 1]]))
    sy.D[c] = sy.T[c] + 1
    return True


def _no_such_executor(sy, s, rng):
    c = int(rng.integers(*sy.sys_chain_off[[s, s + 1]]))
    sy.exec[c] = sy.sys_exec_off[s + 1] - sy.sys_exec_off[s]
    return True


def _same_priority(sy, s, rng):
    lo, hi = sy.sys_chain_off[[s, s + 1]]
    if hi - lo < 2:
        return False
    a, b = rng.choice(np.arange(lo, hi), 2, replace=False)
    sy.prio[a] = sy.prio[b]
    return True


def _same_executor_priority(sy, s, rng):
    lo, hi = sy.sys_exec_off[[s, s + 1]]
    if hi - lo < 2:
        return False
    a, b = rng.choice(np.arange(lo, hi), 2, replace=False)
    sy.exec_core[a] = sy.exec_core[b]
    sy.exec_prio[a] = sy.exec_prio[b]
    return True


def _falling(field, bounds):
    def f(sy, s, rng):
        a = getattr(sy, field)
        lo, hi = bounds(sy, s)
        k = np.arange(lo + 1, hi)
        k = k[a[k + 1] > a[k]]  # past its successor: no longer rising
        if len(k) == 0:
            return False
        i = rng.choice(k)
        a[i] = a[i + 1] + 1
        return True

    return f


def _chains(sy, s):
    return sy.sys_chain_off[s], sy.sys_chain_off[s + 1]


def _callbacks(sy, s):
    c = sy.sys_chain_off[[s, s + 1]]
    return sy.chain_cb_off[c[0]], sy.chain_cb_off[c[1]]


def _range_of_sums(sy, s, rng):
    c = int(rng.integers(*sy.sys_chain_off[[s, s + 1]]))
    sy.T[c] = sy.D[c] = LIMIT  # one long deadline over a 1 ns period
    lo = sy.sys_chain_off[s]
    if sy.sys_chain_off[s + 1] - lo < 2:
        return False
    o = lo if c != lo else lo + 1
    sy.T[o] = sy.D[o] = 1
    return True


FAULTS = {
    "T0": (_put("T", 0), INVAL), "T_neg": (_put("T", -5), INVAL), "D0": (_put("D", 0), INVAL),
    "D_above_T": (_deadline_past_period, INVAL), "spin2": (_put("spin", 2), INVAL), "exec_neg": (_put("exec", -1), INVAL),
    "exec_past": (_no_such_executor, INVAL), "prio_twice": (_same_priority, INVAL),
    "exec_prio_twice": (_same_executor_priority, INVAL), "core_neg": (_put("exec_core", -1), INVAL),
    "E_neg": (_put("E", -1), INVAL), "E_above": (_put("E", LIMIT + 1), INVAL), "A_neg": (_put("A", -1), INVAL),
    "A_above": (_put("A", LIMIT + 1), INVAL), "acc_past": (_put("acc", 4), INVAL), "acc_neg": (_put("acc", -1), INVAL),
    "cb_off_falls": (_falling("chain_cb_off", _chains), INVAL),
    "seg_off_falls": (_falling("cb_seg_off", _callbacks), INVAL), "range": (_range_of_sums, RANGE),
}


@pytest.mark.parametrize("shape", list(SHAPES))
def test_one_bad_entry_is_refused(shape):
    base = _batch(shape)
    assert _code(base) == 0
    rng = np.random.default_rng(7)
    for name, (fault, code) in FAULTS.items():
        for s in (0, 33, 66):
            sy = _copy(base)
            if fault(sy, s, rng):
                assert _code(sy) == code, (name, s)


def test_structure_and_sentinels():
    base = _batch("n64")
    for field in ("sys_chain_off", "chain_cb_off", "cb_seg_off", "sys_exec_off"):
        for i, d in ((0, 1), (-1, -1), (-1, 1)):
            sy = _copy(base)
            getattr(sy, field)[i] += d
            assert _code(sy) == INVAL, (field, i, d)
    # a system of 65 chains; chains without an executor
    cfg = dict(paam_gen.CONFIGS["cfg3"], n_geom_p=0.0, n_min=33, n_max=33, cb_min=1, cb_max=1)
    two = paam_gen.generate(cfg, n_sys=2)
    sy = _copy(two)
    sy.sys_chain_off[1] = 1
    sy.prio[1:] = np.arange(65)
    sy.exec[1:] = 0
    assert _code(sy) == INVAL
    sy = _copy(two)
    sy.sys_exec_off[1] = sy.sys_exec_off[2]
    assert _code(sy) == INVAL


def test_values_on_the_limits():
    """The largest values accepted, and sums whose quick test is not clear, are decided as in 64 bits."""
    import oracle

    cfg = dict(paam_gen.CONFIGS["cfg3"], n_geom_p=0.0, n_min=2, n_max=2, cb_min=1, cb_max=1, x_min=1, x_max=1)
    base = paam_gen.generate(cfg, n_sys=3, p_acc=1.0)
    sy = _copy(base)
    sy.T[:] = sy.D[:] = LIMIT
    sy.E[:] = LIMIT
    sy.A[:] = LIMIT
    assert _code(sy) == 0
    # iteration bound: D / T + ceil(D / 1) + 2 evaluations against 2^20
    for d, code in (((1 << 20) - 3, 0), ((1 << 20) - 2, RANGE)):
        sy = _copy(base)
        sy.T[2], sy.D[2] = d, d
        sy.T[3] = sy.D[3] = 1
        assert _code(sy) == code, d
    # magnitude: n (ceil(Dmax / Tmin) + 1) Cmax against 2^61.  With n = 2 and Cmax = 2^41 + 2^33 + A
    # it is 1.004 x 2^61 x 2^21 / t for a shortest period of t
    for t, code in ((1 << 23, 0), (1 << 22, 0), (1 << 21, RANGE), ((1 << 20) + (1 << 17), RANGE)):
        sy = _copy(base)
        sy.T[:] = sy.D[:] = LIMIT
        sy.T[3] = sy.D[3] = t
        sy.E[:] = LIMIT
        assert _code(sy) == code, t
    b = __import__("paper_2404_06452_gb300").paam_rta_load_systems(ctx(), base)
    assert_same(analyze_poisoned(ctx(), b), oracle.analyze(base))
