"""Host-side checks that need no GPU: the library loads, exports what the header declares,
and rejects bad arguments before touching CUDA."""
import ctypes as C

import numpy as np
import pytest

from paper_2601_16986_b200 import build as lib_build
from paper_2601_16986_b200 import declared_symbols, load_library
from paper_2601_16986_b200.binding import _Cfg


@pytest.fixture(scope="module")
def lib():
    lib_build.build()
    return load_library()


def test_every_declared_symbol_is_exported(lib):
    names = declared_symbols()
    assert {"crystalkv_create", "crystalkv_prefill", "crystalkv_decode_step", "crystalkv_rebudget",
            "crystalkv_get_retained"} <= set(names)
    for n in names:
        assert hasattr(lib, n), n


def good():
    return _Cfg(n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=128, batch=1, dtype=1, budget_per_head=64,
                min_budget=0, max_budget=0, max_answer_tokens=0, max_context=256, top_p=0.9, lam=0.6,
                sm_scale=0.0, mode=0, device=0)


@pytest.mark.parametrize("field,value", [("head_dim", 64), ("dtype", 7), ("n_layers", 0), ("n_q_heads", 7),
                                         ("n_q_heads", 32), ("mode", 3), ("max_context", 1),
                                         ("budget_per_head", 0), ("max_budget", 8), ("min_budget", 65),
                                         ("top_p", 1.5), ("lam", 1.2), ("device", -1), ("batch", 0)])
def test_create_rejects_bad_config_before_cuda(lib, field, value):
    c = good()
    setattr(c, field, value)
    h = C.c_void_p()
    assert lib.crystalkv_create(C.byref(c), C.byref(h)) == -1
    assert not h.value
    assert len(lib.crystalkv_last_error(None)) > 0


def test_null_arguments(lib):
    h = C.c_void_p()
    assert lib.crystalkv_create(None, C.byref(h)) == -1
    assert lib.crystalkv_create(C.byref(good()), None) == -1
    assert lib.crystalkv_destroy(None) == 0
    assert lib.crystalkv_set_stage(None, 0) == -1
    assert lib.crystalkv_rebudget(None, None) == -1
    assert lib.crystalkv_decode_step(None, 0, None, None, None, None, None) == -1
    assert lib.crystalkv_time(None, 0) == -1
    for code in (0, -1, -2, -3, -4, -5):
        assert lib.crystalkv_strerror(code)


def test_binding_refuses_to_run_without_a_gpu():
    import torch
    from paper_2601_16986_b200 import Config, CrystalKV, CrystalKVError
    if torch.cuda.is_available():
        pytest.skip("a GPU is present")
    with pytest.raises(CrystalKVError):
        CrystalKV(Config(n_layers=1, n_q_heads=2, n_kv_heads=1, batch=1, budget_per_head=8, max_context=32))


def _kept(lib, *ops):
    """(what each operation found, whether a set is kept at the end)"""
    arr = (C.c_int32 * (4 * len(ops)))(*[x for op in ops for x in (tuple(op) + (0, 0))[:4]])
    found = (C.c_int32 * len(ops))()
    return list(found) if (rc := lib.crystalkv_debug_kept_kit(arr, len(ops), found)) < 0 else (list(found), rc)


def test_what_a_closed_handle_leaves_outlives_its_context_only_in_name(lib):
    """The place that keeps one set per device: taken by the next handle of the same context; after a device reset (another id) the dead
    set neither serves a handle nor holds the place; a handle of a context that is not the primary one leaves and takes nothing."""
    CLOSE, MAKE = 0, 1
    assert _kept(lib, (CLOSE, 7, 7, 1), (MAKE, 7), (MAKE, 7)) == ([1, 1, 0], 0)
    assert _kept(lib, (CLOSE, 7, 7, 1), (CLOSE, 7, 7, 2), (MAKE, 7)) == ([1, 0, 1], 0)          # one at a time
    assert _kept(lib, (CLOSE, 7, 7, 1), (MAKE, 8), (CLOSE, 8, 8, 2), (MAKE, 8)) == ([1, 0, 1, 2], 0)
    assert _kept(lib, (CLOSE, 7, 7, 1), (CLOSE, 8, 8, 2), (MAKE, 8)) == ([1, 1, 2], 0)          # the new set takes the dead one's place
    assert _kept(lib, (CLOSE, 7, 7, 1), (MAKE, 8)) == ([1, 0], 0)                               # given back: nothing is kept any more
    assert _kept(lib, (CLOSE, 8, 7, 1)) == ([0], 0)                                             # made before the reset, closed after it
    assert _kept(lib, (CLOSE, 7, 7, 1), (MAKE, 0), (CLOSE, 0, 0, 2), (MAKE, 7)) == ([1, 0, 0, 1], 0)
    assert _kept(lib, (CLOSE, 7, 0, 1), (CLOSE, 0, 7, 1)) == ([0, 0], 0)
    assert lib.crystalkv_debug_kept_kit(None, 1, None) == -1 and _kept(lib, (2, 7)) == [0]


def test_trim_of_a_device_that_keeps_nothing_touches_none(lib):
    """No context is made for it: the call works where there is no GPU at all."""
    for device in (0, 1, 63):
        assert lib.crystalkv_trim(device) == 0
    assert lib.crystalkv_trim(-1) == -1 and lib.crystalkv_trim(64) == -1


def _place_runs_one_by_one(whole, runs):
    """Best fit, longest first, one run at a time: the placement the planner performs."""
    free = []            # free warps of every open CTA
    for s in range(7, 0, -1):
        for _ in range(runs[s]):
            fits = [c for c in free if c >= s]
            if fits:
                c = min(fits)
                free.remove(c)
            else:
                c = 8
            if c - s:
                free.append(c - s)
            if c == 8:
                whole += 1   # a CTA was opened
    return whole


def test_the_planners_count_equals_placing_the_runs_one_by_one(lib):
    """The launch planner counts the CTAs a placement needs by moving whole classes of CTAs at
    once; the placement itself goes run by run.  The two must agree for every mix of run lengths,
    or a plan could be chosen that then does not fit the grid."""
    import numpy as np
    rng = np.random.default_rng(7)
    cases = [[0] * 8, [0, 1, 0, 0, 0, 0, 0, 0], [0, 0, 0, 0, 0, 0, 0, 5], [0, 9, 0, 0, 0, 0, 0, 3],
             [0, 0, 4, 0, 0, 0, 2, 0], [0, 3, 3, 3, 3, 3, 3, 3]]
    for _ in range(400):
        top = int(rng.integers(1, 40))
        cases.append([0] + [int(x) for x in rng.integers(0, top, size=7)])
    for runs in cases:
        arr = (C.c_int32 * 8)(*runs)
        for whole in (0, 3):
            got = lib.crystalkv_debug_ctas_needed(whole, arr)
            assert got == _place_runs_one_by_one(whole, runs), (whole, runs, got)
    assert lib.crystalkv_debug_ctas_needed(0, None) == -1
    bad = (C.c_int32 * 8)(0, -1, 0, 0, 0, 0, 0, 0)
    assert lib.crystalkv_debug_ctas_needed(0, bad) == -1
    assert lib.crystalkv_debug_ctas_needed(-1, (C.c_int32 * 8)()) == -1


def test_placed_runs_are_spread_over_the_grid(lib):
    """Heads of one length: with more CTAs than the runs need, every CTA gets a run before one gets two (where ranges of like CTAs allow to say
    so in the planner's memory: always for runs of up to three lengths; heads of one length have one)."""
    rng = np.random.RandomState(11)
    where = np.zeros(1200, dtype=np.int32)
    for trial in range(2000):
        runs, grid, whole = [0] * 8, int(rng.randint(1, 149)), int(rng.randint(0, 5))
        for s in rng.choice(np.arange(1, 8), int(rng.randint(1, 4)), replace=False):
            runs[s] = int(rng.randint(0, 60))
        arr = (C.c_int32 * 8)(*runs)
        if lib.crystalkv_debug_ctas_needed(whole, arr) > grid or whole + sum(runs) == 0:
            continue
        got = lib.crystalkv_debug_spread_runs(whole, arr, grid, where.ctypes.data_as(C.c_void_p), len(where))
        assert got == sum(runs)
        ctas = set((where[:got] // 8).tolist())
        taken, at = np.zeros(8 * grid, dtype=np.int32), 0
        taken[:8 * whole] = 1
        for s in range(7, 0, -1):
            for _ in range(runs[s]):
                assert where[at] % 8 + s <= 8
                taken[where[at]:where[at] + s] += 1
                at += 1
        assert taken.max(initial=0) <= 1
        if whole + sum(runs) <= grid:
            assert len(ctas) == got


def test_placed_runs_fit_their_ctas_and_do_not_overlap(lib):
    """The planner's placement: every run sits inside one CTA, no two share a warp, none touches the CTAs taken
    whole, and it fits a grid exactly when the counting rule says so."""
    rng = np.random.RandomState(9)
    where = np.zeros(1200, dtype=np.int32)
    for trial in range(4000):
        runs = [0] + [int(x) for x in rng.randint(0, rng.choice([2, 8, 40]), 7) * (rng.rand(7) < 0.7)]
        whole = int(rng.randint(0, 5))
        arr = (C.c_int32 * 8)(*runs)
        need = lib.crystalkv_debug_ctas_needed(whole, arr)
        got = lib.crystalkv_debug_place_runs(whole, arr, need, where.ctypes.data_as(C.c_void_p), len(where))
        assert got == sum(runs)
        taken = np.zeros(8 * need, dtype=np.int32)
        taken[:8 * whole] = 1
        at = 0
        for s in range(7, 0, -1):
            for _ in range(runs[s]):
                w = where[at]
                assert 0 <= w and w % 8 + s <= 8
                taken[w:w + s] += 1
                at += 1
        assert taken.max(initial=0) <= 1
        # spread, too, whatever the mix: what does not fit that way falls back to the other walk
        assert lib.crystalkv_debug_spread_runs(whole, arr, need, where.ctypes.data_as(C.c_void_p), len(where)) == sum(runs)
        if need > 0:
            assert lib.crystalkv_debug_place_runs(whole, arr, need - 1, where.ctypes.data_as(C.c_void_p), len(where)) == -2
    assert lib.crystalkv_debug_place_runs(0, None, 1, where.ctypes.data_as(C.c_void_p), 1) == -1
