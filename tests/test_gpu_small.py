"""GPU tests of small levels built several to a launch (lsyn_solve) and one to
a launch (lsyn_enumerate_level): the same complete levels either way and as the
oracle's, for every kind of matrix and for grammars without unary or without
binary operators; answers; a solve that is continued; an arena that fills; and
the way around it (a time limit takes the levels' own launches)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2504_18943_gb300 import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return U.lib()


def _noise(props, traces, lo, hi, bits, seed=3):
    tb = W.draw_traces(W.Stream(W.stream_key(seed, 8)), traces, props, lo, hi, np.full(props, 0.5))
    return W.Problem("small", props, tb, traces // 2, traces - traces // 2, bits)


SHAPES = [
    (2, 60, 8, 60, 64, 6),     # 512-byte matrices
    (3, 31, 8, 32, 32, 6),     # 128
    (2, 200, 8, 60, 64, 5),    # 2 KiB
    (2, 700, 8, 20, 64, 4),    # several warps to a matrix
    (2, 40, 60, 100, 32, 5),   # four words a trace
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ops", [0x7F, 0x5B, 0x46, 0x39])
def test_levels_of_a_solve(L, shape, ops):
    props, traces, lo, hi, bits, depth = shape
    p = _noise(props, traces, lo, hi, bits)
    packed = L.pack_problem(p)
    run = oracle.Spec.from_problem(p).enumerate(depth, ops)
    cfg = dict(op_mask=ops, cache_bytes=256 << 20)
    with L.Synthesizer(packed, L.make_config(**cfg)) as s:
        status, res, _, levels = s.solve(depth)
        assert status == L.LSYN_NOT_FOUND and res.levels_done == depth
        for k in range(1, depth + 1):
            assert levels[k - 1].unique == run.size(k) and s.count(k) == run.size(k), k
            if run.size(k):  # without unary operators the even levels are empty
                want = U.sorted_rows(U.oracle_level_words(run, k, p.traces.lengths, bits, U.planes_of(p)))
                assert np.array_equal(U.sorted_rows(s.export(k)), want), k
    with L.Synthesizer(packed, L.make_config(full_levels=True, time_limit_ms=1e9, **cfg)) as s:
        s.solve(depth)  # a time limit: the levels' own launches
        assert [s.count(k) for k in range(1, depth + 1)] == [run.size(k) for k in range(1, depth + 1)]
    with L.Synthesizer(packed, L.make_config(full_levels=True, **cfg)) as s:
        one = [s.level(k) for k in range(1, depth + 1)]
    for a, b in zip(one, levels):
        assert (a.level, a.candidates, a.unique, a.total) == (b.level, b.candidates, b.unique, b.total)


@pytest.mark.parametrize("seed", range(8))
def test_answers(L, seed):
    p = W.tiny_problem(seed, oracle.labeller)
    spec = oracle.Spec.from_problem(p)
    size = spec.solve(8)[0]
    with L.Synthesizer(L.pack_problem(p), L.make_config(cache_bytes=64 << 20)) as s:
        for _ in range(2):  # again after a reset
            status, res, formula, levels = s.solve(8)
            assert status == L.LSYN_OK and res.size == size and len(levels) == size
            assert spec.separates(formula) and W.formula_size(formula) == size
            s.reset()
        if size > 1:  # stopped below the answer, then continued
            assert s.solve(size - 1)[0] == L.LSYN_NOT_FOUND
            status, res, formula, _ = s.solve(8)
            assert status == L.LSYN_OK and res.size == size and spec.separates(formula)


@pytest.mark.parametrize("traces,bits,row", [(30, 32, 128), (60, 64, 512), (120, 64, 1024)])
def test_arena_fills_in_a_small_level(L, traces, bits, row):
    p = L.pack_problem(_noise(3, traces, 8, 30, bits))
    with L.Synthesizer(p, L.make_config(cache_bytes=64 << 20, full_levels=True)) as s:
        sizes = [s.level(k).unique for k in range(1, 6)]
    room = sum(sizes[:4]) + sizes[4] // 2
    cap = 1024
    while cap // 2 < room:
        cap *= 2
    with L.Synthesizer(p, L.make_config(cache_bytes=cap * 8 + room * (row + 16))) as s:
        status, res, _, levels = s.solve(6)
        assert status == L.LSYN_E_CACHE_FULL and res.levels_done == 5
        assert [lv.unique for lv in levels[:4]] == sizes[:4]
        assert levels[4].cache_full == 1 and levels[4].unique == room - sum(sizes[:4])


def test_threads_solve_small_problems_at_once(L):
    """Eight threads, each with a context and a stream of its own, solve at
    once: the launches whose blocks wait for one another do not wait for those
    of another launch, and every solve has the answer it has alone."""
    import threading
    import torch
    packed = [L.pack_problem(W.tiny_problem(s, oracle.labeller)) for s in range(4)]
    packed += [L.pack_problem(W.batched_problem(1000, i, oracle.labeller)) for i in range(4)]

    def solve(i, out, n):
        stream = torch.cuda.Stream()
        with L.Synthesizer(packed[i], L.make_config(cache_bytes=64 << 20, stream=stream.cuda_stream)) as s:
            for _ in range(n):
                s.reset()
                status, res, _, _ = s.solve(7)
                out[i].add((status, res.size))

    alone = [set() for _ in packed]
    for i in range(len(packed)):
        solve(i, alone, 1)
    out = [set() for _ in packed]
    threads = [threading.Thread(target=solve, args=(i, out, 100)) for i in range(len(packed))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert out == alone


@pytest.mark.parametrize("shape", [(3, 31, 8, 32, 32, 6), (2, 200, 8, 60, 64, 5)])
def test_timed_levels_have_their_time_and_launches(L, shape):
    """With timing on, every level of a solve has device time, whichever launch
    built it, and the levels' times and launches add up to the call's."""
    props, traces, lo, hi, bits, depth = shape
    packed = L.pack_problem(_noise(props, traces, lo, hi, bits))
    with L.Synthesizer(packed, L.make_config(cache_bytes=256 << 20, timing=True)) as s:
        s.solve(depth)
        s.reset()
        status, res, _, levels = s.solve(depth)
        assert status == L.LSYN_NOT_FOUND and len(levels) == depth
        for lv in levels:
            assert 0 < sum(lv.kernel_ms) and 0 < lv.ms
        assert sum(sum(lv.kernel_ms) for lv in levels) <= sum(lv.ms for lv in levels) <= res.ms
        assert sum(lv.launches for lv in levels) == res.launches >= 1
