"""GPU tests of the path-A level kernels (matrices of at most 128 bytes, held
by 1, 2, 4 or 8 lanes): complete levels equal the oracle's at each width, word
type and an odd number of traces, deep enough that warps take many batches, and
an arena with exactly the room that the levels need is filled without loss."""
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


def _problem(props, traces, lo, hi, bits, seed=7):
    tb = W.draw_traces(W.Stream(W.stream_key(seed, 6)), traces, props, lo, hi, np.full(props, 0.5))
    return W.Problem("lanes", props, tb, traces // 2, traces - traces // 2, bits)


CASES = [
    (2, 3, 5, 32, 32, 9, 0x7F),     # one vector
    (2, 2, 20, 64, 64, 9, 0x5B),
    (3, 7, 6, 32, 32, 7, 0x7F),     # two vectors
    (2, 14, 6, 6, 32, 10, 0x5B),    # four vectors, the paper's grammar
    (3, 8, 8, 64, 64, 7, 0x7F),
    (4, 30, 8, 32, 32, 7, 0x7F),    # eight vectors
    (3, 15, 8, 64, 64, 7, 0x2D),    # not, or, X, G
    (1, 32, 1, 32, 32, 11, 0x7F),
]


@pytest.mark.parametrize("props,traces,lo,hi,bits,depth,ops", CASES)
def test_levels_equal_the_oracle(L, props, traces, lo, hi, bits, depth, ops):
    p = _problem(props, traces, lo, hi, bits)
    run = oracle.Spec.from_problem(p).enumerate(depth, ops)
    with L.Synthesizer(L.pack_problem(p), L.torch_config(op_mask=ops, cache_bytes=1 << 30, full_levels=True)) as s:
        for k in range(1, depth + 1):
            st = s.level(k)
            assert st.unique == run.size(k), k
            want = U.sorted_rows(U.oracle_level_words(run, k, p.traces.lengths, bits))
            assert np.array_equal(U.sorted_rows(s.export(k)), want), k


def _bytes_for(entries, row):
    """cache_bytes whose arena holds exactly `entries` rows (a table at most
    half full beside them, 16 bytes of records an entry)."""
    cap = 1024
    while cap // 2 < entries:
        cap *= 2
    return cap * 8 + entries * (row + 16)


@pytest.mark.parametrize("traces,bits,row,depth", [(4, 32, 16, 9), (14, 32, 64, 9), (30, 32, 128, 9)])
def test_arena_of_exactly_the_levels_size(L, traces, bits, row, depth):
    """As many entries as levels 1..depth hold: the last level is complete. One
    fewer: it is not, and says so."""
    p = L.pack_problem(_problem(2, traces, 6, 24, bits))
    with L.Synthesizer(p, L.torch_config(cache_bytes=1 << 30, full_levels=True)) as s:
        sizes = [s.level(k).unique for k in range(1, depth + 1)]
    total = sum(sizes)
    for room, full in ((total, 0), (total - 1, 1)):
        with L.Synthesizer(p, L.make_config(cache_bytes=_bytes_for(room, row), full_levels=True)) as s:
            got = [s.level(k) for k in range(1, depth + 1)]
        assert [st.unique for st in got[:-1]] == sizes[:-1]
        assert got[-1].cache_full == full and got[-1].unique == sizes[-1] - full


def test_large_level_with_little_room_or_log(L):
    """A level of millions of candidates, whose warps reserve ids ahead where
    they can: in an arena of exactly the entries it needs, and with a hole log
    of one entry, it is complete all the same."""
    p = L.pack_problem(_problem(2, 14, 6, 24, 32))
    depth = 11
    with L.Synthesizer(p, L.torch_config(cache_bytes=4 << 30, full_levels=True)) as s:
        stats = [s.level(k) for k in range(1, depth + 1)]
    sizes = [st.unique for st in stats]
    assert stats[-1].candidates > 1 << 21 and not stats[-1].cache_full
    for config in (L.make_config(cache_bytes=_bytes_for(sum(sizes), 64), full_levels=True),
                   L.torch_config(cache_bytes=4 << 30, full_levels=True, hole_cap=1)):
        with L.Synthesizer(p, config) as s:
            got = [s.level(k) for k in range(1, depth + 1)]
        assert [st.unique for st in got] == sizes and not got[-1].cache_full


@pytest.mark.parametrize("traces,bits", [(4, 32), (2, 64), (7, 32), (4, 64), (14, 32), (8, 64), (30, 32), (15, 64)])
def test_grammars_without_some_operators(L, traces, bits):
    """The launches with the paper's operators compiled in build the levels of
    its grammar and of parts of it (a fixed tile gives every level launches of
    its own)."""
    p = _problem(2, traces, 5, 30, bits, seed=11)
    for ops in (L.OPS_PAPER, L.OP_X | L.OP_U, L.OP_NOT | L.OP_AND, L.OPS_PAPER | L.OP_OR, L.OPS_PAPER | L.OP_G):
        run = oracle.Spec.from_problem(p).enumerate(7, ops)
        config = L.torch_config(op_mask=ops, cache_bytes=64 << 20, full_levels=True)
        config.tile_rows = 8
        with L.Synthesizer(L.pack_problem(p), config) as s:
            for k in range(1, 8):
                assert s.level(k).unique == run.size(k), (ops, k)
                if run.size(k):
                    want = U.sorted_rows(U.oracle_level_words(run, k, p.traces.lengths, bits))
                    assert np.array_equal(U.sorted_rows(s.export(k)), want), (ops, k)


def test_level_of_half_a_billion_candidates(L):
    """32-byte matrices: a level of 5 x 10^8 candidates, whose warps reserve ids
    ahead and lose claims to one another in every few batches, is complete and
    the same as without any reserved ahead (a hole log that is too small)."""
    p = L.pack_problem(_problem(2, 8, 8, 32, 32, seed=5))
    got = []
    for hole_cap in (0, 1):
        with L.Synthesizer(p, L.make_config(cache_bytes=40 << 30, full_levels=True, hole_cap=hole_cap)) as s:
            got.append([(st.candidates, st.unique, st.cache_full) for st in (s.level(k) for k in range(1, 16))])
    assert got[0] == got[1]
    assert got[0][-1][0] > 4 * 10 ** 8 and not got[0][-1][2]
