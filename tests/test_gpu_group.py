"""GPU tests of the group kernels (matrices above 512 bytes, several words per
trace among them): complete levels equal the oracle's over the layouts at
which the work is cut differently - one or several warps to a matrix, columns
that do not divide among the threads, several planes, items of several rows -
and for a grammar with some operators switched off."""
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


def _problem(props, traces, lo, hi, bits, seed=11):
    tb = W.draw_traces(W.Stream(W.stream_key(seed, 5)), traces, props, lo, hi, np.full(props, 0.5))
    return W.Problem("group", props, tb, traces // 2, traces - traces // 2, bits)


@pytest.mark.parametrize("props,traces,lo,hi,bits,depth,ops", [
    (3, 65, 8, 64, 64, 5, 0x7F),      # 64 vectors: the narrowest
    (3, 129, 8, 32, 32, 5, 0x7F),
    (2, 191, 8, 64, 64, 5, 0x7F),     # 96 vectors: three columns a thread
    (2, 257, 8, 40, 64, 5, 0x5B),     # 160 vectors, the paper's grammar
    (2, 520, 8, 20, 64, 5, 0x7F),     # 288 vectors: columns that do not divide among the threads
    (2, 1030, 4, 16, 64, 4, 0x7F),    # 544 vectors: three warps or more, two groups a block
    (2, 4000, 4, 12, 64, 4, 0x66),    # 2000 vectors: eight warps; and, or, G, U only
    (2, 70, 30, 64, 32, 5, 0x7F),     # two words a trace
    (2, 1100, 60, 90, 64, 3, 0x7F),   # two words, wide planes
    (2, 33, 100, 160, 32, 4, 0x7F),   # five words
    (2, 9, 300, 512, 32, 4, 0x7F),    # sixteen words
])
def test_levels_equal_the_oracle(L, props, traces, lo, hi, bits, depth, ops):
    U.assert_levels_match(L, _problem(props, traces, lo, hi, bits), depth, op_mask=ops, cache_bytes=512 << 20)


@pytest.mark.parametrize("traces,hi,bits", [(65, 12, 64), (40, 40, 32)])
def test_large_level_equals_the_oracle(L, traces, hi, bits):
    """Deep enough that an item takes several rows and a level pairs with
    itself (levels 5 and 7), one word and two words per trace."""
    p = _problem(3, traces, 8, hi, bits)
    depth = 8
    run = oracle.Spec.from_problem(p).enumerate(depth, 0x7F)
    with L.Synthesizer(L.pack_problem(p), L.torch_config(cache_bytes=4 << 30, full_levels=True)) as s:
        for k in range(1, depth + 1):
            st = s.level(k)
            assert st.unique == run.size(k), k
            want = U.sorted_rows(U.oracle_level_words(run, k, p.traces.lengths, bits, U.planes_of(p)))
            got = U.sorted_rows(s.export(k))
            assert np.array_equal(got, want), k
