"""GPU tests of several contexts alive in one process: what a launch asks of the
device is its own context's, whatever the contexts before it and beside it
needed."""
from __future__ import annotations

import concurrent.futures

import numpy as np
import pytest

import oracle
from paper_2504_18943_gb300 import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    return U.lib()


def _noise(props, traces, lo, hi, bits, seed=5):
    tb = W.draw_traces(W.Stream(W.stream_key(seed, 9)), traces, props, lo, hi, np.full(props, 0.5))
    return W.Problem("contexts", props, tb, traces // 2, traces - traces // 2, bits)


@pytest.mark.parametrize("bits", [32, 64])
def test_contexts_of_unlike_matrices_in_turn(L, bits):
    """Contexts whose small levels need less and less shared memory a block
    (matrices of 32, 2 and 3 KiB and of 512 bytes; five and two words a trace),
    all alive: each is reset and solved in rotation, has the oracle's levels every
    time, and takes the launches for them that it took at first."""
    per = 64 // bits  # traces for the same width
    shapes = [(2, 4000 * per, 4, 12), (3, 250 * per, 8, 30), (2, 380 * per, 8, 30), (3, 60 * per, 8, 30),
              (2, 60 * per, 4 * bits, 5 * bits), (2, 60 * per, bits, 2 * bits)]
    depth = 4
    problems = [_noise(*s, bits) for s in shapes]
    runs = [oracle.Spec.from_problem(p).enumerate(depth, L.OPS_ALL) for p in problems]
    contexts = [L.Synthesizer(L.pack_problem(p), L.make_config(cache_bytes=256 << 20)) for p in problems]
    launches = [None] * len(contexts)
    try:
        for _ in range(2):
            for i, (s, p, run) in enumerate(zip(contexts, problems, runs)):
                s.reset()
                status, res, _, levels = s.solve(depth)
                assert status == L.LSYN_NOT_FOUND and res.levels_done == depth
                assert res.launches == (launches[i] or res.launches), i
                launches[i] = res.launches
                assert [lv.unique for lv in levels] == [run.size(k) for k in range(1, depth + 1)]
                want = U.sorted_rows(U.oracle_level_words(run, depth, p.traces.lengths, bits, U.planes_of(p)))
                assert np.array_equal(U.sorted_rows(s.export(depth)), want)
    finally:
        for s in contexts:
            s.close()


def test_threads_with_contexts_of_unlike_matrices(L):
    """A thread for each of twelve problems of unlike widths, with a context and a
    stream of its own: every solve of every thread succeeds, with the size that
    it has alone and a formula that separates its traces."""
    import torch
    problems = [W.tiny_problem(s, oracle.labeller) for s in range(4)]
    problems += [W.batched_problem(1000, i, oracle.labeller) for i in range(8)]
    specs = [oracle.Spec.from_problem(p) for p in problems]

    def solve(p, n):
        stream = torch.cuda.Stream()
        out = []
        with L.Synthesizer(L.pack_problem(p), L.make_config(cache_bytes=64 << 20, stream=stream.cuda_stream)) as s:
            for _ in range(n):
                s.reset()
                status, res, formula, _ = s.solve(7)
                out.append((status, res.size, formula))
        return out

    alone = [solve(p, 1)[0] for p in problems]
    with concurrent.futures.ThreadPoolExecutor(len(problems)) as pool:
        results = [f.result() for f in [pool.submit(solve, p, 60) for p in problems]]
    for spec, (status, size, _), out in zip(specs, alone, results):
        assert [o[:2] for o in out] == [(status, size)] * 60
        if status == L.LSYN_OK:
            assert all(spec.separates(f) for f in {o[2] for o in out})
