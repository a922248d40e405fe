"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public entry points (``paper_2504_18943_gb300.lsyn``,
the binding of ``include/lsyn.h``) and comes in one of these kinds:

  label     lsyn_eval_noalloc: a learnt formula applied to traces on the device
  evaluate  lsyn_eval: a formula over a data set in host memory
  solve     lsyn_reset + lsyn_solve on a kept context, traces labelled by a
            hidden formula: the answer comes after a few small levels
  new       lsyn_create + lsyn_solve + lsyn_destroy: one problem, all of it
  search    lsyn_reset + lsyn_solve on labels that no small formula explains
            (noise): every level up to a size is built; then the first levels
            are exported
  levels    lsyn_reset + lsyn_enumerate_level with full levels: the distinct
            formulas themselves are wanted; then the first levels are exported
  batch     lsyn_batch_solve over many problems of unlike sizes
  serve     lsyn_submit for a burst of problems, then lsyn_wait for each

Answers that depend on the order in which the GPU meets candidates (which of
several minimal formulas, the order of a level's rows, what a level held when it
was stopped at an answer) are returned in a form that does not: the truth of the
formula on the traces, rows in an order of their own, complete levels only.
"""
import math

import numpy as np
import torch

from paper_2504_18943_gb300 import lsyn as L
from paper_2504_18943_gb300 import workloads as W

GIB = 1 << 30
OPS = {"all": L.OPS_ALL, "paper": L.OPS_PAPER}

# Distinct formulas of each size 1, 2, ... by number of propositions, on traces
# many and long enough to tell formulas apart (128 traces of 8..32 positions).
# They say how much a search must store; few or short traces give fewer.
DISTINCT = {
    "all": {
        1: [1, 4, 9, 17, 56, 172, 450, 1296, 3944, 11993, 36083, 109429, 337165, 1044776, 3241093, 10104548],
        2: [2, 8, 21, 77, 333, 1197, 4687, 19650, 79709, 331310, 1401671, 5936830, 25356323],
        3: [3, 12, 37, 181, 876, 3861, 19314, 96681, 480434, 2461282, 12634655],
        4: [4, 16, 57, 329, 1729, 8930, 51495, 290969, 1666254, 9739157],
        5: [5, 20, 81, 521, 2936, 17206, 109854, 686305, 4393251, 28456230],
        6: [6, 24, 109, 757, 4541, 29428, 202634, 1374381, 9581220],
        8: [8, 32, 177, 1361, 9121, 68846, 532226, 4125846, 32784127],
        10: [10, 40, 261, 2141, 15819, 133596, 1129870, 9740803],
    },
    "paper": {
        1: [1, 3, 6, 16, 39, 106, 284, 775, 2194, 6305, 18142, 52443, 152832, 448819, 1324783, 3929859, 11705586],
        2: [2, 6, 15, 53, 181, 654, 2387, 8887, 33824, 131034, 512106, 2021277, 8042521, 32198376],
        3: [3, 9, 27, 113, 452, 1957, 8564, 38555, 177387, 826593, 3890689, 18478330],
        4: [4, 12, 42, 196, 877, 4329, 21441, 109877, 573921, 3033809, 16210491],
        5: [5, 15, 60, 302, 1481, 8092, 44120, 250285, 1443563, 8425851],
        6: [6, 18, 81, 431, 2289, 13570, 79803, 491825, 3069204, 19410720],
        8: [8, 24, 132, 758, 4617, 30812, 204987, 1433629, 10096457],
        10: [10, 30, 195, 1177, 8061, 58685, 431524, 3325139, 25788380],
    },
}


def _sizes(ops, props):
    table = DISTINCT[ops]
    return table[min(p for p in table if p >= props)]


def _row_bytes(case):
    """Bytes of one formula's characteristic matrix: a word per trace, or several for long traces."""
    words = -(-case["len_hi"] // case["bits"])
    return case["traces"] * words * case["bits"] // 8


def _entries(case, upto):
    return sum(_sizes(case["ops"], case["props"])[:max(upto, 0)])


# ----------------------------------------------------------------------------
# The cases
# ----------------------------------------------------------------------------

def listed():
    return [
        # The smallest call: a formula of 7 nodes on about a thousand traces that are on the device already,
        # as a monitoring loop applies it; the launch is all there is.
        {"name": "label_device", "kind": "label", "props": 5, "traces": 997, "bits": 32, "len_lo": 8, "len_hi": 32,
         "size": 7},
        # A data set in host memory labelled by a formula, as the workload generator and an evaluation script do.
        {"name": "evaluate_host", "kind": "evaluate", "props": 6, "traces": 20011, "bits": 64, "len_lo": 8,
         "len_hi": 64, "size": 13},
        # The smallest problem (the tiny configuration): 8 short traces, a hidden formula of 5 nodes.
        {"name": "solve_tiny", "kind": "solve", "props": 2, "traces": 8, "bits": 32, "len_lo": 3, "len_hi": 8,
         "ops": "all", "hidden": 5, "size": 8, "cache_gb": 1.0},
        # An ordinary problem from start to end (the mid configuration's traces): create, solve, destroy. Most
        # answers come within a few small levels.
        {"name": "new_mid", "kind": "new", "props": 5, "traces": 128, "bits": 32, "len_lo": 8, "len_hi": 32,
         "ops": "all", "hidden": 7, "size": 8, "cache_gb": 2.0},
        # Traces of the paper's worked example (14 of 6 positions over two propositions, its grammar): matrices of
        # 56 bytes, deep levels.
        {"name": "levels_example", "kind": "levels", "props": 2, "traces": 14, "bits": 32, "len_lo": 6, "len_hi": 6,
         "ops": "paper", "size": 15, "export": 7, "cache_gb": 8.0},
        # Thirty traces (an odd 120 bytes): the widest matrices that one thread holds.
        {"name": "levels_thirty", "kind": "levels", "props": 4, "traces": 30, "bits": 32, "len_lo": 8, "len_hi": 32,
         "ops": "all", "size": 10, "export": 5, "cache_gb": 4.0},
        # The mid configuration searched through size 10: matrices of 512 bytes, 33 million of them.
        {"name": "search_mid", "kind": "search", "props": 5, "traces": 128, "bits": 32, "len_lo": 8, "len_hi": 32,
         "ops": "all", "size": 10, "export": 4, "cache_gb": 24.0},
        # Traces of up to 64 positions, an odd number of them, as most problems of the batched configuration:
        # matrices of 2000 bytes.
        {"name": "search_odd", "kind": "search", "props": 3, "traces": 250, "bits": 64, "len_lo": 8, "len_hi": 64,
         "ops": "all", "size": 10, "export": 4, "cache_gb": 8.0},
        # The large configuration: 10 propositions, 2048 traces, matrices of 16 KiB, through size 7.
        {"name": "search_large", "kind": "search", "props": 10, "traces": 2048, "bits": 64, "len_lo": 16,
         "len_hi": 64, "ops": "all", "size": 7, "export": 2, "cache_gb": 28.0},
        # Traces longer than a word (several words each).
        {"name": "search_long", "kind": "search", "props": 3, "traces": 200, "bits": 64, "len_lo": 100,
         "len_hi": 200, "ops": "all", "size": 9, "export": 3, "cache_gb": 8.0},
        # Many problems at once (the batched configuration), each capped at the default cache.
        {"name": "batch_64", "kind": "batch", "problems": 64, "props_lo": 2, "props": 8, "traces_lo": 8,
         "traces": 512, "bits": 64, "len_lo": 8, "len_hi": 64, "ops": "all", "hidden_lo": 5, "hidden": 13,
         "size": 12, "cache_gb": 1.0, "pool_gb": 24.0},
        # A burst of requests to a running server (the served configuration's problems).
        {"name": "serve_24", "kind": "serve", "problems": 24, "props_lo": 2, "props": 8, "traces_lo": 8,
         "traces": 512, "bits": 64, "len_lo": 8, "len_hi": 64, "ops": "all", "hidden_lo": 5, "hidden": 13,
         "size": 12, "cache_gb": 1.0, "pool_gb": 24.0},
    ]


def _log(rng, lo, hi):
    """A whole number, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _depth(case, budget_bytes, budget_entries):
    """The deepest size whose levels together keep to the budgets."""
    per = _row_bytes(case) + 16
    k, total = 0, 0
    for n in _sizes(case["ops"], case["props"]):
        if total + n > budget_entries or (total + n) * per > budget_bytes:
            break
        total, k = total + n, k + 1
    return max(3, k)


def _cache_gb(case, upto):
    """Room for the levels, the table and what searches leave unused."""
    need = _entries(case, upto) * (_row_bytes(case) * 1.3 + 64)
    words = -(-case["len_hi"] // case["bits"])
    if words > 1 or _row_bytes(case) > 512:  # rows are padded to 512 bytes a word
        need = _entries(case, upto) * (-(-_row_bytes(case) // words // 512) * 512 * words * 1.3 + 64)
    elif _row_bytes(case) > 128:
        need = _entries(case, upto) * (512 * 1.3 + 64)
    return float(max(1.0, math.ceil(need / GIB)))


def draw(rng):
    kind = rng.choice(["label", "evaluate", "solve", "new", "levels", "levels", "search", "search", "search",
                       "batch", "serve"])
    bits = rng.choice([32, 64])
    props = rng.randint(1, 10)
    if kind == "label":
        size = rng.randint(3, 15)
        return {"kind": kind, "props": props, "traces": _log(rng, 100, (8 << 20) // (size * 8)), "bits": bits,
                "len_lo": 4, "len_hi": bits, "size": size}
    if kind == "evaluate":
        words = rng.choice([1, 1, 1, 2, 3])
        return {"kind": kind, "props": props, "traces": _log(rng, 64, 20000 // words), "bits": bits, "len_lo": 4,
                "len_hi": rng.randint((words - 1) * bits + 8, words * bits), "size": rng.randint(3, 15)}
    if kind in ("solve", "new"):
        case = {"kind": kind, "props": rng.randint(2, 6), "traces": _log(rng, 8, 512), "bits": bits, "len_lo": 4,
                "len_hi": rng.randint(8, bits), "ops": rng.choice(["all", "paper"]), "hidden": rng.randint(3, 9)}
        case["size"] = min(case["hidden"] + 1, _depth(case, 2e9, 2e6))
        case["cache_gb"] = _cache_gb(case, case["size"])
        return case
    if kind == "levels":  # few traces: a matrix of at most 128 bytes
        case = {"kind": kind, "props": rng.randint(1, 5), "traces": rng.randint(5, 1024 // bits), "bits": bits,
                "len_lo": 4, "len_hi": rng.randint(6, bits), "ops": rng.choice(["all", "paper"])}
        case["size"] = _depth(case, 3e9, _log(rng, 20000, 30000000))
        case["export"] = min(4, case["size"])
        case["cache_gb"] = _cache_gb(case, case["size"])
        return case
    if kind == "search":
        words = rng.choice([1, 1, 1, 1, 2, 3])
        case = {"kind": kind, "props": props, "traces": _log(rng, 48, 2500 // words), "bits": bits, "len_lo": 8,
                "len_hi": rng.randint((words - 1) * bits + 16, words * bits), "ops": rng.choice(["all", "paper"])}
        case["size"] = _depth(case, _log(rng, 10 ** 8, 12 * 10 ** 9) / words, 3e7)
        case["export"] = 3
        case["cache_gb"] = _cache_gb(case, case["size"])
        return case
    return {"kind": kind, "problems": rng.randint(4, 48 if kind == "batch" else 20), "props_lo": 2,
            "props": rng.randint(3, 8), "traces_lo": 8, "traces": rng.randint(64, 512), "bits": 64, "len_lo": 8,
            "len_hi": rng.randint(24, 64), "ops": rng.choice(["all", "all", "paper"]), "hidden_lo": 4,
            "hidden": rng.randint(6, 12), "size": rng.randint(8, 12), "cache_gb": 1.0, "pool_gb": 24.0}


def work(case):
    """Bytes in and out: the traces once, and each distinct matrix that is built, stored once; bitwise operations
    are not counted. Where a hidden formula ends the search, the levels below half its size stand for what has to be
    built."""
    if case["kind"] in ("label", "evaluate"):
        rows = _row_bytes(case)
        return {"bytes": rows * (case["props"] + 1) + 4 * case["traces"], "flops": 0}
    if case["kind"] in ("batch", "serve"):
        total = 0
        for props in range(case["props_lo"], case["props"] + 1):
            for hidden in range(case["hidden_lo"], case["hidden"] + 1):
                one = dict(case, props=props, traces=(case["traces_lo"] + case["traces"]) // 2)
                total += _entries(one, hidden // 2 + 1) * _row_bytes(one)
        kinds = (case["props"] - case["props_lo"] + 1) * (case["hidden"] - case["hidden_lo"] + 1)
        return {"bytes": case["problems"] * total / kinds, "flops": 0}
    upto = case["size"] if case["kind"] in ("search", "levels") else case["hidden"] // 2 + 1
    return {"bytes": (case["props"] + _entries(case, upto)) * _row_bytes(case), "flops": 0}


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------

def _traces(seed, props, count, lo, hi):
    return W.draw_traces(W.Stream(W.stream_key(seed, 101)), count, props, lo, hi, np.full(props, 0.5))


def _split(traces, label, bits):
    """Positives first, then negatives."""
    order = np.concatenate([np.flatnonzero(label), np.flatnonzero(~label)])
    taken = traces.take(order)
    return L.pack_traces(taken.bits, taken.lengths, int(label.sum()), int((~label).sum()), bits)


def _hidden_problem(seed, props, count, lo, hi, bits, hidden):
    """Traces labelled by a hidden formula; one that leaves under an eighth of them on a side is drawn again."""
    traces = _traces(seed, props, count, lo, hi)
    for attempt in range(40):
        formula = W.random_formula(W.Stream(W.stream_key(seed, 102, attempt)), hidden, props)
        label = L.labeller(formula, traces, props)
        if count <= 8 * min(int(label.sum()), int((~label).sum())):
            return _split(traces, label, bits)
    return _noise_problem(seed, props, count, lo, hi, bits)


def _noise_problem(seed, props, count, lo, hi, bits):
    """Traces with labels of their own accord, half and half."""
    traces = _traces(seed, props, count, lo, hi)
    label = np.zeros(count, dtype=bool)
    label[np.argsort(W.Stream(W.stream_key(seed, 103)).block(count))[:(count + 1) // 2]] = True
    return _split(traces, label, bits)


class _OnDevice:
    """A problem's traces on the device, for lsyn_eval_noalloc: one word per trace."""

    def __init__(self, packed):
        words = packed.atom_words.view(np.int32 if packed.word_bits == 32 else np.int64)
        self.packed = packed
        self.words = torch.from_numpy(np.ascontiguousarray(words)).cuda()
        self.lengths = torch.from_numpy(packed.lengths).cuda()

    def matrix(self, formula, out=None):
        p = self.packed
        if out is None:
            out = torch.empty(p.n_traces, dtype=self.words.dtype, device="cuda")
        L.lsyn_eval_noalloc(p.n_props, p.n_traces, p.word_bits, self.words.data_ptr(), self.lengths.data_ptr(),
                            formula, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return out


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind in ("label", "evaluate"):
        traces = _traces(seed, case["props"], case["traces"], case["len_lo"], case["len_hi"])
        state["packed"] = L.pack_traces(traces.bits, traces.lengths, case["traces"], 0, case["bits"])
        state["formula"] = W.random_formula(W.Stream(W.stream_key(seed, 104)), case["size"], case["props"])
        if kind == "label":
            state["device"] = _OnDevice(state["packed"])
        return state
    if kind in ("batch", "serve"):
        problems = []
        for i in range(case["problems"]):
            st = W.Stream(W.stream_key(seed, 105, i))
            props = st.randint(case["props_lo"], case["props"])
            count = st.randint(case["traces_lo"], case["traces"])
            hidden = st.randint(case["hidden_lo"], case["hidden"])
            problems.append(_hidden_problem(W.stream_key(seed, 106, i) >> 1, props, count, case["len_lo"],
                                            case["len_hi"], case["bits"], hidden))
        state["problems"] = problems
        state["device"] = [_OnDevice(p) for p in problems]
        cfg = L.make_config(op_mask=OPS[case["ops"]], cache_bytes=int(case["cache_gb"] * GIB))
        tune = L.make_tuning(pool_bytes=int(case["pool_gb"] * GIB))
        state["handle"] = L.Batch(problems, cfg, tune) if kind == "batch" else L.Server(cfg, tune)
        return state
    shape = (case["props"], case["traces"], case["len_lo"], case["len_hi"], case["bits"])
    if kind in ("solve", "new"):
        state["packed"] = _hidden_problem(seed, *shape, case["hidden"])
        state["device"] = _OnDevice(state["packed"])
    else:
        state["packed"] = _noise_problem(seed, *shape)
    state["config"] = L.torch_config(op_mask=OPS[case["ops"]], cache_bytes=int(case["cache_gb"] * GIB),
                                     full_levels=kind == "levels")
    if kind != "new":
        state["handle"] = L.Synthesizer(state["packed"], state["config"])
    return state


# ----------------------------------------------------------------------------
# A pass
# ----------------------------------------------------------------------------

def _in_order(rows):
    """A level's rows in an order that does not depend on the run: by a 64-bit key of their words."""
    flat = rows.reshape(rows.shape[0], -1).astype(np.uint64, copy=False)
    keys = W.Stream(W.stream_key(107)).block(flat.shape[1]) | np.uint64(1)
    with np.errstate(over="ignore"):
        order = np.argsort((flat * keys).sum(axis=1, dtype=np.uint64))
    out = flat[order]
    return out.view(np.int64)


def _complete(levels, size):
    """Candidates and new formulas of every level that was built to its end, a row for each size (zeros: no such
    level)."""
    out = np.zeros((size, 4), dtype=np.int64)
    for lv in levels:
        if not (lv.solved or lv.early_exit or lv.cache_full):
            out[lv.level - 1] = lv.level, lv.candidates, lv.unique, lv.total
    return out


def _rows(case, s, done):
    """The first levels, exported: a block of rows for each, the rest of a block zero."""
    blocks = []
    for k in range(1, case["export"] + 1):
        block = np.zeros((2 * _sizes(case["ops"], case["props"])[k - 1] + 8, _row_words(case)), dtype=np.int64)
        if k <= done:
            rows = _in_order(s.export(k))
            block[:rows.shape[0], :rows.shape[1]] = rows
        blocks.append(block)
    return blocks


def _row_words(case):
    return case["traces"] * -(-case["len_hi"] // case["bits"])


def _solved(case, status, result, formula, levels, device):
    out = {"status": status, "size": result.size, "exact": result.exact, "levels": _complete(levels, case["size"]),
           "nodes": W.formula_size(formula) if formula else 0}
    if formula is None:
        out["labels"] = torch.full_like(device.words[0], -1)
    else:
        out["labels"] = device.matrix(formula) & 1  # its truth at position 0 of every trace
    return out


def _many(case, answers, device):
    out = {"status": np.array([a[0] for a in answers], dtype=np.int64),
           "size": np.array([a[1].size for a in answers], dtype=np.int64),
           "exact": np.array([a[1].exact for a in answers], dtype=np.int64),
           "nodes": np.array([W.formula_size(a[2]) if a[2] else 0 for a in answers], dtype=np.int64)}
    labels = torch.zeros(len(answers), case["traces"], dtype=torch.int64, device="cuda")
    for i, (a, d) in enumerate(zip(answers, device)):
        if a[2]:
            d.matrix(a[2], labels[i, :d.packed.n_traces])
    out["labels"] = labels & 1
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "label":
        return state["device"].matrix(state["formula"])
    if kind == "evaluate":
        out = L.lsyn_eval(state["packed"], state["formula"])
        return out.view(np.int32 if case["bits"] == 32 else np.int64)
    if kind == "solve":
        s = state["handle"]
        s.reset()
        return _solved(case, *s.solve(case["size"]), state["device"])
    if kind == "new":
        with L.Synthesizer(state["packed"], state["config"]) as s:
            return _solved(case, *s.solve(case["size"]), state["device"])
    if kind == "search":
        s = state["handle"]
        s.reset()
        status, result, _, levels = s.solve(case["size"])
        out = {"status": status, "size": result.size, "levels": _complete(levels, case["size"])}
        return dict(out, rows=_rows(case, s, int(np.count_nonzero(out["levels"][:, 0]))))
    if kind == "levels":
        s = state["handle"]
        s.reset()
        levels = [s.level(k) for k in range(1, case["size"] + 1)]
        table = np.array([[lv.level, lv.solved, lv.cache_full, lv.candidates, lv.unique, lv.total] for lv in levels],
                         dtype=np.int64)
        return {"levels": table, "rows": _rows(case, s, len(levels))}
    if kind == "batch":
        statuses, results, formulas = state["handle"].solve(case["size"])
        return _many(case, list(zip(statuses, results, formulas)), state["device"])
    tickets = [state["handle"].submit(p, case["size"]) for p in state["problems"]]
    return _many(case, [state["handle"].wait(t) for t in tickets], state["device"])


# ----------------------------------------------------------------------------
# What the evaluations return, by the definition of satisfaction
# ----------------------------------------------------------------------------

def _truth(text, bits, inside):
    """bool [traces, positions]: where the formula holds; nothing holds at or past a trace's end."""
    tokens = text.replace("(", " ").replace(")", " ").split()
    at = 0

    def node():
        nonlocal at
        token = tokens[at]
        at += 1
        if token[0] == "p":
            return bits[:, :, int(token[1:])] & inside
        a = node()
        if token == "!":
            return ~a & inside
        if token == "X":
            return np.concatenate([a[:, 1:], np.zeros_like(a[:, :1])], axis=1)
        if token in "FG":
            a = ~a & inside if token == "G" else a
            a = np.logical_or.accumulate(a[:, ::-1], axis=1)[:, ::-1] & inside
            return ~a & inside if token == "G" else a
        b = node()
        if token == "&":
            return a & b
        if token == "|":
            return a | b
        out = b.copy()
        for t in range(b.shape[1] - 2, -1, -1):
            out[:, t] |= a[:, t] & out[:, t + 1]
        return out

    return node()


def exact(case, seed):
    if case["kind"] not in ("label", "evaluate"):
        return None  # whole numbers that only a search of its own could give
    traces = _traces(seed, case["props"], case["traces"], case["len_lo"], case["len_hi"])
    formula = W.random_formula(W.Stream(W.stream_key(seed, 104)), case["size"], case["props"])
    inside = np.arange(traces.bits.shape[1])[None, :] < traces.lengths[:, None]
    truth = _truth(formula, traces.bits, inside)
    bits = case["bits"]
    words = -(-int(traces.lengths.max()) // bits)
    truth = np.pad(truth, ((0, 0), (0, max(0, words * bits - truth.shape[1]))))[:, :words * bits]
    packed = np.packbits(truth.reshape(truth.shape[0], words, bits), axis=2, bitorder="little")
    out = packed.view("<i4" if bits == 32 else "<i8")[:, :, 0]
    return out[:, 0] if words == 1 else out
