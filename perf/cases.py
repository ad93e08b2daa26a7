"""What is timed: whole combinator programs run fused through the Python binding, as a user's program runs them.

A program is built, planned and bound once; then `Graph.run(FUSED)` is called on it again and again.  The programs
are the five benchmark programs (1-D chain, transpose-fuse-reduce, random gather + scan, Jacobi chain, scatter
histogram + diamond) and the further ones that `bench.py` and the tests run beside them (segmented sums, scans with
readers, per-row scans), from the smallest calls, where launches and the host count, to arrays several times the L2,
with extents that allow 128-bit rows and extents that do not.
"""
import math

import torch

import workloads as W
from paper_2407_13585_b200 import binding as B

# ---- the cases -----------------------------------------------------------------------------------


def listed():
    return [
        # The first benchmark configuration at its own size, called as the quick start calls it: the caller waits for
        # every result, so what counts is the time of one call.
        {"name": "chain_64k_waited", "program": "chain", "n": 1 << 16, "wait": True},
        # The same chain over an array of twice the L2 eight times over: a stream that is read once.
        {"name": "chain_256m", "program": "chain", "n": 1 << 28, "wait": False},
        # The second configuration at full size: an array read as it lies and transposed, row sums.
        {"name": "transpose_8192", "program": "transpose", "rows": 8192, "wait": False},
        # The same on a matrix of odd extent that fits L2 (rows without 128-bit alignment).
        {"name": "transpose_1999", "program": "transpose", "rows": 1999, "wait": False},
        # The third configuration at full size: random 4-byte gathers from an array beyond L2, then a running sum.
        {"name": "gather_scan_64m", "program": "gather_scan", "n": 1 << 26, "wait": False},
        # The same on an odd number of elements whose source fits L2 (an index column of a medium table).
        {"name": "gather_scan_5m_odd", "program": "gather_scan", "n": 5000003, "wait": False},
        # The fourth configuration at full size, planned by the paper's rules: four iterations, a cluster each.
        {"name": "jacobi_8192", "program": "jacobi", "rows": 8192, "cols": 8192, "iters": 4, "depth": 0, "wait": False},
        # A rectangular grid planned with recomputation allowed: two iterations to a cluster.
        {"name": "jacobi_pairs_3000x5000", "program": "jacobi", "rows": 3000, "cols": 5000, "iters": 4, "depth": 2, "wait": False},
        # The fifth configuration at full size: a skewed histogram, the total and the quotient.
        {"name": "histogram_128m", "program": "histogram", "n": 1 << 27, "bins": 1 << 16, "wait": False},
        # Sums and maxima of a million segments of very unequal lengths (ragged batches).
        {"name": "segmented_128m", "program": "segmented", "n": 1 << 27, "segments": 1 << 20, "wait": False},
        # Three scans in both directions with element-wise readers: the most memory traffic of all programs.
        {"name": "scan_consumers_64m", "program": "scan_consumers", "n": 1 << 26, "wait": False},
        # Per-row running sums and maxima of a rank-2 array whose rows are no multiple of anything.
        {"name": "row_scans_4099x3001", "program": "row_scans", "rows": 4099, "cols": 3001, "wait": False},
    ]


def _size(rng, lo, hi):
    """An integer between lo and hi, even over the logarithm; every third one is a multiple of 64, the others as they fall."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 1 / 3:
        v -= v % 64
    return max(lo, min(hi, v))


def draw(rng):
    program = rng.choice(["chain", "transpose", "gather_scan", "jacobi", "histogram", "segmented", "scan_consumers", "row_scans"])
    case = {"program": program}
    if program == "chain":
        case["n"] = _size(rng, 1 << 10, 1 << 28)
    elif program == "transpose":
        case["rows"] = _size(rng, 64, 8192)
    elif program == "gather_scan":
        case["n"] = _size(rng, 1 << 12, 3 << 24)
    elif program == "jacobi":
        case["rows"], case["cols"] = _size(rng, 64, 4096), _size(rng, 64, 4096)
        case["iters"], case["depth"] = rng.choice([2, 4]), rng.choice([0, 2])
    elif program == "histogram":
        case["n"] = _size(rng, 1 << 14, 1 << 27)
        case["bins"] = min(case["n"] // 16, rng.choice([_size(rng, 1 << 8, 1 << 16), 1 << rng.randint(8, 16)]))
    elif program == "segmented":
        case["n"] = _size(rng, 1 << 14, 1 << 27)
        case["segments"] = max(1, case["n"] // _size(rng, 8, 4096))
    elif program == "scan_consumers":
        case["n"] = _size(rng, 1 << 12, 3 << 24)
    else:
        case["rows"] = _size(rng, 1, 8192)
        case["cols"] = _size(rng, 64, max(64, min(1 << 22, (3 << 24) // case["rows"])))
    case["wait"] = rng.random() < 1 / 3
    return case


def _program(case):
    p = case["program"]
    if p == "chain":
        return W.config1(case["n"])
    if p == "transpose":
        return W.config2(case["rows"])
    if p == "gather_scan":
        return W.config3(case["n"])
    if p == "jacobi":
        return W.config4(case["rows"], case["cols"], case["iters"])
    if p == "histogram":
        return W.config5(case["n"], case["bins"])
    if p == "segmented":
        return W.segmented_sums(case["n"], case["segments"])
    if p == "scan_consumers":
        return W.scan_consumers(case["n"])
    return W.row_scans(case["rows"], case["cols"])


# ---- inputs, one pass -------------------------------------------------------------------------------


def _inputs(case, prog, seed):
    """Inputs with the distributions of the benchmark: U[-1, 1), N(0, 1) for the Jacobi grid, uniform indices, Zipf(1.1) keys
    over 2^20 ids, segment lengths shared out in proportion to rank^-1.1."""
    if case["program"] != "gather_scan":
        return W.make_inputs(prog, seed=seed, device="cuda")
    n = case["n"]                                        # (any number of elements, not only powers of two)
    x = W.inputs.uniform_int(seed, 0, n, 1 << 31, device="cuda")
    idx = W.inputs.uniform_int(seed, 2, n, 1 << 31, device="cuda").remainder_(n)
    return {prog.id("x"): x, prog.id("idx"): idx}


def prepare(case, seed):
    prog = _program(case)
    g = B.Graph(prog.nodes, prog.outputs)
    # small graphs: the best of all legal clusterings; larger ones: branch and bound from the greedy result
    mode = "enumerate" if sum(nd.kind != "input" for nd in prog.nodes) <= 12 else "branch_bound"
    if case.get("depth", 0):
        g.plan_recompute(mode, "bytes", case["depth"])
    else:
        g.plan(mode, "bytes")
    g.refine_to_kernels()
    for i, t in _inputs(case, prog, seed & 0x1FFFFF).items():
        g.bind(i, t)
    outs = {}
    for o in prog.outputs:
        nd = prog.nodes[o]
        outs[nd.name] = torch.empty(nd.shape, dtype=torch.float32 if nd.dtype == "f32" else torch.int32, device="cuda")
        g.bind(o, outs[nd.name])
    g.ensure_workspace(B.FUSED)
    return {"graph": g, "outs": outs, "wait": case["wait"]}


def run(state):
    state["graph"].run(B.FUSED, finish=state["wait"])
    return state["outs"]


# ---- what a pass cannot do without ---------------------------------------------------------------------


def _count(nd):
    return math.prod(nd.shape)


# element operations per element of the program's largest array
_OPS = {"chain": 4, "transpose": 3, "gather_scan": 5, "histogram": 6, "segmented": 4, "scan_consumers": 9, "row_scans": 4}


def work(case):
    """Every program input read once and every program output written once; the element operations of the combinators."""
    prog = _program(case)
    moved = 4 * (sum(_count(prog.nodes[i]) for i in prog.input_ids()) + sum(_count(prog.nodes[o]) for o in prog.outputs))
    ops = 5 * case["iters"] if case["program"] == "jacobi" else _OPS[case["program"]]
    return {"bytes": moved, "flops": ops * max(_count(nd) for nd in prog.nodes)}


def tolerance(case):
    """Whole numbers and fp32 element chains (rounded after every operation, in the written order) are exact.  fp32 sums
    and scans may be added up in any order: about four times the largest difference from the same sums in fp64 that sizes
    from 2^14 to 2^28 showed (chain: more, since its one number is a sum of terms of both signs and may come out small
    beside the sum of their magnitudes)."""
    return {
        "gather_scan": "exact",
        "jacobi": "exact",
        "chain": {"rel": 5e-5, "max": 5e-5},
        "transpose": {"rel": 3e-7, "max": 1e-6},
        "histogram": {"rel": 4e-7, "max": 1e-6},
        "segmented": {"rel": 1e-6, "max": 4e-6},
        "scan_consumers": {"rel": 2e-6, "max": 5e-6},
        "row_scans": {"rel": 2e-6, "max": 5e-6},
    }[case["program"]]
