"""The work that a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  ``listed()`` names the fixed ones, ``draw()``
gives more of the same ranges, ``prepare()`` makes what a program holds before
the call (a resident packed forest, rows, output buffers), ``run()`` is one call
through the public binding, ``work()`` counts what the call cannot do without,
and ``exact()`` evaluates forests with real leaf values in 64 bits.

Forests and rows are the repository's seeded stand-ins (``datagen``): a forest
is trained once per process and its first ``trees`` trees are used; the rows of
a seed are a fresh stream of the same distribution.
"""
from __future__ import annotations

import functools
import math

import torch

import datagen
import paper_1806_07300_gb300 as fp

# internal nodes per tree and internal nodes visited per (row, tree), measured
# on each forest's own test rows
_SHAPE = {"tiny": (80, 7.8), "wide": (5419, 13.1), "image": (15436, 22.1), "hbm": (78834, 22.5),
          "regress": (31871, 18.6), "boosted": (52, 6.0)}

# the most rows a drawn case of a forest has (784-feature rows are 3 KB each)
_MAX_ROWS = {"tiny": 100_000, "wide": 100_000, "image": 250_000, "hbm": 4_000_000, "regress": 4_000_000,
             "boosted": 4_000_000}

# layouts that the benchmark's autotuner settles on; "default" is the library's own
_TUNED = {
    "tiny": dict(bin_size=16, interleave_depth=7, head_select=2, obs_tile=256, bin_buffers=2),
    "wide": dict(bin_size=8, interleave_depth=7, head_select=2, obs_tile=224, bin_buffers=2),
    "image": dict(bin_size=32, interleave_depth=3, head_select=2, obs_tile=64, refill_lanes=16, bin_buffers=2),
    "hbm": dict(bin_size=5, interleave_depth=9, head_select=2, obs_tile=992, refill_lanes=16, bin_buffers=2),
    "regress": dict(bin_size=4, interleave_depth=9, head_select=2, obs_tile=1024, refill_lanes=16, bin_buffers=2),
    "boosted": dict(bin_size=64, interleave_depth=5, head_select=2, obs_tile=768, refill_lanes=16, bin_buffers=3),
}

# the forests that the serving workload keeps resident side by side
_SERVED = "tiny,wide,image,hbm"


def _case(call, forest, rows, trees=0, layout="default", votes=False, classes=False, name=None):
    c = {"call": call, "forest": forest, "rows": rows, "trees": trees, "layout": layout, "votes": votes,
         "classes": classes}
    return c if name is None else {"name": name, **c}


def listed() -> list[dict]:
    return [
        # one serving request of the median size, alone on the GPU: latency
        _case("predict", "wide", 32, votes=True, classes=True, name="wide_request"),
        # the smallest benchmark workload: a small forest over a few thousand rows
        _case("predict", "tiny", 10_000, votes=True, classes=True, name="tiny_10k"),
        # a mid-size ragged batch on the forest that does not fit in L2
        _case("predict", "hbm", 20_011, classes=True, name="hbm_20k"),
        # the headline: bulk scoring with a tuned layout
        _case("predict", "hbm", 4_000_000, layout="tuned", votes=True, classes=True, name="hbm_4m"),
        # 784-feature rows, a validation-set-size batch and a large one
        _case("predict", "image", 10_000, votes=True, classes=True, name="image_10k"),
        _case("predict", "image", 250_000, classes=True, name="image_250k"),
        # a regression forest: mean of the trees' leaf values
        _case("values", "regress", 1_000_003, name="regress_1m"),
        # gradient-boosted shallow trees, all of them in shared memory
        _case("values", "boosted", 2_000_000, layout="tuned", name="boosted_2m"),
        # what the serving runtime launches: a few requests for each resident forest
        _case("batched", _SERVED, "41,96,33,178", classes=True, name="serving_mix"),
        # uneven batches of several forests in one launch
        _case("batched", _SERVED, "9973,52001,3,8209", votes=True, classes=True, name="uneven_batches"),
        # rows and classes in host memory, copies overlapped with the kernels
        _case("host", "hbm", 1_000_000, layout="tuned", classes=True, name="hbm_host_1m"),
        # the leaf of every (row, tree), for statistics over observations
        _case("leaves", "wide", 50_021, name="wide_leaves"),
    ]


def _log_uniform(rng, lo: int, hi: int) -> int:
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng) -> dict:
    call = rng.choice(["predict", "predict", "predict", "values", "values", "batched", "leaves", "host"])
    layout = rng.choice(["default", "default", "tuned"])
    if call == "batched":
        names = rng.sample(_SERVED.split(","), rng.randint(2, 4))
        if rng.random() < 0.5:  # requests of log-normal sizes
            rows = [min(4096, max(1, round(math.exp(rng.gauss(math.log(32), 1.5))))) for _ in names]
        else:  # batches spread over 1 .. 100,000 rows
            rows = [_log_uniform(rng, 1, 100_000) for _ in names]
        return _case(call, ",".join(names), ",".join(map(str, rows)), layout=layout, votes=rng.random() < 0.5,
                     classes=True)
    if call == "values":
        name = rng.choice(["regress", "boosted"])
    else:
        name = rng.choice(["tiny", "wide", "image", "hbm", "hbm"])
    cap = _MAX_ROWS[name]
    if call == "leaves":
        cap = min(cap, 100_000)  # one leaf id per (row, tree) is written
    if call == "host":
        cap = min(cap, 1_000_000)
    top = datagen.RECIPES[name]["T"]
    votes = rng.random() < 0.5
    if call in ("values", "leaves"):
        return _case(call, name, _log_uniform(rng, 1, cap), _log_uniform(rng, 8, top), layout)
    return _case(call, name, _log_uniform(rng, 1, cap), _log_uniform(rng, 8, top), layout, votes,
                 not votes or rng.random() < 0.5)


def _parts(case) -> list[tuple[str, int]]:
    """(forest, rows) of each batch of the case."""
    return list(zip(str(case["forest"]).split(","), map(int, str(case["rows"]).split(","))))


def _n_trees(case, name: str) -> int:
    return case["trees"] or datagen.RECIPES[name]["T"]


@functools.lru_cache(maxsize=None)
def _trained(name: str):
    try:
        return datagen.forest(name)
    except OSError:  # no place to keep it
        return datagen.forest(name, use_cache=False)


@functools.lru_cache(maxsize=None)
def _forest(name: str, trees: int):
    """The first `trees` trees of a workload's forest."""
    f = _trained(name)
    if trees == f.n_trees:
        return f
    m = int(f.node_begin[trees])
    scale = 1.0 / trees if name == "regress" else f.value_scale
    return datagen.Forest(f.n_features, f.n_classes, f.node_begin[:trees + 1], f.left[:m], f.right[:m],
                          f.feature[:m], f.threshold[:m], f.leaf_class[:m], f.cardinality[:m], f.tree_depth[:trees],
                          None if f.leaf_value is None else f.leaf_value[:m], scale, f.value_bias)


@functools.lru_cache(maxsize=16)
def _packed(name: str, trees: int, layout: str):
    return fp.fp_pack_forest(_forest(name, trees), **(_TUNED[name] if layout == "tuned" else {}))


def _rows(name: str, seed: int, n: int):
    """Rows of the workload's distribution, a stream of their own per seed."""
    return torch.from_numpy(datagen.rows(name, 16 + seed, n)[0])


def prepare(case, seed):
    parts = []
    for k, (name, n) in enumerate(_parts(case)):
        df = fp.fp_upload(_packed(name, _n_trees(case, name), case["layout"]))
        X = _rows(name, seed + k, n)
        host = case["call"] == "host"
        X = X.pin_memory() if host else X.cuda()

        def out(*shape, dtype=torch.int32):
            t = torch.empty(shape, dtype=dtype, pin_memory=host) if host else torch.empty(shape, dtype=dtype,
                                                                                          device="cuda")
            return t

        p = {"df": df, "X": X, "votes": None, "classes": None}
        if case["votes"]:
            p["votes"] = out(n, df.info["n_classes"])
        if case["classes"]:
            p["classes"] = out(n)
        if case["call"] == "values":
            p["out"] = out(n, dtype=torch.float32)
        if case["call"] == "leaves":
            p["leaves"] = out(n, df.info["n_trees"])
        parts.append(p)
    torch.cuda.synchronize()
    return {"call": case["call"], "parts": parts}


def run(state):
    parts = state["parts"]
    p = parts[0]
    call = state["call"]
    if call == "batched":
        votes = [q["votes"] for q in parts]
        fp.fp_predict_batched([q["df"] for q in parts], [q["X"] for q in parts],
                              None if votes[0] is None else votes, [q["classes"] for q in parts])
        return [{k: q[k] for k in ("votes", "classes") if q[k] is not None} for q in parts]
    if call == "values":
        fp.fp_predict_values(p["df"], p["X"], p["out"], p["df"].value_scale, p["df"].value_bias)
        return {"out": p["out"]}
    if call == "leaves":
        fp.fp_predict_leaves(p["df"], p["X"], p["leaves"])
        return {"leaves": p["leaves"]}
    if call == "host":
        fp.fp_predict_host(p["df"], p["X"], p["votes"], p["classes"])
        torch.cuda.current_stream().synchronize()  # the results are read on the host next
    else:
        fp.fp_predict(p["df"], p["X"], p["votes"], p["classes"])
    return {k: p[k] for k in ("votes", "classes") if p[k] is not None}


def work(case) -> dict:
    """Bytes: the rows, the outputs, and 8 bytes (threshold, feature, child)
    for each internal node that the rows can reach; operations: one compare
    per internal node visited."""
    nbytes = flops = 0.0
    for name, n in _parts(case):
        r = datagen.RECIPES[name]
        T = _n_trees(case, name)
        nodes, visits = _SHAPE[name]
        per_row = {"values": 4, "leaves": 4 * T}.get(case["call"],
                                                     4 * (r["C"] * case["votes"] + case["classes"]))
        nbytes += n * (4 * r["d"] + per_row) + 8 * T * min(nodes, n * visits)
        flops += n * T * visits
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """Forests with leaf values: bias + scale * the sum, in float64, of the
    leaf values that a plain level-by-level walk reaches.  The other calls
    give whole numbers."""
    if case["call"] != "values":
        return None
    (name, n), = _parts(case)
    f = _forest(name, _n_trees(case, name))
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    X = _rows(name, seed, n).to(dev).double()
    total = torch.zeros(n, dtype=torch.float64, device=dev)
    row = torch.arange(n, device=dev)
    for t in range(f.n_trees):
        a, b = int(f.node_begin[t]), int(f.node_begin[t + 1])
        left, right, feat, thr, val = (torch.from_numpy(v[a:b]).to(dev) for v in (
            f.left, f.right, f.feature, f.threshold, f.leaf_value))
        # a leaf leads to itself, so every row can take as many steps as the tree is deep
        self_id = torch.arange(b - a, dtype=torch.int32, device=dev)
        leaf = left < 0
        left, right = torch.where(leaf, self_id, left), torch.where(leaf, self_id, right)
        feat, thr, val = feat.clamp(min=0), thr.double(), val.double()
        node = torch.zeros(n, dtype=torch.int32, device=dev)
        for _ in range(int(f.tree_depth[t])):
            go_left = X[row, feat[node]] <= thr[node]
            node = torch.where(go_left, left[node], right[node])
        total += val[node]
    return {"out": f.value_bias + f.value_scale * total}
