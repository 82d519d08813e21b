"""The work that a solver has this library do, as cases to be timed: single
tables from the smallest to the largest, networks, searches, the construction
of a table and the learned branching order, each through the public entry
points (paper_2507_18413_gb300.ct). Sizes are those of this repository's
configurations, tests and benchmark: the synthetic configurations (arity 3 of
200 tuples up to 1e7 tuples of arity 5), the paper's instance shapes (80-150
variables, domains up to 600, 5,000-10,000 tuples), the many-table network,
the 20-variable search and the learned-order instances.

A stream is planned in prepare(): edits are drawn on the domains that the
previous propagation left, as a search would make them, and run() replays the
planned calls. Every result but the learned order's is a set of bits or a
count: whole numbers, the same for every correct propagation.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2507_18413_gb300 import ct as C
from paper_2507_18413_gb300 import inputs as G


def listed():
    return [
        # configuration 1: the smallest table, propagated at every node of a
        # small search from host buffers; launches and waits are all there is
        {"name": "tiny_stream", "kind": "stream", "arity": 3, "dom": 8, "tuples": 200, "calls": 32, "depth": 8,
         "host": True, "star": 0.0, "negative": False},
        # a mid-size table inside a search, domains in host memory
        {"name": "small_stream", "kind": "stream", "arity": 6, "dom": 32, "tuples": 100_000, "calls": 32, "depth": 8,
         "host": True, "star": 0.0, "negative": False},
        # the headline stream of the benchmark: delta and reset edits on a
        # large table, domains on the device
        {"name": "large_stream", "kind": "stream", "arity": 6, "dom": 32, "tuples": 4_000_000, "calls": 32, "depth": 8,
         "host": False, "star": 0.0, "negative": False},
        # the paper's instances (LIN_B): a wide scope with large domains and few tuples
        {"name": "wide_stream", "kind": "stream", "arity": 100, "dom": 500, "tuples": 10_000, "calls": 16, "depth": 6,
         "host": False, "star": 0.0, "negative": False},
        # a negative table (forbidden tuples), odd sizes
        {"name": "negative_stream", "kind": "stream", "arity": 4, "dom": 13, "tuples": 20_011, "calls": 24, "depth": 8,
         "host": True, "star": 0.0, "negative": True},
        # the largest table: every variable loses half its values at once, the
        # call that reads the most (one per restart or per cut of a solver)
        {"name": "bulk_reset", "kind": "bulk", "arity": 5, "dom": 64, "tuples": 10_000_000, "calls": 2, "keep": 31},
        # the construction of a table from its tuples and its first propagation
        {"name": "build_table", "kind": "build", "arity": 6, "dom": 32, "tuples": 1_000_000},
        # configuration 3: a network of many tables, the fixpoint after a few
        # variables were cut
        {"name": "network", "kind": "network", "tables": 512, "vars": 1024, "dom": 128, "tuples": 100_000, "calls": 8},
        # configuration 2: the plain depth-first search, one fixpoint per node
        {"name": "search_dfs", "kind": "dfs", "vars": 20, "tables": 8, "arity": 6, "dom": 32, "tuples": 100_000,
         "nodes": 200},
        # all solutions of an instance by the search that runs on the device
        {"name": "search_device", "kind": "device", "vars": 10, "tables": 14, "dom": 16, "log2_solutions": 0,
         "slots": 512, "split": 10},
        # the learned order trained on collected samples, then scoring them all
        {"name": "train_order", "kind": "train", "samples": 20_000, "epochs": 1, "batch": 128},
        # a learned order's view of search nodes: the fixpoint and the features of a cut
        {"name": "node_features", "kind": "features", "vars": 25, "tables": 40, "dom": 16, "tuples": 20_000,
         "calls": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stream", "stream", "wide", "negative", "bulk", "build", "network", "dfs", "device", "train",
                       "features"])
    if kind == "stream":
        arity = rng.randint(3, 6)
        return {"kind": "stream", "arity": arity, "dom": _log(rng, 8, 64), "tuples": _log(rng, 200, 4_000_000),
                "calls": rng.randint(8, 32), "depth": rng.randint(4, 8), "host": rng.random() < 0.5,
                "star": rng.choice([0.0, 0.0, 0.1]), "negative": False}
    if kind == "wide":
        return {"kind": "stream", "arity": rng.randint(80, 120), "dom": rng.randint(200, 600),
                "tuples": rng.randint(5_000, 10_000), "calls": rng.randint(8, 16), "depth": rng.randint(3, 6),
                "host": rng.random() < 0.5, "star": 0.0, "negative": False}
    if kind == "negative":
        dom = rng.randint(8, 15)
        return {"kind": "stream", "arity": 4, "dom": dom, "tuples": rng.randint(dom ** 4 // 4, dom ** 4),
                "calls": rng.randint(8, 24), "depth": rng.randint(4, 8), "host": rng.random() < 0.5, "star": 0.0,
                "negative": True}
    if kind == "bulk":
        arity, dom = rng.choice([(5, 64), (6, 32), (4, 100)])
        return {"kind": "bulk", "arity": arity, "dom": dom, "tuples": _log(rng, 300_000, 8_000_000), "calls": 2,
                "keep": rng.randint(dom // 4, dom // 2)}
    if kind == "build":
        return {"kind": "build", "arity": rng.randint(3, 8), "dom": _log(rng, 8, 128),
                "tuples": _log(rng, 10_000, 2_000_000)}
    if kind == "network":
        tables = _log(rng, 16, 400)
        return {"kind": "network", "tables": tables, "vars": 2 * tables + rng.randint(0, 9), "dom": rng.randint(16, 128),
                "tuples": _log(rng, 10_000, 100_000), "calls": rng.randint(2, 8)}
    if kind == "dfs":
        return {"kind": "dfs", "vars": rng.randint(12, 24), "tables": rng.randint(6, 12), "arity": rng.randint(4, 6),
                "dom": rng.randint(16, 32), "tuples": _log(rng, 5_000, 100_000), "nodes": rng.randint(60, 200)}
    if kind == "device":
        return {"kind": "device", "vars": rng.randint(9, 10), "tables": rng.randint(14, 18),
                "dom": rng.randint(13, 16), "log2_solutions": rng.randint(-6, 0), "slots": rng.randint(64, 512),
                "split": rng.randint(6, 10)}
    if kind == "train":
        return {"kind": "train", "samples": _log(rng, 500, 20_000), "epochs": 1, "batch": rng.randint(32, 128)}
    return {"kind": "features", "vars": rng.randint(20, 30), "tables": rng.randint(30, 50), "dom": rng.randint(8, 16),
            "tuples": _log(rng, 1_000, 20_000), "calls": rng.randint(2, 8)}


# --------------------------------------------------------------------------
# what a program keeps between calls
# --------------------------------------------------------------------------
class Owned:
    """A handle of the library, destroyed with the state that holds it."""

    def __init__(self, handle, destroy):
        self.h = handle
        self._destroy = destroy

    def __del__(self):
        if self.h is not None:
            self._destroy(self.h)
            self.h = None


def _tuples(case, seed):
    """Uniform tuples over {0..dom-1}; duplicates may occur, as in extracted relations."""
    g = np.random.default_rng(seed)
    tup = g.integers(0, case["dom"], (case["tuples"], case["arity"]), dtype=np.int32)
    if case.get("star"):
        tup[g.random(tup.shape) < case["star"]] = C.CT_STAR
    return tup


def _table(case, seed):
    n, d = case["arity"], case["dom"]
    st, h = C.ct_create(n, [0] * n, [d] * n, _tuples(case, seed), stream=torch.cuda.current_stream(),
                        negative=case.get("negative", False))
    C.check(st)
    return Owned(h, C.ct_destroy)


def _edit(rng, masks):
    """What a search does to the domains between two propagations: one or two
    values off (a right branch), or most of a domain off (a left branch)."""
    new, i = (G.delta_step if rng.int(2) else G.reset_step)(rng, masks)
    if i is None:
        new, _ = G.remove_random_values(rng, masks, 1)
    return new


def _prepare_stream(case, seed):
    n, d = case["arity"], case["dom"]
    own = _table(case, seed)
    h, size = own.h, [d] * n
    off, nw = C.dom_layout(size)
    DW = int(off[-1])
    words = C.masks_to_words([np.ones(d, bool)] * n)
    C.check(C.ct_propagate_host(h, words)[0])  # the root
    C.check(C.ct_save(h)[0])
    root = C.words_to_masks(words, size)
    rng = G.Rng(seed)
    masks, depth, ops, inputs = root, 0, [], []
    for _ in range(case["calls"]):
        C.check(C.ct_save(h)[0])
        w = C.masks_to_words(_edit(rng, masks))
        inputs.append(w.copy())
        st, _ = C.ct_propagate_host(h, w)
        C.check(st)
        ops.append(("call", st == C.CT_OK))
        depth += 1
        if st != C.CT_OK or depth >= case["depth"]:
            C.check(C.ct_restore(h, 1))
            ops.append(("back", True))
            masks, depth = root, 0
        else:
            masks = C.words_to_masks(w, size)
    C.check(C.ct_restore(h, 0))
    C.check(C.ct_save(h)[0])
    # the domains of a failed call are unspecified: they go to rows of their own at the end
    ok = [good for op, good in ops if op == "call"]
    failed = [k for k, good in enumerate(ok) if not good]
    given = np.stack(inputs + [inputs[k] for k in failed])
    at = {k: len(ok) + i for i, k in enumerate(failed)}
    state = {"own": own, "calls": len(ok), "words": int(C.ct_get_info(h)[1]["words"]),
             "room": (case["tuples"] + 31) // 32}
    if case["host"]:
        state["given"], state["work"] = given, np.zeros_like(given)
        base = state["work"].ctypes.data
    else:
        state["given"] = torch.from_numpy(given.view(np.int32)).cuda()
        state["work"] = torch.zeros_like(state["given"])
        base = state["work"].data_ptr()
    nch = (n + 31) // 32
    state["changed"] = np.zeros((len(ok), nch), np.uint32)
    lib, lv, u32 = C.load(), ctypes.c_int(0), ctypes.POINTER(ctypes.c_uint32)
    state["level"] = lv
    seq, k = [], 0
    for op, good in ops:
        if op == "back":
            seq.append((lib.ct_restore, (h, 1)))
            continue
        seq.append((lib.ct_save, (h, ctypes.byref(lv))))
        p = base + at.get(k, k) * DW * 4
        ch = ctypes.cast(state["changed"].ctypes.data + k * nch * 4, u32)
        seq.append((lib.ct_propagate_host, (h, ctypes.cast(p, u32), ch)) if case["host"] else (lib.ct_propagate, (h, p, ch)))
        k += 1
    state["seq"] = seq
    return state


def _run_stream(s):
    h = s["own"].h
    if isinstance(s["work"], np.ndarray):
        np.copyto(s["work"], s["given"])
    else:
        s["work"].copy_(s["given"])
    status = []
    for f, a in s["seq"]:
        r = f(*a)
        if r < 0:
            raise RuntimeError(C.last_error())
        status.append(r)
    # the state the stream left, then back to the root
    if status[-1] == C.CT_OK:
        st, table, live = C.ct_get_currtable(h, s["words"])
        C.check(st)
    else:
        table, live = np.zeros(s["words"], np.uint32), 0
    if len(table) < s["room"]:  # a negative table keeps each tuple once
        table = np.concatenate([table, np.zeros(s["room"] - len(table), np.uint32)])
    C.check(C.ct_restore(h, 0))
    C.check(C.ct_save(h)[0])
    return {"domains": s["work"][: s["calls"]], "changed": s["changed"], "status": np.array(status), "table": table,
            "live": live}


def _prepare_bulk(case, seed):
    n, d = case["arity"], case["dom"]
    own = _table(case, seed)
    g = np.random.default_rng(seed + 7)
    rows = []
    for _ in range(case["calls"]):
        masks = []
        for _ in range(n):
            m = np.zeros(d, bool)
            m[g.permutation(d)[: case["keep"]]] = True
            masks.append(m)
        rows.append(C.masks_to_words(masks).view(np.int32))
    given = torch.from_numpy(np.stack(rows)).cuda()
    C.check(C.ct_save(own.h)[0])
    return {"own": own, "given": given, "work": torch.zeros_like(given), "words": (case["tuples"] + 31) // 32}


def _run_bulk(s):
    h, table = s["own"].h, None
    s["work"].copy_(s["given"])
    status, live = [], []
    for k in range(s["work"].shape[0]):
        st, _ = C.ct_propagate(h, s["work"][k], 1)
        status.append(C.check(st))
        if k == s["work"].shape[0] - 1:
            st, table, nz = C.ct_get_currtable(h, s["words"])
            live.append(nz)
        C.check(C.ct_restore(h, 0))
        C.check(C.ct_save(h)[0])
    return {"domains": s["work"], "status": np.array(status), "table": table, "live": np.array(live)}


def _prepare_build(case, seed):
    g = np.random.default_rng(seed + 3)
    d, keep = case["dom"], max(2, (3 * case["dom"]) // 4)
    masks = []
    for _ in range(case["arity"]):
        m = np.zeros(d, bool)
        m[g.permutation(d)[:keep]] = True
        masks.append(m)
    return {"case": dict(case), "tuples": _tuples(case, seed), "domains": C.masks_to_words(masks)}


def _run_build(s):
    n, d = s["case"]["arity"], s["case"]["dom"]
    st, h = C.ct_create(n, [0] * n, [d] * n, s["tuples"], stream=torch.cuda.current_stream())
    C.check(st)
    try:
        w = s["domains"].copy()
        st, changed = C.ct_propagate_host(h, w, (n + 31) // 32)
        C.check(st)
        st2, table, live = C.ct_get_currtable(h, (len(s["tuples"]) + 31) // 32)
        C.check(st2)
        st3, row = C.ct_get_support_row(h, n * d - 1, (len(s["tuples"]) + 31) // 32)
        C.check(st3)
    finally:
        C.ct_destroy(h)
    return {"domains": w, "changed": changed, "status": st, "table": table, "live": live, "row": row}


def _model(spec):
    st, m = C.ct_model_create(spec.dom_lo, spec.dom_size, stream=torch.cuda.current_stream())
    C.check(st)
    own = Owned(m, C.ct_model_destroy)
    for tb in spec.tables:
        C.check(C.ct_model_add_table(m, tb.scope, tb.tuples))
    return own


def _network_spec(case, seed):
    """Tables of arity 2-8 over random scopes, log-uniform tuple counts, half of
    them with skewed columns."""
    g = np.random.default_rng(seed)
    nv = case["vars"]
    sizes = [int(v) for v in np.random.default_rng(nv).integers(8, case["dom"] + 1, nv)]  # the model's, not the data's
    spec = G.CspSpec(nvars=nv, dom_lo=[0] * nv, dom_size=sizes)
    for k in range(case["tables"]):
        scope = [int(v) for v in g.choice(nv, int(g.integers(2, 9)), replace=False)]
        ds = np.array([sizes[v] for v in scope])
        t = int(round(math.exp(g.uniform(math.log(1e3), math.log(case["tuples"])))))
        u = g.random((t, len(scope)))
        spec.tables.append(G.TableSpec(scope, ((u if k % 2 == 0 else u * u) * ds).astype(np.int32)))
    return spec


def _random_spec(case, seed):
    g = np.random.default_rng(seed)
    nv, d = case["vars"], case["dom"]
    spec = G.CspSpec(nvars=nv, dom_lo=[0] * nv, dom_size=[d] * nv)
    for _ in range(case["tables"]):
        scope = [int(v) for v in g.choice(nv, case["arity"], replace=False)]
        spec.tables.append(G.TableSpec(scope, g.integers(0, d, (case["tuples"], case["arity"]), dtype=np.int32)))
    return spec


def _order_spec(case, seed):
    """An instance of the learned-order family (tables of arity 3-4, 1e3-2e4 tuples)."""
    d = case["dom"]
    return G.learned_csp(seed, nvars=(case["vars"],) * 2, dom=(max(2, d // 2), d), ntables=(case["tables"],) * 2,
                         arity=(3, 4), tuples=(1e3, case.get("tuples", 2e4)),
                         log2_solutions=float(case.get("log2_solutions", 4)))


def _prepare_cuts(case, seed, spec):
    """A network at its root fixpoint, and for every call the domains of a node: a few variables cut."""
    own = _model(spec)
    st = C.check(C.ct_model_propagate(own.h))
    nwords = int(C.dom_layout(spec.dom_size)[0][-1])
    if st == C.CT_INFEASIBLE:
        raise RuntimeError("the network has no solution at its root")
    _, root = C.ct_model_get_domains(own.h, nwords)
    rng, cuts = G.Rng(seed), []
    masks = C.words_to_masks(root, spec.dom_size)
    for _ in range(case["calls"]):
        new = masks
        for _ in range(max(1, spec.nvars // 100)):
            new = _edit(rng, new)
        cuts.append(C.masks_to_words(new))
    return {"own": own, "cuts": cuts, "nwords": nwords, "nvars": spec.nvars}


def _run_cuts(s, features):
    m, domains, status, feats = s["own"].h, [], [], []
    for cut in s["cuts"]:
        st, level = C.ct_model_save(m)
        C.check(st)
        C.check(C.ct_model_set_domains(m, cut))
        st = C.check(C.ct_model_propagate(m))
        status.append(st)
        if st == C.CT_OK:
            domains.append(C.ct_model_get_domains(m, s["nwords"])[1])
            if features:
                st, f = C.ct_model_features(m, s["nvars"])
                C.check(st)
                feats.append(f)
        else:
            domains.append(np.zeros(s["nwords"], np.uint32))
            if features:
                feats.append(np.zeros((s["nvars"], C.MLP_FEATURES), np.float32))
        C.check(C.ct_model_restore(m, level))
    out = {"domains": np.stack(domains), "status": np.array(status)}
    if features:
        out["features"] = np.stack(feats)
    return out


def _counts(d):
    return {"counts": np.array([d["nodes"], d["fails"], d["solutions"], d["max_depth"], d["complete"]]),
            "first": np.array(d["first_solution"] if d["first_solution"] is not None else [], np.int64)}


def _train_data(case, seed):
    """Samples as the collection makes them: features of [0, 1] size, a label that mostly follows them."""
    g = np.random.default_rng(seed)
    X = g.random((case["samples"], 8)).astype(np.float32)
    y = (0.6 * X[:, 0] * X[:, 3] + 0.3 * np.maximum(0, X[:, 5] - X[:, 4]) + 0.05 * g.random(len(X))).astype(np.float32)
    orders = np.stack([g.permutation(len(X)).astype(np.int32) for _ in range(case["epochs"])])
    return X, y, G.mlp_init_weights(seed), orders


def _prepare_train(case, seed):
    X, y, w, orders = _train_data(case, seed)
    st, net = C.ct_mlp_create(w, stream=torch.cuda.current_stream())
    C.check(st)
    return {"own": Owned(net, C.ct_mlp_destroy), "X": X, "y": y, "w": w, "orders": orders, "batch": case["batch"],
            "dev": torch.from_numpy(X).cuda(), "scores": torch.zeros(len(X), device="cuda")}


def _run_train(s):
    m = s["own"].h
    C.check(C.ct_mlp_set_weights(m, s["w"]))
    st, losses = C.ct_mlp_train(m, s["X"], s["y"], s["orders"], s["batch"], 1e-3)
    C.check(st)
    C.check(C.ct_mlp_forward(m, s["dev"], len(s["X"]), s["scores"]))
    st, w = C.ct_mlp_get_weights(m)
    C.check(st)
    return {"weights": w, "losses": losses, "scores": s["scores"]}


def prepare(case, seed):
    k = case["kind"]
    if k == "stream":
        s = _prepare_stream(case, seed)
    elif k == "bulk":
        s = _prepare_bulk(case, seed)
    elif k == "build":
        s = _prepare_build(case, seed)
    elif k == "network":
        s = _prepare_cuts(case, seed, _network_spec(case, seed))
    elif k == "features":
        s = _prepare_cuts(case, seed, _order_spec(case, seed))
    elif k == "dfs":
        s = {"own": _model(_random_spec(case, seed)), "nvars": case["vars"]}
    elif k == "device":
        s = {"own": _model(_order_spec(case, seed)), "nvars": case["vars"]}
    else:
        s = _prepare_train(case, seed)
    s.update(kind=k, case=dict(case))
    return s


def run(s):
    k, case = s["kind"], s["case"]
    if k == "stream":
        return _run_stream(s)
    if k == "bulk":
        return _run_bulk(s)
    if k == "build":
        return _run_build(s)
    if k in ("network", "features"):
        return _run_cuts(s, k == "features")
    if k == "dfs":
        st, d = C.ct_search_dfs(s["own"].h, s["nvars"], case["nodes"], True)
        C.check(st)
        return _counts(d)
    if k == "device":
        st, d, _ = C.ct_search_batch_device(s["own"].h, s["nvars"], case["slots"], case["split"])
        C.check(st)
        return _counts(d)
    return _run_train(s)


def work(case):
    """Bytes that the path cannot do without. One supports row or currTable of a
    table is t / 8 bytes. An update reads the rows of the removed or remaining
    values and currTable and writes it; of a stream's calls, half remove one or
    two values and half keep about a quarter of a domain, on a table of which
    about half is still live on average."""
    k = case["kind"]
    if k in ("stream", "bulk", "build"):
        row, rows = case["tuples"] / 8, case["arity"] * case["dom"]
    if k == "stream":
        return {"bytes": case["calls"] * (0.5 * row * (2 + 0.75 + case["dom"] / 8) + 8 * rows / 32 + 4 * rows),
                "flops": 0}
    if k == "bulk":
        return {"bytes": case["calls"] * row * (2 + case["arity"] * case["keep"]), "flops": 0}
    if k == "build":  # the tuples in, the rows and currTable out, and the first propagation's
        return {"bytes": 4.0 * case["tuples"] * case["arity"] + row * (rows + 1) + row * (2 + rows / 4), "flops": 0}
    if k == "network":  # the tables of the cut variables: a few rows of each
        return {"bytes": case["calls"] * max(1, case["vars"] // 100) * 2.5 * 4 * case["tuples"] / 8 / 4.6, "flops": 0}
    if k == "features":  # every row of every table at a third of its tuples live, and currTable
        return {"bytes": case["calls"] * case["tables"] * (3.5 * case["dom"] + 1) * case["tuples"] / 8 / 3, "flops": 0}
    if k == "dfs":  # about two tables of a node's change, by a few rows each
        return {"bytes": case["nodes"] * 2 * 6 * case["tuples"] / 8, "flops": 0}
    if k == "device":  # some 15,000 nodes at one expected solution, six rows of about six tables in each
        return {"bytes": 15_000 * 2.0 ** (case["log2_solutions"] / 4) * 6 * 6 * 5_000 / 8, "flops": 0}
    n, w = case["samples"], 8 * 64 + 64 * 64 + 64
    return {"bytes": 4.0 * n * (8 + 1 + 1 + case["epochs"]), "flops": 2.0 * n * w * (3 * case["epochs"] + 1)}


# --------------------------------------------------------------------------
# the floating-point results in 64 bits
# --------------------------------------------------------------------------
def _exact_train(case, seed):
    X, y, w, orders = _train_data(case, seed)
    X, y, w = X.astype(np.float64), y.astype(np.float64), w.astype(np.float64)
    cut = np.cumsum([64 * 8, 64, 64 * 64, 64, 64])
    shapes = [(64, 8), (64,), (64, 64), (64,), (64,), (1,)]
    P = [p.reshape(s).copy() for p, s in zip(np.split(w, cut), shapes)]
    M, V = [np.zeros_like(p) for p in P], [np.zeros_like(p) for p in P]

    def forward(x):
        h1 = np.maximum(x @ P[0].T + P[1], 0)
        h2 = np.maximum(h1 @ P[2].T + P[3], 0)
        return h1, h2, h2 @ P[4] + P[5][0]

    step, losses, lr = 0, [], float(np.float32(1e-3))
    for order in orders:
        part = []
        for i in range(0, len(order), case["batch"]):
            b = order[i:i + case["batch"]]
            h1, h2, out = forward(X[b])
            r = out - y[b]
            part.append(float((r * r).sum() / (2 * len(b))))
            do = r / len(b)
            d2 = do[:, None] * P[4] * (h2 > 0)
            d1 = (d2 @ P[2]) * (h1 > 0)
            g = [d1.T @ X[b], d1.sum(0), d2.T @ h1, d2.sum(0), do @ h2, np.array([do.sum()])]
            step += 1
            for p, m, v, q in zip(P, M, V, g):
                m += 0.1 * (q - m)
                v += 0.001 * (q * q - v)
                p -= lr * (m / (1 - 0.9 ** step)) / (np.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
        losses.append(sum(part) / len(part))
    return {"weights": np.concatenate([p.reshape(-1) for p in P]), "losses": np.array(losses), "scores": forward(X)[2]}


def _project(spec, masks):
    """The common fixpoint of a network by projections of the valid tuples; None if a table has none."""
    masks = [m.copy() for m in masks]
    while True:
        valid, changed = [], False
        for tb in spec.tables:
            ok = np.ones(len(tb.tuples), bool)
            for i, v in enumerate(tb.scope):
                ok &= masks[v][tb.tuples[:, i]]
            if not ok.any():
                return None, None
            valid.append(ok)
            for i, v in enumerate(tb.scope):
                new = np.zeros_like(masks[v])
                new[tb.tuples[ok, i]] = True
                new &= masks[v]
                if new.sum() != masks[v].sum():
                    masks[v], changed = new, True
        if not changed:
            return masks, valid


def _exact_features(case, seed):
    spec = _order_spec(case, seed)
    deg = np.zeros(spec.nvars)
    for tb in spec.tables:
        deg[tb.scope] += 1
    root, _ = _project(spec, [np.ones(d, bool) for d in spec.dom_size])
    rng, feats = G.Rng(seed), []
    for _ in range(case["calls"]):
        new = root
        for _ in range(max(1, spec.nvars // 100)):
            new = _edit(rng, new)
        masks, valid = _project(spec, new)
        f = np.zeros((spec.nvars, 8))
        feats.append(f)
        if masks is None:
            continue
        s = np.array([m.sum() for m in masks], np.float64)
        per = [[] for _ in masks]
        for tb, ok in zip(spec.tables, valid):
            live = float(ok.sum())
            for i, v in enumerate(tb.scope):
                p = np.bincount(tb.tuples[ok, i], minlength=spec.dom_size[v])[masks[v]] / live
                q = p[p > 0]
                per[v].append((s[v] * p.min(), p.max(), -(q * np.log2(q)).sum(), np.log2(1 + live) / 32))
        for v in range(spec.nvars):
            if s[v] < 2:
                continue
            a = np.array(per[v]).mean(0) if per[v] else np.zeros(4)
            f[v] = [s[v] / spec.dom_size[v], np.log2(s[v]) / 8, deg[v] / max(1, deg.max()), a[0], a[1],
                    a[2] / np.log2(s[v]), a[3], s[v] / s[s > 1].max()]
    return {"domains": None, "status": None, "features": np.stack(feats)}


def exact(case, seed):
    """Only the learned order computes with floating-point numbers; domains,
    tables and counts are whole numbers that either are the fixpoint's or are wrong."""
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "features":
        return _exact_features(case, seed)
    return None
