"""The work that a user of the race checker has it do, as measurable cases.

A case is one pass through the public entry points: the models (or keys) are
created, uploaded and given a workspace in ``prepare``, as a program does that
checks a kernel model more than once; ``run`` enqueues the check and reads its
result.  Models come from the repository's own seeded generators.  Another seed
is another model of the same size: for the random affine models the generator
seeds are tried in order until one has the stated number of access instances
per thread (within 3 %).
"""
import math
import random

import numpy as np
import torch

import paper_2503_08946_gb300 as rc
import workloads as w
from paper_2503_08946_gb300.binding import RC_OPT_GRAPH


def listed():
    return [
        # the tree reduction of the documentation: one block of 256 threads, 765
        # instances; the latency of the smallest useful check
        {"name": "reduction_256", "kind": "reduction", "threads": 256},
        # the tiled transposition, 2048 x 2048 in 32 x 32 tiles (16.8 M instances),
        # padded or not, with or without its barrier (by the seed)
        {"name": "transpose_2048", "kind": "transpose", "n": 2048},
        # the benchmark's model: 1 M threads, 36 statements, about 1e9 instances
        {"name": "affine_4096x256", "kind": "affine", "blocks": 4096, "block": 256, "tail": 0, "stmts": 36,
         "per_thread": 1000, "plant": False},
        # a middle-sized model of odd sizes with a planted race: 777 blocks of 192
        # threads of which the last 101 are guarded off
        {"name": "affine_777x192_racy", "kind": "affine", "blocks": 777, "block": 192, "tail": 101, "stmts": 24,
         "per_thread": 650, "plant": True},
        # one rank's share of a model split over eight ranks by hash part
        {"name": "affine_part_1of8", "kind": "part", "blocks": 1024, "block": 256, "tail": 0, "stmts": 36,
         "per_thread": 1000, "plant": False, "parts": 8},
        # a sparse address space (rows of 2^24 cells): keys wider than 63 bits, checked
        # in cell-range chunks
        {"name": "affine_wide", "kind": "wide", "blocks": 512, "block": 256, "tail": 0, "stmts": 36,
         "per_thread": 1000, "plant": False, "row_bits": 24},
        # the paper's Ge-SpMM on a CSR matrix of skewed row lengths: data-dependent
        # loop bounds, ten barrier intervals
        {"name": "spmm_csr", "kind": "spmm", "rows": 2048, "cols": 256, "k": 8, "max_len": 150},
        # the same with rows of up to 600 non-zeros: 38 barrier intervals
        {"name": "spmm_csr_long_rows", "kind": "spmm", "rows": 512, "cols": 128, "k": 4, "max_len": 600},
        # per-block atomic histograms, read back after a barrier or in the same interval
        {"name": "atomic_histogram", "kind": "histogram", "threads": 256, "bins": 64, "blocks": 16384},
        # thousands of small models of uneven size checked as one batch, the captured graph replayed
        {"name": "batch_2000", "kind": "batch", "models": 2000, "graph": True},
        # what a server admits at once: two dozen small models, a new batch each time
        {"name": "batch_24", "kind": "batch", "models": 24, "graph": False},
        # the stable radix sort alone, on the 30 cell bits of 54-bit keys
        {"name": "sort_keys", "kind": "sort", "n": 20000003, "lo": 24, "hi": 54},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["affine", "affine", "affine", "transpose", "reduction", "part", "wide", "spmm", "spmm",
                       "histogram", "batch", "batch", "sort"])
    if kind in ("affine", "part", "wide"):
        block = rng.choice([32, 64, 96, 128, 160, 192, 224, 256, 320, 500, 512])
        top = {"affine": 1 << 20, "part": 1 << 18, "wide": 1 << 17}[kind]
        low = 1 if kind == "affine" else 32
        blocks = min(_log_int(rng, low, top // block), top // block)
        stmts = rng.randint(12, 36)
        c = {"kind": kind, "blocks": blocks, "block": block, "tail": rng.choice([0, 0, rng.randint(1, block - 1)]),
             "stmts": stmts, "per_thread": int(27 * stmts), "plant": rng.random() < 0.3}
        if kind == "part":
            c["parts"] = rng.choice([2, 4, 8, 16])
        if kind == "wide":
            # rows long enough that the packed key needs 64 to 67 bits
            other = 4 + (blocks - 1).bit_length() + (block - 1).bit_length()
            c["row_bits"] = 63 + rng.randint(0, 3) - other - (blocks * block - c["tail"]).bit_length()
        return c
    if kind == "transpose":
        return {"kind": kind, "n": 32 * _log_int(rng, 2, 100)}
    if kind == "reduction":
        return {"kind": kind, "threads": 1 << rng.choice([5, 6, 7, 9, 10])}
    if kind == "spmm":
        rows = _log_int(rng, 8, 2048)
        return {"kind": kind, "rows": rows, "cols": 32 * rng.randint(1, 8), "k": rng.randint(1, 8),
                "max_len": rng.choice([40, 100, 150, 250, 400]) if rows > 512 else rng.choice([100, 250, 400, 600])}
    if kind == "histogram":
        return {"kind": kind, "threads": 32 * rng.randint(1, 16), "bins": rng.randint(3, 200),
                "blocks": _log_int(rng, 1, 16384)}
    if kind == "batch":
        return {"kind": kind, "models": _log_int(rng, 2, 2000), "graph": rng.random() < 0.5}
    lo = rng.choice([0, 7, 16, 24])
    return {"kind": "sort", "n": _log_int(rng, 1000, 60000000), "lo": lo, "hi": lo + rng.randint(9, 34)}


def _per_thread(model):
    n = 0
    for s in model.stmts:
        p = len(s.accesses)
        for lp in s.loops:
            p *= lp.upper.args[0]
        n += p
    return n


def _affine(case, seed):
    """The first random affine model of the seeds from ``seed`` on whose
    instances per thread are within 3 % of the case's (the nearest of 200)."""
    best = None
    for k in range(200):
        s = (seed * 200 + k) & 0x7FFFFFFF
        m = w.random_affine(s, n_blocks=1, block=case["block"], n_stmts=case["stmts"], plant=case["plant"])
        off = abs(_per_thread(m) / case["per_thread"] - 1)
        if best is None or off < best[0]:
            best = (off, s)
        if off <= 0.03:
            break
    threads = case["blocks"] * case["block"]
    return w.random_affine(best[1], n_blocks=case["blocks"], block=case["block"], n_stmts=case["stmts"],
                           plant=case["plant"], n_threads=threads - case["tail"] if case["tail"] else None,
                           row_global=1 << case["row_bits"] if "row_bits" in case else 256)


def _models(case, seed):
    kind = case["kind"]
    if kind in ("affine", "part", "wide"):
        return [_affine(case, seed)]
    if kind == "transpose":
        return [w.transpose(pad=bool(seed & 2), barrier=bool(seed & 1), n=case["n"])]
    if kind == "reduction":
        return [w.reduction_tree(barriers=bool(seed & 1), T=case["threads"])]
    if kind == "spmm":
        return [w.ge_spmm_csr(w.csr_row_lengths(seed, case["rows"], max_len=case["max_len"]), N=case["cols"],
                              K=case["k"], trailing_barrier=bool(seed & 1))]
    if kind == "histogram":
        return [w.atomic_histogram(case["threads"], case["bins"], n_blocks=case["blocks"], barrier=bool(seed & 1))]
    return w.batch_models(case["models"], seed0=(seed & 0xFFFF) * 100003)


def prepare(case, seed):
    if case["kind"] == "sort":
        # keys as an expansion writes them: random cells above, random threads below
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["n"]
        keys = torch.randint(0, 1 << 54, (n,), generator=g, device="cuda", dtype=torch.int64)
        return {"kind": "sort", "keys": keys, "out": torch.empty_like(keys), "n": n, "lo": case["lo"],
                "hi": case["hi"], "ws": rc.workspace(rc.rc_sort_workspace_size(n))}
    models = [rc.rc_model_create(m) for m in _models(case, seed)]
    opts = None
    if case["kind"] == "part":
        opts = {"part_count": case["parts"], "part_index": random.Random(seed).randrange(case["parts"])}
    if case["kind"] == "batch":
        opts = {"flags": RC_OPT_GRAPH} if case["graph"] else None
        size = rc.rc_batch_workspace_size(models, opts)
    else:
        size = rc.rc_workspace_size(models[0], opts)
    return {"kind": case["kind"], "models": models, "opts": opts, "ws": rc.workspace(size)}


def run(state):
    if state["kind"] == "sort":
        rc.rc_sort_keys(state["keys"], state["out"], state["n"], state["lo"], state["hi"], 0, state["ws"])
        return state["out"]
    if state["kind"] == "batch":
        ticket = rc.rc_check_batch(state["models"], state["opts"], state["ws"])
        # the result records, byte for byte
        return np.frombuffer(rc.rc_report_array(ticket).tobytes(), dtype=np.uint8)
    r = rc.rc_report(rc.rc_check(state["models"][0], state["opts"], state["ws"]))[0]
    return {"status": r.status, "verdict": r.verdict, "racy_cells": r.racy_cells, "instances": r.instances,
            "cell": [r.w_array, r.w_scope, r.w_addr], "x": list(r.x), "y": list(r.y)}


def work(case):
    """A check reads the lowered program and writes one result record (the keys
    in between are the method's own); every instance costs about ten integer
    operations: its index, its bounds, its cell and its part in the cell's
    verdict.  A sort reads and writes every key once."""
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 16.0 * case["n"], "flops": 2.0 * case["n"]}
    if kind in ("affine", "part", "wide"):
        inst = (case["blocks"] * case["block"] - case["tail"]) * case["per_thread"]
        return {"bytes": 28000.0 + 256, "flops": 10.0 * inst}
    if kind == "batch":
        # log-uniform thread counts in 32..65536, 4.5 statements of one access
        inst = case["models"] * 4.5 * (65536 - 32) / math.log(65536 / 32)
        return {"bytes": case["models"] * (4000.0 + 256), "flops": 10.0 * inst}
    if kind == "transpose":
        return {"bytes": 2000.0 + 256, "flops": 10.0 * 4 * case["n"] ** 2}
    if kind == "reduction":
        return {"bytes": 4000.0 + 256, "flops": 10.0 * 3 * (case["threads"] - 1)}
    if kind == "histogram":
        return {"bytes": 1000.0 + 256, "flops": 10.0 * 2 * case["threads"] * case["blocks"]}
    lens = w.csr_row_lengths(0, case["rows"], max_len=case["max_len"])
    inst = case["cols"] * sum(2 + 4 * n / 32 + (4 + case["k"]) * n for n in lens)
    return {"bytes": 8.0 * case["rows"] + 4000 + 256, "flops": 10.0 * inst}


def exact(case, seed):
    """The closed forms of the generators (verdict and number of racy cells), and
    the stable sort; no value for the other outputs."""
    kind = case["kind"]
    if kind == "sort":
        g = torch.Generator(device="cuda").manual_seed(seed)
        keys = torch.randint(0, 1 << 54, (case["n"],), generator=g, device="cuda", dtype=torch.int64)
        field = (keys >> case["lo"]) & ((1 << (case["hi"] - case["lo"])) - 1)
        return keys[torch.sort(field, stable=True).indices]
    racy = None
    if kind == "reduction":
        racy = 0 if seed & 1 else case["threads"] // 2 - 1
    elif kind == "transpose":
        racy = 0 if seed & 1 else 992 * (case["n"] // 32) ** 2
    elif kind in ("affine", "wide"):
        threads = case["blocks"] * case["block"] - case["tail"]
        racy = threads if case["plant"] and threads > 1 else 0
    elif kind == "histogram":
        racy = 0 if seed & 1 or case["threads"] < 2 * case["bins"] else case["blocks"] * case["bins"]
    if racy is None:
        return None
    return {"status": 0, "verdict": int(racy > 0), "racy_cells": racy, "instances": None, "cell": None, "x": None,
            "y": None}
