"""The work this library is used for, as cases that can be timed and compared.

A proof system that commits to an execution trace extends the trace (NTT,
LDE), hashes its rows into Merkle trees, and answers queries with
authentication paths.  Each case below is one such call through the public
binding, at sizes from the benchmark's workloads and the tests: trees of 2^10
to 2^22 leaves and widths that are and are not multiples of the sponge's eight
words, batches of trees, rows in host memory, raw permutations, row digests,
path queries, transforms both ways and the low-degree extension.

All values are 64-bit field words; results are exact residues, so two
implementations agree bit for bit.
"""
import random

import torch

import paper_2506_09505_gb300 as pg

# 32-bit multiply results of one width-12 permutation (118 S-boxes of two
# squares and two products, eight 12x12 matrices, 22 sparse rounds), and of one
# radix-2 butterfly (one field product).
PERM_MULS = 16568
BUTTERFLY_MULS = 8
# a drawn case costs at most about as much as the largest listed one
MAX_PERMS = 1 << 23
MAX_WORDS = 1 << 25


def listed():
    return [
        # the smallest commitment in the benchmark: a chain of eleven tree levels, all latency
        {"name": "tree_2e10x8", "kind": "tree", "log_n": 10, "width": 8},
        # a mid-sized trace with an odd number of columns (rows not 16-byte aligned, last chunk ragged)
        {"name": "tree_2e15x13", "kind": "tree", "log_n": 15, "width": 13},
        # the headline: the paper's 2^22 leaves of eight columns, rows on the device
        {"name": "tree_2e22x8", "kind": "tree", "log_n": 22, "width": 8},
        # wide rows: the sponge over eight chunks dominates
        {"name": "tree_2e20x64", "kind": "tree", "log_n": 20, "width": 64},
        # the same commitment end to end, rows arriving from page-locked host memory
        {"name": "host_2e22x8", "kind": "host", "log_n": 22, "width": 8},
        # a prover's trees of mixed sizes and widths in one call
        {"name": "batch_24", "kind": "batch", "trees": 24, "lo": 12, "hi": 18, "shapes": 4, "graph": False},
        # many small trees, captured once and replayed (a served stream of small proofs)
        {"name": "graph_32_small", "kind": "batch", "trees": 32, "lo": 8, "hi": 12, "shapes": 5, "graph": True},
        # raw permutations, an odd number of states
        {"name": "permute_4000037", "kind": "permute", "n": 4000037},
        # digests of a ragged matrix: neither rows nor columns fill a tile
        {"name": "rows_100003x21", "kind": "rows", "n": 100003, "width": 21},
        # the query phase: open and check paths in a 2^20-leaf tree
        {"name": "query_2e20_k1021", "kind": "query", "log_n": 20, "k": 1021},
        # interpolation of a few columns (inverse transform, an odd column count)
        {"name": "intt_2e16x3", "kind": "ntt", "log_n": 16, "cols": 3, "inverse": True},
        # the benchmark's trace extension, 2^21 rows of eight columns to twice as many
        {"name": "lde_2e21x8", "kind": "lde", "log_n": 21, "cols": 8, "blowup": 1},
    ]


def _log_uniform(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def _tree_perms(n, width):
    return n * ((width + 7) // 8) + n - 1


def draw(rng):
    kind = rng.choice(["tree", "tree", "tree", "host", "batch", "permute", "rows", "query", "ntt", "ntt", "lde"])
    if kind in ("tree", "host"):
        while True:
            log_n, width = rng.randint(4 if kind == "tree" else 14, 22), _log_uniform(rng, 1, 256)
            if _tree_perms(1 << log_n, width) <= MAX_PERMS and (width << log_n) <= 2 * MAX_WORDS:
                return {"kind": kind, "log_n": log_n, "width": width}
    if kind == "batch":
        while True:
            lo = rng.randint(0, 14)
            case = {"kind": "batch", "trees": _log_uniform(rng, 2, 64), "lo": lo, "hi": rng.randint(lo, 18),
                    "shapes": rng.randrange(1 << 20), "graph": rng.random() < 0.5}
            if sum(_tree_perms(1 << k, w) for k, w in _shapes(case)) <= MAX_PERMS:
                return case
    if kind == "permute":
        return {"kind": kind, "n": _log_uniform(rng, 1, 4000037)}
    if kind == "rows":
        width = _log_uniform(rng, 1, 256)
        return {"kind": kind, "n": _log_uniform(rng, 1, MAX_PERMS // ((width + 7) // 8 * 2)), "width": width}
    if kind == "query":
        return {"kind": kind, "log_n": rng.randint(1, 20), "k": _log_uniform(rng, 1, 20000)}
    if kind == "ntt":
        log_n = rng.randint(1, 21)
        cols = _log_uniform(rng, 1, min(100, MAX_WORDS >> log_n))
        return {"kind": kind, "log_n": log_n, "cols": cols, "inverse": rng.random() < 0.5}
    log_n, blowup = rng.randint(1, 20), rng.randint(0, 3)
    while log_n + blowup > 22:
        blowup -= 1
    cols = _log_uniform(rng, 1, min(100, MAX_WORDS >> (log_n + blowup)))
    return {"kind": "lde", "log_n": log_n, "cols": cols, "blowup": blowup}


def _shapes(case):
    """(log2 leaves, width) of each tree of a batch."""
    rng = random.Random(case["shapes"])
    return [(rng.randint(case["lo"], case["hi"]), rng.choice((8, 16, 32, 64, 8, 12, 5)))
            for _ in range(case["trees"])]


def _words(gen, rows, cols):
    """Uniform 64-bit words (one in 2^32 is not below the modulus; the library reads any word mod p)."""
    return torch.randint(-2**63, 2**63 - 1, (rows, cols), dtype=torch.int64, device="cuda", generator=gen)


def prepare(case, seed):
    pg.init(0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "tree":
        state["rows"] = _words(gen, 1 << case["log_n"], case["width"])
    elif kind == "host":
        rows = _words(gen, 1 << case["log_n"], case["width"])
        state["host"] = rows.cpu().pin_memory()
        state["staging"] = rows.zero_()
        state["nodes"] = torch.empty(((2 << case["log_n"]) - 1, 4), dtype=torch.int64, device="cuda")
    elif kind == "batch":
        state["rows"] = [_words(gen, 1 << k, w) for k, w in _shapes(case)]
        if case["graph"]:
            state["graph"] = pg.BatchGraph(state["rows"])
        else:
            state["nodes"] = pg.alloc_nodes(state["rows"])
    elif kind == "permute":
        state["states"] = _words(gen, case["n"], 12)
    elif kind == "rows":
        state["rows"] = _words(gen, case["n"], case["width"])
    elif kind == "query":
        n = 1 << case["log_n"]
        state["n"] = n
        state["nodes"] = pg.merkle_build(_words(gen, n, 8))
        state["indices"] = torch.randint(0, n, (case["k"],), dtype=torch.int64, device="cuda", generator=gen)
        state["leaves"] = state["nodes"][state["indices"]].contiguous()
        state["root"] = state["nodes"][-1].contiguous()
    elif kind == "ntt":
        state["data"] = _words(gen, 1 << case["log_n"], case["cols"])
        state["inverse"] = case["inverse"]
    else:
        state["evals"] = _words(gen, 1 << case["log_n"], case["cols"])
        state["blowup"] = case["blowup"]
    torch.cuda.synchronize()
    return state


def run(state):
    kind = state["kind"]
    if kind == "tree":
        return pg.merkle_build(state["rows"])
    if kind == "host":
        return pg.merkle_build_host(state["host"], state["staging"], state["nodes"])
    if kind == "batch":
        if "graph" in state:
            return state["graph"].launch()
        return pg.merkle_build_batch(state["rows"], state["nodes"])
    if kind == "permute":  # in place; the caller keeps its input
        return pg.permute_batch(state["states"].clone())
    if kind == "rows":
        return pg.hash_rows(state["rows"])
    if kind == "query":
        paths = pg.merkle_open(state["nodes"], state["n"], state["indices"])
        ok = pg.merkle_verify(state["root"], state["n"], state["leaves"], state["indices"], paths)
        return [paths, ok]
    if kind == "ntt":  # in place; the caller keeps its input
        return pg.ntt(state["data"].clone(), inverse=state["inverse"])
    return pg.lde(state["evals"], state["blowup"])


def _tree_work(n, width):
    return 8 * n * width + 32 * (2 * n - 1), _tree_perms(n, width) * PERM_MULS


def work(case):
    kind = case["kind"]
    if kind in ("tree", "host"):
        b, f = _tree_work(1 << case["log_n"], case["width"])
    elif kind == "batch":
        parts = [_tree_work(1 << k, w) for k, w in _shapes(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "permute":
        b, f = 2 * 96 * case["n"], case["n"] * PERM_MULS
    elif kind == "rows":
        b = case["n"] * (8 * case["width"] + 32)
        f = case["n"] * ((case["width"] + 7) // 8) * PERM_MULS
    elif kind == "query":
        steps = case["k"] * case["log_n"]
        # siblings read and the paths written; leaves, indices, verdicts; one permutation a step
        b, f = 2 * 32 * steps + case["k"] * (32 + 8 + 1) + 32, steps * PERM_MULS
    elif kind == "ntt":
        n = 1 << case["log_n"]
        b, f = 16 * n * case["cols"], n // 2 * case["log_n"] * case["cols"] * BUTTERFLY_MULS
    else:
        n, big = 1 << case["log_n"], 1 << (case["log_n"] + case["blowup"])
        b = 8 * (n + big) * case["cols"]
        f = (n + big) // 2 * case["log_n"] * case["cols"] * BUTTERFLY_MULS
    return {"bytes": b, "flops": f}


def exact(case, seed):
    """Outputs are whole field words: equal or wrong, with no rounding to measure."""
    return None
