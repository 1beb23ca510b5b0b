"""The work that users of this framework have it do, as cases that can be timed.

Each case is one call (or one burst of calls) of a public entry point of
paper_2403_00306_gb300 on instances of the planted-motif model: n i.i.d. uniform sequences of
length m, one random l-mer planted in each with exactly d substitutions. The sizes are those of
the repository's own benchmark (plain, quorum and protein configurations, the batch, the request
stream) and the ranges around them.

A program that uses the library keeps a context for as long as it runs and passes it new
sequences, so the contexts are made once per kind of call and a state holds the sequences (and,
for the device entry point, the output buffers).
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2403_00306_gb300 as pms

CAPACITY = 1 << 16   # motif codes a device caller has room for

#: (l, d) of the benchmark's DNA workloads: plain, batched and served
DNA_LD = ((9, 2), (11, 3), (13, 4), (15, 4), (17, 5), (19, 6))
BATCH_LD = ((11, 3), (13, 4), (15, 4))
SERVED_LD = ((13, 4), (15, 4), (17, 5))


def listed():
    return [
        # the smallest plain configuration: launches and latency are most of it
        {"name": "device_9_2", "call": "device", "l": 9, "d": 2, "n": 20, "m": 600},
        # the flagship plain configuration, data already on the device
        {"name": "device_15_4", "call": "device", "l": 15, "d": 4, "n": 20, "m": 600},
        # the larger plain configurations: long motifs, many tree nodes per seed
        {"name": "device_17_5", "call": "device", "l": 17, "d": 5, "n": 20, "m": 600},
        {"name": "device_19_6", "call": "device", "l": 19, "d": 6, "n": 20, "m": 600},
        # long sequences in which chance occurrences are common: the heavy class of the batch and the stream
        {"name": "device_13_4_long", "call": "device", "l": 13, "d": 4, "n": 20, "m": 1000},
        # a one-off call on host memory, result back on the host
        {"name": "host_15_4", "call": "host", "l": 15, "d": 4, "n": 20, "m": 600},
        # odd sizes from host memory (a sequence set as it comes, not padded to anything)
        {"name": "host_11_3_ragged", "call": "host", "l": 11, "d": 3, "n": 17, "m": 733},
        # noisy data: a motif need only occur in half of the sequences
        {"name": "quorum_15_4_q10", "call": "quorum", "l": 15, "d": 4, "n": 20, "m": 600, "q": 10},
        # protein sequences (20 letters), a quick and a heavy setting
        {"name": "protein_9_3", "call": "protein", "l": 9, "d": 3, "n": 20, "m": 600},
        {"name": "protein_9_4", "call": "protein", "l": 9, "d": 4, "n": 20, "m": 600},
        # throughput: 256 mixed instances in one call
        {"name": "batch_256", "call": "batch", "count": 256},
        # a service under load: 64 requests of the stream's mix submitted at once, each waited for
        {"name": "served_64", "call": "served", "count": 64},
    ]


def draw(rng):
    call = rng.choice(("device", "device", "host", "quorum", "protein", "batch", "served"))
    if call in ("batch", "served"):
        return {"call": call, "count": _spread(rng, 8, 128 if call == "batch" else 64)}
    n, m = rng.randint(10, 30), _spread(rng, 200, 1200)
    if call == "protein":
        l, d = rng.choice(((9, 3), (9, 3), (9, 4), (11, 4)))
        return {"call": call, "l": l, "d": d, "n": min(n, 22), "m": min(m, 600)}
    if call == "quorum":
        l, d = rng.choice(((15, 4), (15, 4), (13, 4)))
        n, m = (min(n, 20), min(m, 600)) if l == 15 else (n + 8, min(m, 500))
        q = rng.randint(n // 2, n - 1)
        while q < n - 1 and _chance_motifs(l, d, n, m, q) > CAPACITY / 8:
            q += 1
        return {"call": call, "l": l, "d": d, "n": n, "m": m, "q": q}
    l, d = rng.choice(DNA_LD)
    # enough sequences that chance motifs fit the caller's buffer
    while _chance_motifs(l, d, n, m) > CAPACITY / 8:
        n += 1
    return {"call": call, "l": l, "d": d, "n": n, "m": m}


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ball(l, d, sigma=4):
    return sum(math.comb(l, k) * (sigma - 1) ** k for k in range(d + 1))


def _chance_motifs(l, d, n, m, q=None):
    """Strings expected within d of some window of each of n random sequences (of q of them)."""
    p = 1.0 - math.exp(-(m - l + 1) * _ball(l, d) / 4.0 ** l)
    return 4.0 ** l * sum(math.comb(n, k) * p ** k * (1 - p) ** (n - k) for k in range(q or n, n + 1))


# ------------------------------------------------------------------ inputs

def _planted(rng, letters, n, m, l, d):
    codes = rng.integers(0, len(letters), (n, m))
    motif = rng.integers(0, len(letters), l)
    at = rng.integers(0, m - l + 1, n)
    for i in range(n):
        copy = motif.copy()
        where = rng.permutation(l)[:d]
        copy[where] = (copy[where] + rng.integers(1, len(letters), d)) % len(letters)
        codes[i, at[i]:at[i] + l] = copy
    return np.ascontiguousarray(letters[codes])


_DNA = np.frombuffer(b"ACGT", dtype=np.uint8)
_AMINO = np.frombuffer(pms.PROTEIN, dtype=np.uint8)


def _shapes(case):
    """(l, d, n, m, q) of every instance of the case; those of a batch or a burst are the same mix for every seed."""
    if case["call"] not in ("batch", "served"):
        return [(case["l"], case["d"], case["n"], case["m"], case.get("q", case["n"]))]
    rng = np.random.default_rng(case["count"])
    got = []
    for k in range(case["count"]):
        if case["call"] == "batch":
            l, d = BATCH_LD[rng.integers(len(BATCH_LD))]
            n, m = int(rng.integers(10, 31)), int(rng.integers(300, 1001))
        else:
            l, d = SERVED_LD[rng.integers(len(SERVED_LD))]
            n, m = 20, int(rng.integers(200, 1201))
        got.append((l, d, n, m, n))
    return got


def _instances(case, seed):
    rng = np.random.default_rng(seed)
    letters = _AMINO if case["call"] == "protein" else _DNA
    return [(_planted(rng, letters, n, m, l, d), l, d) for l, d, n, m, _ in _shapes(case)]


# ------------------------------------------------------------------ a program's contexts and calls

_contexts = {}


def _context(kind, **options):
    key = (kind,) + tuple(sorted(options.items()))
    if key not in _contexts:
        stream = torch.cuda.Stream() if kind == "device" else None
        ctx = pms.Context(torch.cuda.current_device(), stream=stream)
        if options:
            ctx.set_options(**options)
        _contexts[key] = (ctx, stream)
    return _contexts[key]


def prepare(case, seed):
    call = case["call"]
    insts = _instances(case, seed)
    state = {"call": call, "insts": insts}
    if call in ("device", "quorum"):
        state["ctx"], stream = _context("device", **({"quorum": case["q"]} if call == "quorum" else {}))
        seqs, state["l"], state["d"] = insts[0]
        state["n"], state["m"] = seqs.shape
        state["seqs"] = torch.from_numpy(seqs).cuda()
        state["motifs"] = torch.zeros(CAPACITY, dtype=torch.int64, device="cuda")
        state["status"] = torch.zeros(4, dtype=torch.int32, device="cuda")
        stream.wait_stream(torch.cuda.current_stream())   # the solves run on the context's stream
    else:
        state["ctx"], _ = _context(call)
        # the program's own array for the answers, with room to spare
        if call == "protein":
            state["letters"] = np.zeros((CAPACITY, case["l"]), dtype=np.uint8)
        else:
            room = sum(1024 + int(2 * _chance_motifs(*shape[:4])) for shape in _shapes(case))
            state["codes"] = np.zeros(room, dtype=np.uint64)
    return state


def _gather(codes, sets):
    at = 0
    for s in sets:
        codes[at:at + len(s)] = s
        at += len(s)
    return codes, np.array([len(s) for s in sets])


def run(state):
    ctx, call = state["ctx"], state["call"]
    if call in ("device", "quorum"):
        ctx.solve_device(state["seqs"], state["n"], state["m"], state["l"], state["d"], state["motifs"], CAPACITY,
                         state["status"])
        return state["motifs"], state["status"]
    if call == "host":
        return _gather(state["codes"], [ctx.solve(*state["insts"][0])])
    if call == "protein":
        found = ctx.solve_sigma(*state["insts"][0], alphabet=pms.PROTEIN)
        state["letters"][:len(found)] = found
        return state["letters"], len(found)
    if call == "batch":
        sets = ctx.solve_batch(state["insts"])
    else:
        tickets = [ctx.submit(*inst) for inst in state["insts"]]
        sets = []
        for t in tickets:
            sets.append(ctx.wait(t))
            ctx.release(t)
    return _gather(state["codes"], sets)


def work(case):
    """Bytes: every sequence read once, a status and a motif written. Operations: what the method cannot
    do without, the distance of every seed l-mer to every window of the other sequences, and one
    distance for each set of changed positions of every seed (four integer operations each)."""
    moved = ops = 0
    for l, d, n, m, q in _shapes(case):
        W = m - l + 1
        seeds = W * (n - q + 1)
        moved += n * m + 24
        ops += 4 * seeds * ((n - 1) * W + sum(math.comb(l, k) for k in range(d + 1)))
    return {"bytes": moved, "flops": ops}


# ------------------------------------------------------------------ the answer without the library

def exact(case, seed):
    """Short DNA motifs: the strings of every window's ball marked per sequence, the marks of all sequences combined."""
    if case["call"] not in ("device", "host") or case["l"] > 11 or case["m"] > 800:
        return None
    seqs, l, d = _instances(case, seed)[0]
    code = np.searchsorted(_DNA, seqs).astype(np.int64)
    place = 4 ** np.arange(l - 1, -1, -1, dtype=np.int64)
    changes = [np.zeros(1, dtype=np.int64)]
    for k in range(1, d + 1):
        for where in itertools.combinations(range(l), k):
            digits = np.array(list(itertools.product((1, 2, 3), repeat=k)), dtype=np.int64)
            changes.append(digits @ place[list(where)])
    changes = np.concatenate(changes)   # exclusive-or changes of the two-bit letters: every string within d
    alive, first = np.ones(4 ** l, dtype=bool), None
    for row in code:
        windows = np.lib.stride_tricks.sliding_window_view(row, l) @ place
        marks = np.zeros(4 ** l, dtype=np.int64)
        for w in windows:
            marks[w ^ changes] += 1
        first = marks if first is None else first
        alive &= marks > 0
    motifs = np.flatnonzero(alive)
    if case["call"] == "host":
        return _gather(np.zeros(1024 + int(2 * _chance_motifs(l, d, *seqs.shape)), dtype=np.uint64), [motifs])
    out = np.zeros(CAPACITY, dtype=np.int64)
    out[:len(motifs)] = motifs
    return out, np.array([first[motifs].sum(), len(motifs), 0, 0], dtype=np.int32)
