"""The work that users of libmsadp have it do, as measurable cases.

Every case goes through a public entry point of ``paper_2311_17530_gb300.msadp``
on seeded synthetic sequences (an ancestor mutated by substitutions and indels,
or independent uniform residues), with the alphabets, scores, rates and sizes of
the repository's workloads, serving stream and tests:

* ``plan``     one problem on device buffers (``Plan.execute``): a program that
               aligns many problems of one shape and keeps its plan;
* ``align``    one problem on host buffers (``msa_align``), copies included;
* ``noalloc``  one problem on the library's fixed scratch (``msa_align_noalloc``);
* ``pruned``   the exact search-space pruning (``msa_align_pruned``);
* ``near``     optimal and near-optimal enumeration (``msa_near_optimal``);
* ``serve``    a burst of mixed requests (``msa_submit`` .. ``msa_poll``).

Every result is whole numbers: scores, move masks (the lowest mask wins a tie)
and the gapped rows they spell.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2311_17530_gb300 import msadp

ALPHABETS = {"dna": "ACGT", "protein": "ARNDCQEGHILKMFPSTWYV"}
GAPS = {"dna": -8, "protein": -6}
SUB_RATE = {2: 0.2, 3: 0.2, 4: 0.15, 5: 0.25, 6: 0.25, 7: 0.25, 8: 0.25}
INDEL_RATE = 0.05
SERVE_LENS = {2: (200, 2000), 3: (40, 300), 4: (20, 80)}  # the serving stream's ranges per k


def listed():
    return [
        # the smallest call: a pair of short reads from host buffers, where launches and copies count
        {"name": "align_k2_dna_reads", "kind": "align", "lens": "150,170", "scoring": "dna", "related": True},
        # one long protein pair on a kept plan: a single wavefront
        {"name": "plan_k2_protein_long", "kind": "plan", "lens": "5000,4800", "scoring": "protein", "related": True},
        # three short unrelated DNA sequences on a kept plan: the latency-bound end of k = 3
        {"name": "plan_k3_dna_128", "kind": "plan", "lens": "128,128,128", "scoring": "dna", "related": False},
        # three whole protein chains: the headline workload
        {"name": "plan_k3_protein", "kind": "plan", "lens": "700,760,800", "scoring": "protein", "related": True},
        # four DNA sequences of unequal length
        {"name": "plan_k4_dna", "kind": "plan", "lens": "110,118,124,130", "scoring": "dna", "related": True},
        # five protein fragments, odd and ragged lengths
        {"name": "plan_k5_protein", "kind": "plan", "lens": "37,41,33,45,39", "scoring": "protein", "related": True},
        # six short protein fragments: the widest recurrence of the line kernels
        {"name": "plan_k6_protein", "kind": "plan", "lens": "23,24,24,21,24,24", "scoring": "protein",
         "related": True},
        # seven peptides: the generic tile kernel at k = 7
        {"name": "plan_k7_protein", "kind": "plan", "lens": "11,9,12,10,9,11,10", "scoring": "protein",
         "related": True},
        # a caller that must not allocate: one mid-size triple on the fixed scratch
        {"name": "noalloc_k3_protein", "kind": "noalloc", "lens": "120,110,130", "scoring": "protein",
         "related": True},
        # exact pruning of the headline workload with the bound the device builds
        {"name": "pruned_k3_protein", "kind": "pruned", "lens": "700,760,800", "scoring": "protein", "related": True},
        # all alignments within 3 of the optimum, up to 256 of them
        {"name": "near_k3_protein", "kind": "near", "lens": "120,110,130", "scoring": "protein", "related": True,
         "delta": 3, "max_count": 256},
        # a burst of the serving stream's mix (half pairs, a third triples, the rest quadruples)
        {"name": "serve_mixed_256", "kind": "serve", "requests": 256, "mix": 5},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# lengths a drawn problem takes per kind and k, and the most cells it may have
_RANGES = {
    "align": ({2: (50, 2000), 3: (30, 300), 4: (16, 80)}, 3e7),
    "plan": ({2: (200, 5000), 3: (40, 800), 4: (20, 130), 5: (12, 45), 6: (8, 32), 7: (5, 12), 8: (4, 8)}, 2.0e8),
    "noalloc": ({2: (100, 1500), 3: (30, 130), 4: (12, 45), 5: (8, 18)}, 2.5e6),
    "pruned": ({2: (200, 2000), 3: (60, 700), 4: (20, 90)}, 1.5e8),
    "near": ({2: (60, 800), 3: (30, 120), 4: (12, 36)}, 1.7e6),
}


def draw(rng: random.Random):
    kind = rng.choice(["plan", "plan", "plan", "align", "noalloc", "pruned", "near", "serve"])
    if kind == "serve":
        return {"kind": kind, "requests": _log_int(rng, 8, 256), "mix": rng.randrange(1, 10**6)}
    ranges, most = _RANGES[kind]
    k = rng.choice(sorted(ranges))
    if kind == "plan" and k >= 7:
        most = 2.5e7
    lo, hi = ranges[k]
    while True:
        base = _log_int(rng, lo, hi)
        lens = [min(hi, max(lo, int(round(base * rng.uniform(0.8, 1.25))))) for _ in range(k)]
        if math.prod(n + 1 for n in lens) <= most:
            break
    case = {"kind": kind, "lens": ",".join(map(str, lens)), "scoring": rng.choice(["dna", "protein"]),
            "related": rng.random() < 0.8}
    if kind == "near":
        case["delta"] = rng.randrange(0, 4)
        case["max_count"] = _log_int(rng, 8, 96)
    return case


def _lens(case):
    return [int(v) for v in case["lens"].split(",")]


# --------------------------------------------------------------------------
# Inputs

def _table(rng, scoring):
    """DNA: match 5, mismatch -4. Protein: a symmetric table, diagonal 4..11, the rest -4..3."""
    if scoring == "dna":
        return np.where(np.eye(4, dtype=bool), 5, -4).astype(np.int32)
    upper = np.triu(rng.integers(-4, 4, size=(20, 20)), 1)
    return (upper + upper.T + np.diag(rng.integers(4, 12, size=20))).astype(np.int32)


def _descendant(rng, ancestor, letters, sub, n):
    """One mutated copy of ``ancestor``, cut or padded to ``n`` residues: at a
    position an indel starts with INDEL_RATE (half deletions, half insertions,
    geometric lengths), otherwise the residue changes with rate ``sub``."""
    m = len(ancestor)
    out = ancestor.copy()
    changed = rng.random(m) < sub
    out[changed] = (out[changed] + rng.integers(1, letters, size=int(changed.sum()))) % letters
    indel = rng.random(m) < INDEL_RATE
    deletion = indel & (rng.random(m) < 0.5)
    size = rng.geometric(0.5, size=m)
    keep = np.ones(m, dtype=bool)
    for at in np.flatnonzero(deletion):
        keep[at:at + size[at]] = False
    extra = np.where(indel & ~deletion, size, 0)
    grown = np.repeat(out, np.where(keep, 1 + extra, 0))
    # the residues a position gained are uniform, the last of its run its own
    last = np.cumsum(np.where(keep, 1 + extra, 0))[keep] - 1
    own = np.zeros(len(grown), dtype=bool)
    own[last] = True
    grown[~own] = rng.integers(0, letters, size=int((~own).sum()))
    if len(grown) >= n:
        return grown[:n]
    return np.concatenate([grown, rng.integers(0, letters, size=n - len(grown))])


def _codes(rng, lens, scoring, related):
    letters = len(ALPHABETS[scoring])
    if not related:
        return [rng.integers(0, letters, size=n) for n in lens]
    ancestor = rng.integers(0, letters, size=int(round(sum(lens) / len(lens))))
    return [_descendant(rng, ancestor, letters, SUB_RATE[len(lens)], n) for n in lens]


def _problem(case, seed):
    """(codes of every sequence, the sequences, alphabet, table, gap)"""
    rng = np.random.default_rng(seed)
    scoring = case["scoring"]
    table = _table(rng, scoring)
    codes = _codes(rng, _lens(case), scoring, case["related"])
    alphabet = ALPHABETS[scoring]
    return codes, ["".join(alphabet[c] for c in s) for s in codes], alphabet, table, GAPS[scoring]


def _serve_mix(case):
    """(lens, scoring) of every request of a burst: a property of the case, not of the inputs' seed."""
    rng = random.Random(case["mix"])
    mix = []
    for _ in range(case["requests"]):
        k = rng.choices([2, 3, 4], weights=[50, 35, 15])[0]
        mix.append(([rng.randint(*SERVE_LENS[k]) for _ in range(k)], rng.choice(["dna", "protein"])))
    return mix


def _serve_problems(case, seed):
    return [_problem({"lens": ",".join(map(str, lens)), "scoring": scoring, "related": True}, [seed, i])
            for i, (lens, scoring) in enumerate(_serve_mix(case))]


def prepare(case, seed):
    if case["kind"] == "serve":
        return {"kind": "serve", "requests": [p[1:] for p in _serve_problems(case, seed)]}
    codes, seqs, alphabet, table, gap = _problem(case, seed)
    state = {"kind": case["kind"], "seqs": seqs, "alphabet": alphabet, "table": table, "gap": gap}
    if case["kind"] in ("plan", "noalloc"):
        residues = np.frombuffer("".join(seqs).encode(), dtype=np.uint8).copy()
        state["lens"] = _lens(case)
        state["residues"] = torch.from_numpy(residues).cuda()
        state["subst"] = torch.from_numpy(table.reshape(-1).copy()).cuda()
        state["result"], state["masks"] = msadp.device_outputs(len(residues), "cuda")
        if case["kind"] == "plan":
            state["plan"] = msadp.Plan(len(seqs), state["lens"], alphabet)
    if case["kind"] == "near":
        state["delta"], state["max_count"] = case["delta"], case["max_count"]
    return state


def _text(alignments, shapes):
    """The gapped rows of one alignment after another as bytes, a row of (k, total residues) taking
    ``total`` of them, zeros after its end (the layout of the C interface's buffers)."""
    out = np.zeros(sum(k * total for k, total in shapes), dtype=np.uint8)
    at = 0
    for rows, (k, total) in zip(alignments, shapes):
        for i, row in enumerate(rows):
            out[at + i * total:at + i * total + len(row)] = np.frombuffer(row.encode(), dtype=np.uint8)
        at += k * total
    return out


def _shape(seqs):
    return len(seqs), sum(map(len, seqs))


def _enumeration(found, more, seqs, most):
    """Outputs of an enumeration of up to ``most`` alignments (score, masks first column first, rows)."""
    masks = np.zeros((most, _shape(seqs)[1]), dtype=np.uint8)
    scores = np.zeros(most, dtype=np.int64)
    for a, (score, moves, _) in enumerate(found):
        scores[a] = score
        masks[a, :len(moves)] = moves
    return {"count": len(found), "more": int(more), "scores": scores, "masks": masks,
            "rows": _text([f[2] for f in found], [_shape(seqs)] * most)}


def run(state):
    kind = state["kind"]
    if kind == "serve":
        return _run_serve(state["requests"])
    seqs, alphabet, table, gap = state["seqs"], state["alphabet"], state["table"], state["gap"]
    if kind in ("plan", "noalloc"):
        args = (state["residues"].data_ptr(), state["subst"].data_ptr(), gap, state["result"].data_ptr(),
                state["masks"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if kind == "plan":
            state["plan"].execute(*args)
        else:
            msadp.msa_align_noalloc(state["lens"], alphabet, *args)
        return {"result": state["result"], "masks": state["masks"]}
    if kind == "align":
        score, rows = msadp.msa_align(seqs, alphabet, table, gap)
        return {"score": score, "rows": _text([rows], [_shape(seqs)])}
    if kind == "pruned":
        score, rows, stats = msadp.msa_align_pruned(seqs, alphabet, table, gap)
        return {"score": score, "rows": _text([rows], [_shape(seqs)]), "stats": stats}
    found, more = msadp.msa_near_optimal(seqs, alphabet, table, gap, state["delta"], state["max_count"])
    return _enumeration(found, more, seqs, state["max_count"])


def _run_serve(requests):
    shapes = {}
    for seqs, alphabet, table, gap in requests:
        handle = msadp.msa_submit(seqs, alphabet, table, gap)
        shapes[handle] = _shape(seqs)
    done = {}
    while len(done) < len(shapes):
        handle = msadp.msa_wait_any(1_000_000)
        if handle is not None and handle in shapes:
            done[handle] = msadp.msa_poll(handle, *shapes[handle])
    return {"scores": np.array([done[h][0] for h in shapes], dtype=np.int64),
            "rows": _text([done[h][1] for h in shapes], list(shapes.values()))}


def work(case):
    """Bytes: the residues and the table read, the result and the alignment written. Operations: an
    addition and a maximum for every cell and move (the serving burst: over all its requests)."""
    if case["kind"] == "serve":
        parts = [work({"kind": "align", "lens": ",".join(map(str, lens)), "scoring": scoring})
                 for lens, scoring in _serve_mix(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    lens = _lens(case)
    k, total, letters = len(lens), sum(lens), len(ALPHABETS[case["scoring"]])
    out = total if case["kind"] in ("plan", "noalloc") else k * max(lens)
    count = case.get("max_count", 1)
    return {"bytes": total + 4 * letters * letters + 16 + out * count,
            "flops": 2 * (2**k - 1) * math.prod(n + 1 for n in lens)}


# --------------------------------------------------------------------------
# The same results from plain torch in 64 bits

def _moves(codes, table, gap):
    """(H, move) of every cell, flat row-major: cells of one index sum at a time, each taking the
    best of its 2^k - 1 lower neighbours, the lowest mask among equals."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    k = len(codes)
    rho = [len(c) + 1 for c in codes]
    n = math.prod(rho)
    stride = [math.prod(rho[i + 1:]) for i in range(k)]
    letters = len(table)
    sub = torch.from_numpy(table.astype(np.int64).reshape(-1)).to(dev)
    code = [torch.from_numpy(np.concatenate([[0], c]).astype(np.int64)).to(dev) for c in codes]
    level = torch.zeros(1, dtype=torch.int16, device=dev)
    for r in rho:
        level = (level[:, None] + torch.arange(r, dtype=torch.int16, device=dev)).reshape(-1)
    order = torch.sort(level, stable=True)[1]
    ends = torch.cumsum(torch.bincount(level.to(torch.int32)), 0).tolist()
    del level
    h = torch.zeros(n, dtype=torch.int64, device=dev)
    move = torch.zeros(n, dtype=torch.uint8, device=dev)
    low = torch.tensor(-2**60, dtype=torch.int64, device=dev)
    for begin, end in zip(ends[:-1], ends[1:]):
        cells = order[begin:end]
        x = [(cells // stride[i]) % rho[i] for i in range(k)]
        inside = [v > 0 for v in x]
        pair = {(i, j): sub[code[i][x[i]] * letters + code[j][x[j]]] for i in range(k) for j in range(i + 1, k)}
        best = low.expand(len(cells))
        pick = torch.zeros(len(cells), dtype=torch.uint8, device=dev)
        for m in range(1, 2**k):
            members = [i for i in range(k) if m >> i & 1]
            ok = inside[members[0]]
            for i in members[1:]:
                ok = ok & inside[i]
            cost = h[(cells - sum(stride[i] for i in members)).clamp_(min=0)] + gap * len(members) * (k - len(members))
            for a, i in enumerate(members):
                for j in members[a + 1:]:
                    cost += pair[i, j]
            better = ok & (cost > best)
            best = torch.where(better, cost, best)
            pick = torch.where(better, torch.tensor(m, dtype=torch.uint8, device=dev), pick)
        h[cells] = best
        move[cells] = pick
    return h, move, stride


def _walk(move, stride, lens):
    """Move masks from the far corner back, last column first."""
    move = move.cpu().numpy()
    at = sum(n * s for n, s in zip(lens, stride))
    masks = []
    while at:
        m = int(move[at])
        masks.append(m)
        at -= sum(s for i, s in enumerate(stride) if m >> i & 1)
    return masks


def _spell(seqs, masks):
    rows = []
    for i, s in enumerate(seqs):
        residues = iter(s)
        rows.append("".join(next(residues) if m >> i & 1 else "-" for m in masks))
    return rows


def _within(h, stride, codes, table, gap, delta, most):
    """Every alignment within ``delta`` of the optimum, in increasing order of its columns read from
    the last one back: (score, masks last column first), up to ``most`` of them, and whether more remain."""
    k = len(codes)
    h = h.cpu().numpy()
    table = table.tolist()
    least = int(h[-1]) - delta
    pairs = [(i, j) for i in range(k) for j in range(i + 1, k)]
    masks_of = [[i for i in range(k) if m >> i & 1] for m in range(2**k)]

    def successors(x, at, fixed):
        for m in range(1, 2**k):
            if any(x[i] == 0 for i in masks_of[m]):
                continue
            gain = 0
            for i, j in pairs:
                a, b = m >> i & 1, m >> j & 1
                gain += table[codes[i][x[i] - 1]][codes[j][x[j] - 1]] if a and b else gap if a or b else 0
            back = at - sum(stride[i] for i in masks_of[m])
            if int(h[back]) + gain + fixed >= least:
                yield m, tuple(v - (m >> i & 1) for i, v in enumerate(x)), back, fixed + gain

    found, path = [], []
    corner = tuple(len(c) for c in codes)
    stack = [successors(corner, len(h) - 1, 0)]
    while stack:
        step = next(stack[-1], None)
        if step is None:
            stack.pop()
            if path:
                path.pop()
            continue
        m, x, at, fixed = step
        path.append(m)
        if at == 0:
            if len(found) == most:
                return found, True
            found.append((fixed, list(path)))
            path.pop()
        else:
            stack.append(successors(x, at, fixed))
    return found, False


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None  # hundreds of problems: more than 20 seconds
    codes, seqs, _, table, gap = _problem(case, seed)
    h, move, stride = _moves(codes, table, gap)
    score = int(h[-1])
    if kind == "near":
        found, more = _within(h, stride, codes, table, gap, case["delta"], case["max_count"])
        found = [(fixed, path[::-1], _spell(seqs, path[::-1])) for fixed, path in found]
        return _enumeration(found, more, seqs, case["max_count"])
    masks = _walk(move, stride, _lens(case))
    if kind in ("plan", "noalloc"):
        padded = torch.zeros(sum(_lens(case)), dtype=torch.uint8)
        padded[:len(masks)] = torch.tensor(masks, dtype=torch.uint8)
        return {"result": torch.tensor([score, len(masks), 0, 0], dtype=torch.int32), "masks": padded}
    out = {"score": score, "rows": _text([_spell(seqs, masks[::-1])], [_shape(seqs)])}
    if kind == "pruned":
        out["stats"] = dict.fromkeys(["lower_bound", "tiles", "tiles_skipped", "cells_skipped", "cells"])
    return out
