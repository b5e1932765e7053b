"""The work whose speed is measured: whole calls of the public entry points on
synthetic CDR3 repertoires, over the range of sizes, radii and options they
take in use.

``listed()`` names the cases; ``draw(rng)`` gives another one of the same
ranges.  A case is a dict of plain values:

  kind     which entry points run (see ``run``)
  n        sequences (receptors for "paired", reference entries for "query"
           and "build")
  d        radius
  metric   "levenshtein" or "hamming"
  reps     repertoires the sequences are split into (0: one, unsplit)
  q        query sequences ("query", "build")
  passes   passes a search in passes is asked for ("stream")

Sequences are drawn on the GPU from the laws of ``cdr3_synth`` (length, end
residues and residue frequencies, 15% derived from an earlier sequence by one
or two edits, 1% exact copies): those are the only properties the search's cost
depends on, and drawing there keeps preparation short.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import cdr3_synth as gen
import paper_2403_09010_gb300 as xtn

WIDTH = gen.WIDTH
DERIVED, COPIES = 0.15, 0.01
MAX_SCORE = 24  # the TCRdist radius of the repository's benchmark


def listed():
    def case(name, kind, n, d, metric="levenshtein", reps=0, q=0, passes=0):
        return dict(name=name, kind=kind, n=n, d=d, metric=metric, reps=reps, q=q, passes=passes)

    return [
        # a small repertoire, exact radius one: launches and waits count
        case("self_10k_d1", "self", 10_000, 1),
        # one donor's repertoire at the widest radius, then the TCRdist filter on
        # its neighbours (the similarity-metric experiment of the paper)
        case("tcrdist_40k_d3", "tcrdist", 40_000, 3),
        # a host program's arrays, copied in and out by the call
        case("host_200k_d2", "host", 200_003, 2),
        # the headline search
        case("self_1m_d2", "self", 1_000_000, 2),
        # a pooled cohort at radius one
        case("self_10m_d1", "self", 10_000_019, 1),
        # overlap between repertoires with the metric of the overlap tools
        case("overlap_500k_d2_hamming", "between", 500_009, 2, "hamming", reps=8),
        # a cohort of repertoires of uneven size in one planned launch
        case("plan_64reps_d2", "plan", 2_300_017, 2, reps=64),
        # receptors with both chains known
        case("paired_300k_d2", "paired", 300_001, 2),
        # a search that has to stay inside a memory budget
        case("stream_1m_d2", "stream", 1_000_003, 2, passes=4),
        # interactive lookups in a resident reference: few queries, and a batch
        case("query_40_of_1m_d2", "query", 1_000_000, 2, q=40),
        case("query_10k_of_10m_d2", "query", 10_000_000, 2, q=10_007),
        # a reference used once: built, then looked up
        case("build_300k_query_30k_d2", "build", 300_007, 2, q=30_011),
    ]


# Deletion variants of a 14.5-residue sequence by radius (what bounds a drawn case).
VARIANTS = {1: 15.7, 2: 105.0, 3: 450.0}
MOST_RECORDS = 230e6


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1

    kind = rng.choice(["self", "self", "host", "tcrdist", "between", "plan", "paired", "stream",
                       "query", "query", "build"])
    d = {"tcrdist": rng.choice([2, 3]), "plan": rng.choice([1, 2]), "stream": 2,
         "paired": rng.choice([1, 2])}.get(kind, rng.choice([1, 2, 2, 3] if kind == "self" else [1, 2]))
    variants = VARIANTS[d] * (3.5 if kind == "paired" else 1.0)
    lo, hi = {"self": (5_000, 10_000_000), "host": (2_000, 500_000), "tcrdist": (5_000, 400_000),
              "between": (20_000, 2_000_000), "plan": (50_000, 2_300_000),
              "paired": (5_000, 400_000), "stream": (200_000, 1_500_000),
              "query": (100_000, 10_000_000), "build": (20_000, 500_000)}[kind]
    n = log(lo, min(hi, MOST_RECORDS / variants if kind != "query" else hi))
    return dict(kind=kind, n=n, d=d,
                metric=rng.choice(["levenshtein", "hamming"])
                if kind in ("self", "between", "query", "stream") else "levenshtein",
                reps=rng.randint(2, 100) if kind in ("between", "plan") else 0,
                q={"query": log(1, 20_000), "build": log(1_000, 50_000)}.get(kind, 0),
                passes=rng.randint(2, 9) if kind == "stream" else 0)


# ----------------------------------------------------------------- inputs
def _length_law(mean, sd, lo, hi):
    """P(length) of a normal rounded to integers and redrawn until in [lo, hi]."""
    def cdf(x):
        return 0.5 * (1.0 + math.erf((x - mean) / (sd * math.sqrt(2.0))))
    return lo, [cdf(k + 0.5) - cdf(k - 0.5) for k in range(lo, hi + 1)]


BETA = (b"CAS", _length_law(gen.LEN_MEAN, gen.LEN_SD, gen.LEN_MIN, gen.LEN_MAX))
ALPHA = (gen.ALPHA_PREFIX, _length_law(*gen.ALPHA_LENGTHS))


class _Draw:
    """Letter matrices (rows 0-padded to WIDTH) and lengths, drawn on `device`."""

    def __init__(self, seed, device):
        self.device = device
        self.g = torch.Generator(device=device).manual_seed(int(seed))
        counts = np.rint(gen.FREQ * 100).astype(np.int64)  # the frequencies are whole per cents
        self.letters = torch.from_numpy(np.repeat(gen.AA_BYTES, counts)).to(device)
        self.alphabet = torch.from_numpy(gen.AA_BYTES.copy()).to(device)
        self.columns = torch.arange(WIDTH, device=device)

    def below(self, hi, n):
        """Whole numbers, uniform below `hi` (a number or one per draw)."""
        u = torch.rand(n, generator=self.g, device=self.device, dtype=torch.float64)
        top = hi - 1
        return torch.minimum((u * hi).long(), top) if torch.is_tensor(top) else (u * hi).long().clamp_(max=top)

    def residues(self, shape):
        at = torch.randint(0, 100, shape, generator=self.g, device=self.device, dtype=torch.int32)
        return torch.index_select(self.letters, 0, at.reshape(-1)).reshape(shape)

    def fresh(self, n, law):
        prefix, (lo, p) = law
        p = torch.tensor(p, device=self.device)
        L = torch.multinomial(p, n, replacement=True, generator=self.g) + lo
        M = self.residues((n, WIDTH))
        for at, letter in enumerate(prefix):
            keep = torch.rand(n, generator=self.g, device=self.device) < gen.FLANK_P
            M[:, at] = torch.where(keep, torch.full_like(M[:, at], letter), M[:, at])
        last = (torch.rand(n, generator=self.g, device=self.device) < gen.FLANK_P).nonzero()[:, 0]
        M[last, L[last] - 1] = ord("F")
        M[self.columns[None, :] >= L[:, None]] = 0
        return M, L

    def edit(self, M, L, rows):
        """One edit (substitution, insertion or deletion) of each row listed."""
        if not rows.numel():
            return
        m, l = M[rows], L[rows]
        k = rows.numel()
        kind = self.below(3, k)
        kind = torch.where((kind == 1) & (l >= WIDTH), 0, kind)
        kind = torch.where((kind == 2) & (l <= gen.MIN_AFTER_DELETE), 0, kind)
        at = self.below(l + (kind == 1), k)[:, None]
        col = self.columns[None, :]
        # insertion reads one column to the left past the position, deletion one to the right
        src = torch.where((kind[:, None] == 1) & (col > at), col - 1, col)
        src = torch.where((kind[:, None] == 2) & (col >= at), col + 1, src)
        padded = torch.cat([m, torch.zeros_like(m[:, :1])], 1)
        old = torch.gather(m, 1, at.clamp(max=WIDTH - 1))[:, 0]
        place = torch.searchsorted(self.alphabet.int(), old.int())
        other = self.alphabet[(place + 1 + self.below(19, k)) % 20]  # never the old residue
        new = torch.where(kind == 0, other, self.residues((k,)))
        m = torch.gather(padded, 1, src)
        m = torch.where((kind[:, None] != 2) & (col == at), new[:, None], m)
        M[rows] = m
        L[rows] = l + (kind == 1).long() - (kind == 2).long()

    def related(self, n, laws=(BETA,)):
        """n entries of one chain per law: fresh ones, edited copies and exact
        copies; an edited entry has one or two edits over its chains."""
        chains = [self.fresh(n, law) for law in laws]
        u = torch.rand(n, generator=self.g, device=self.device)
        u[0] = 1.0
        other = (u < DERIVED + COPIES).nonzero()[:, 0]
        if other.numel():
            fresh = (u >= DERIVED + COPIES).nonzero()[:, 0]
            before = torch.searchsorted(fresh, other)
            src = fresh[self.below(before, other.numel())]
            for M, L in chains:
                M[other], L[other] = M[src], L[src]
            derived = other[u[other] < DERIVED]
            twice = derived[torch.rand(derived.numel(), generator=self.g, device=self.device) < 0.5]
            for rows in (derived, twice):
                chain = self.below(len(chains), rows.numel())
                for c, (M, L) in enumerate(chains):
                    self.edit(M, L, rows[chain == c])
        return chains

    def queries(self, M, L, n):
        """Half edited copies of entries of (M, L), half fresh, mixed."""
        src = self.below(L.numel(), n // 2)
        A, a = M[src].clone(), L[src].clone()
        rows = torch.arange(n // 2, device=self.device)
        self.edit(A, a, rows)
        self.edit(A, a, rows[torch.rand(n // 2, generator=self.g, device=self.device) < 0.5])
        B, b = self.fresh(n - n // 2, BETA)
        order = torch.randperm(n, generator=self.g, device=self.device)
        return torch.cat([A, B])[order], torch.cat([a, b])[order]


def _pack(M, L):
    off = torch.zeros(L.numel() + 1, dtype=torch.int64, device=L.device)
    torch.cumsum(L, 0, out=off[1:])
    return M[M != 0], off


def _split(n, reps, seed):
    """Offsets of `reps` repertoires of uneven (log-uniform) sizes."""
    rng = np.random.default_rng(seed)
    share = np.exp(rng.uniform(0.0, math.log(200.0), reps))
    off = np.rint(np.concatenate([[0.0], np.cumsum(share) / share.sum()]) * n).astype(np.int64)
    off[-1] = n
    return off


def _inputs(case, seed, device):
    draw_ = _Draw(seed, device)
    chains = draw_.related(case["n"], (ALPHA, BETA) if case["kind"] == "paired" else (BETA,))
    s = {"chains": [_pack(*c) for c in chains]}
    if case["q"]:
        s["queries"] = _pack(*draw_.queries(*chains[0], case["q"]))
    if case["reps"]:
        s["reps"] = _split(case["n"], case["reps"], seed)
    return s


def prepare(case, seed):
    s = dict(_inputs(case, seed, "cuda"), case=case)
    kind, n, d = case["kind"], case["n"], case["d"]
    if kind == "host":
        s["chains"] = [(a.cpu().numpy(), b.cpu().numpy()) for a, b in s["chains"]]
    elif kind == "plan":
        s["plan"] = xtn.Plan(s["chains"][0][1], d, s["reps"])
    elif kind == "query":
        s["index"] = xtn.index_build(*s["chains"][0], d)
    elif kind == "stream":
        s["budget"] = int(1.05 * n * VARIANTS[d] / case["passes"])
    # the program's own row buffers (a result's length depends on the sequences)
    most = 8 * case["q"] + 1024 if case["q"] else (8 if d == 3 else 1) * n + 1024
    s["out"] = [np.zeros((most, 3), np.uint32) if kind == "host" else
                torch.zeros((most, 3), dtype=torch.int32, device="cuda")
                for _ in range(2 if kind == "tcrdist" else 1)]
    return s


def _rows(state):
    case = state["case"]
    kind, n, d, metric = case["kind"], case["n"], case["d"], case["metric"]
    seqs, off = state["chains"][0]
    if kind in ("self", "host"):
        return [xtn.search_self(seqs, off, d, metric=metric)]
    if kind == "tcrdist":
        rows = xtn.search_self(seqs, off, d, cap=8 * n + 1024)
        return [rows, xtn.tcrdist_filter(seqs, off, rows, MAX_SCORE)]
    if kind == "between":
        return [xtn.search_between(seqs, off, d, state["reps"], metric=metric)]
    if kind == "plan":
        state["plan"].run(seqs)
        return [state["plan"].result(cap=n + 1024, like=seqs)]
    if kind == "paired":
        return [xtn.search_paired(seqs, off, *state["chains"][1], d)]
    if kind == "stream":
        return [xtn.search_self_streaming(seqs, off, d, metric=metric,
                                          max_pass_records=state["budget"])[0]]
    index = state["index"] if kind == "query" else xtn.index_build(seqs, off, d)
    return [xtn.search_query(index, *state["queries"], metric=metric)]


def run(state):
    """The rows, collected in the program's own buffers, and how many they are."""
    got = _rows(state)
    for out, rows in zip(state["out"], got):
        out[:rows.shape[0]] = rows
    return {"rows": state["out"], "count": [rows.shape[0] for rows in got]}


def work(case):
    """Letters and offsets read once, rows written once; a lookup reads one
    directory entry and one record per query variant instead of the index."""
    rows = {1: 0.15, 2: 0.3, 3: 3.0}[case["d"]]
    per_seq = 14.5 + 8.0
    n, q = case["n"], case["q"]
    read = n * per_seq * (2 if case["kind"] == "paired" else 1)
    if case["kind"] == "query":
        read = 0.0
    read += q * (per_seq + VARIANTS[case["d"]] * 12.0)
    return {"bytes": read + 12.0 * rows * (q or n), "flops": 0.0}


# ------------------------------------------------------- the plain definition
def _lev(a, b):
    row = list(range(len(b) + 1))
    for i, x in enumerate(a, 1):
        prev, row[0] = row[0], i
        for j, y in enumerate(b, 1):
            prev, row[j] = row[j], min(row[j] + 1, row[j - 1] + 1, prev + (x != y))
    return row[-1]


def exact(case, seed):
    """The rows of a small search by dictionaries of deletion variants and the
    dynamic programme; None for the larger cases and the other kinds."""
    n, d = case["n"], case["d"]
    if case["kind"] not in ("self", "host") or case["metric"] != "levenshtein" \
            or n * VARIANTS[d] > 1.5e6:
        return None
    s = _inputs(case, seed, "cuda")
    seqs, off = (x.cpu().numpy() for x in s["chains"][0])
    strs = gen.to_strings(seqs, off)
    groups = {}
    for i, t in enumerate(strs):
        variants = {t}
        for k in range(1, d + 1):
            for cut in itertools.combinations(range(len(t)), k):
                variants.add("".join(ch for p, ch in enumerate(t) if p not in cut))
        for v in variants:
            groups.setdefault(v, []).append(i)
    pairs = {p for g in groups.values() if len(g) > 1 for p in itertools.combinations(g, 2)}
    rows = sorted((i, j, x) for i, j in pairs if (x := _lev(strs[i], strs[j])) <= d)
    out = np.zeros((n + 1024, 3), np.int64)
    out[:len(rows)] = np.array(rows, dtype=np.int64).reshape(-1, 3)
    return {"rows": [out if case["kind"] == "host" else torch.from_numpy(out)],
            "count": [len(rows)]}
