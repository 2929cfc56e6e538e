"""The work this library is measured on: whole alignments, their parts and the
tree, through the public entry points of `paper_1704_00878_gb300.binding`.

Inputs are synthetic sequence sets with the distributions of the library's own
workloads (windows of random ancestors, substitutions drawn from the scoring
matrix's conditional probabilities, indels), made on the GPU from the seed.
Every case is one of six kinds:

  msa       one whole alignment: load the letters, choose the center, align
            every sequence to it, merge, rows and the sum-of-pairs cost
  center    the sampled exact center alone: load, choose, row sums
  anchored  similar nucleotides through center segments, then merge and cost
  pairs     Smith-Waterman scores of a list of pairs of a loaded set
  grad      loss and gradient of one training batch of the center selector
  tree      the neighbour-joining tree of a merged alignment
"""
import math

import numpy as np
import torch

from paper_1704_00878_gb300 import binding as B

# BLOSUM62 (Henikoff and Henikoff 1992) in the conventional 24-letter order,
# the scores of the protein cases (gap 11 / 1).
LETTERS = "ARNDCQEGHILKMFPSTWYVBZX*"
_BLOSUM62 = """
 4 -1 -2 -2  0 -1 -1  0 -2 -1 -1 -1 -1 -2 -1  1  0 -3 -2  0 -2 -1  0 -4
-1  5  0 -2 -3  1  0 -2  0 -3 -2  2 -1 -3 -2 -1 -1 -3 -2 -3 -1  0 -1 -4
-2  0  6  1 -3  0  0  0  1 -3 -3  0 -2 -3 -2  1  0 -4 -2 -3  3  0 -1 -4
-2 -2  1  6 -3  0  2 -1 -1 -3 -4 -1 -3 -3 -1  0 -1 -4 -3 -3  4  1 -1 -4
 0 -3 -3 -3  9 -3 -4 -3 -3 -1 -1 -3 -1 -2 -3 -1 -1 -2 -2 -1 -3 -3 -2 -4
-1  1  0  0 -3  5  2 -2  0 -3 -2  1  0 -3 -1  0 -1 -2 -1 -2  0  3 -1 -4
-1  0  0  2 -4  2  5 -2  0 -3 -3  1 -2 -3 -1  0 -1 -3 -2 -2  1  4 -1 -4
 0 -2  0 -1 -3 -2 -2  6 -2 -4 -4 -2 -3 -3 -2  0 -2 -2 -3 -3 -1 -2 -1 -4
-2  0  1 -1 -3  0  0 -2  8 -3 -3 -1 -2 -1 -2 -1 -2 -2  2 -3  0  0 -1 -4
-1 -3 -3 -3 -1 -3 -3 -4 -3  4  2 -3  1  0 -3 -2 -1 -3 -1  3 -3 -3 -1 -4
-1 -2 -3 -4 -1 -2 -3 -4 -3  2  4 -2  2  0 -3 -2 -1 -2 -1  1 -4 -3 -1 -4
-1  2  0 -1 -3  1  1 -2 -1 -3 -2  5 -1 -3 -1  0 -1 -3 -2 -2  0  1 -1 -4
-1 -1 -2 -3 -1  0 -2 -3 -2  1  2 -1  5  0 -2 -1 -1 -1 -1  1 -3 -1 -1 -4
-2 -3 -3 -3 -2 -3 -3 -3 -1  0  0 -3  0  6 -4 -2 -2  1  3 -1 -3 -3 -1 -4
-1 -2 -2 -1 -3 -1 -1 -2 -2 -3 -3 -1 -2 -4  7 -1 -1 -4 -3 -2 -2 -1 -2 -4
 1 -1  1  0 -1  0  0  0 -1 -2 -2  0 -1 -2 -1  4  1 -3 -2 -2  0  0  0 -4
 0 -1  0 -1 -1 -1 -1 -2 -2 -1 -1 -1 -1 -2 -1  1  5 -2 -2  0 -1 -1  0 -4
-3 -3 -4 -4 -2 -2 -3 -2 -2 -3 -2 -3 -1  1 -4 -3 -2 11  2 -3 -4 -3 -2 -4
-2 -2 -2 -3 -2 -1 -2 -3  2 -1 -1 -2 -1  3 -3 -2 -2  2  7 -1 -3 -2 -1 -4
 0 -3 -3 -3 -1 -2 -2 -3 -3  3  1 -2  1 -1 -2 -2  0 -3 -1  4 -3 -2 -1 -4
-2 -1  3  4 -3  0  1 -1  0 -3 -4  0 -3 -3 -2  0 -1 -4 -3 -3  4  1 -1 -4
-1  0  0  1 -3  3  4 -2  0 -3 -3  1 -1 -3 -1  0 -1 -3 -2 -2  1  4 -1 -4
 0 -1 -1 -1 -2 -1 -1 -1 -1 -1 -1 -1 -1 -1 -2  0  0 -2 -1 -1 -1 -1 -1 -4
-4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4 -4  1
"""
_AA_BACKGROUND = [0.074, 0.052, 0.045, 0.054, 0.025, 0.034, 0.054, 0.074, 0.026, 0.068,
                  0.099, 0.058, 0.025, 0.047, 0.039, 0.057, 0.051, 0.013, 0.032, 0.073]


def _protein():
    M = np.array(_BLOSUM62.split(), dtype=np.int8).reshape(24, 24)
    return LETTERS, M, 11, 1, np.array(_AA_BACKGROUND) / sum(_AA_BACKGROUND)


def _dna():
    M = np.full((4, 4), -3, np.int8)
    np.fill_diagonal(M, 2)
    return "ACGT", M, 5, 2, np.full(4, 0.25)


# ------------------------------------------------------------------ cases

def listed():
    return [
        # a handful of short proteins from a user's file: launches, copies and
        # synchronisations, hardly any cells
        dict(name="msa_24_short_proteins", kind="msa", alphabet="protein", n=24, median=60,
             sigma=0.25, lo=30, hi=120, families=1, ancestor=150, sub=0.30, indel=0.03, center="exact", many=0),
        # the plain protein family: 200 proteins of 200-400 residues, exact center
        dict(name="msa_200_proteins", kind="msa", alphabet="protein", n=200, median=290, sigma=0.2,
             lo=200, hi=400, families=1, ancestor=400, sub=0.30, indel=0.03, center="exact", many=0),
        # the headline: 10,000 uneven proteins of five families, all-pairs center
        dict(name="msa_10k_proteins", kind="msa", alphabet="protein", n=10000, median=350,
             sigma=0.6, lo=50, hi=2000, families=5, ancestor=2000, sub=0.40, indel=0.05, center="exact", many=0),
        # long chains beyond the 16-bit cells' range (the first one 3,600 residues
        # or more), as the longest of a protein collection are
        dict(name="msa_240_long_proteins", kind="msa", alphabet="protein", n=240, median=2200,
             sigma=0.4, lo=900, hi=5000, families=2, ancestor=5000, sub=0.40, indel=0.05, center="longest", many=0),
        # short peptides against their 500-residue precursor (a given center)
        dict(name="msa_200k_peptides", kind="msa", alphabet="protein", n=200000, median=90, sigma=0.6,
             lo=30, hi=200, families=1, ancestor=500, sub=0.30, indel=0.03, center="ancestor", many=0),
        # similar nucleotides, the first sequence as the center (the paper's choice)
        dict(name="msa_20k_similar_dna", kind="msa", alphabet="dna", n=20000, median=1500, sigma=0.04,
             lo=1400, hi=1600, families=1, ancestor=1600, sub=0.02, indel=0.005, center="first", many=0),
        # the learned center: the network's 64 best candidates refined exactly
        dict(name="msa_10k_proteins_learned", kind="msa", alphabet="protein", n=10000, median=350,
             sigma=0.6, lo=50, hi=2000, families=5, ancestor=2000, sub=0.40, indel=0.05, center="refined", many=64),
        # the exact center over a reference sample, where all pairs are too many
        dict(name="center_3k_dna_100_refs", kind="center", alphabet="dna", n=3000, median=1500,
             sigma=0.04, lo=1400, hi=1600, families=1, ancestor=1600, sub=0.02, indel=0.005, center="sampled", many=100),
        # similar nucleotides through 8-residue center segments (the paper's trie path)
        dict(name="anchored_50k_similar_dna", kind="anchored", alphabet="dna", n=50000, median=1500,
             sigma=0.04, lo=1400, hi=1600, families=1, ancestor=1600, sub=0.02, indel=0.005, center="first", many=8),
        # exact scores of a list of pairs: the selector's training targets
        dict(name="scores_60k_pairs", kind="pairs", alphabet="protein", n=5000, median=300, sigma=0.6,
             lo=50, hi=2000, families=20, ancestor=2000, sub=0.40, indel=0.05, center="", many=60000),
        # one training batch of the selector: 256 pairs, forward and backward
        dict(name="selector_grad_256_pairs", kind="grad", alphabet="protein", n=2000, median=300,
             sigma=0.6, lo=50, hi=2000, families=20, ancestor=2000, sub=0.40, indel=0.05, center="", many=256),
        # the neighbour-joining tree of a merged protein alignment
        dict(name="tree_4k_proteins", kind="tree", alphabet="protein", n=4000, median=350, sigma=0.6,
             lo=50, hi=2000, families=5, ancestor=2000, sub=0.40, indel=0.05, center="first", many=0),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["msa", "msa", "msa", "center", "anchored", "pairs", "grad", "tree"])
        dna = kind == "anchored" or (kind in ("msa", "center", "pairs") and rng.random() < 0.3)
        median = _log(rng, 1000, 1900) if kind == "anchored" else _log(rng, 45, 2400)
        c = dict(kind=kind, alphabet="dna" if dna else "protein", median=median,
                 sigma=round(rng.uniform(0.02, 0.08) if dna else rng.uniform(0.1, 0.6), 2))
        c["lo"] = max(20, int(median * (0.9 if dna else rng.uniform(0.2, 0.7))))
        c["hi"] = int(median * (1.1 if dna else rng.uniform(1.5, 4.0)))
        c["ancestor"] = c["hi"]
        c["families"] = 1 if dna else rng.randint(1, 20)
        c["sub"], c["indel"] = (0.02, 0.005) if dna else (round(rng.uniform(0.3, 0.4), 2),
                                                          round(rng.uniform(0.03, 0.05), 3))
        c["center"], c["many"] = "", 0
        if kind == "msa":
            c["center"] = rng.choice(["exact", "exact", "first", "first", "ancestor", "longest", "refined"])
            c["n"] = _log(rng, 8, {"exact": 10000, "refined": 10000}.get(c["center"], 200000))
            c["many"] = min(c["n"], rng.randint(16, 128)) if c["center"] == "refined" else 0
        elif kind == "center":
            c["center"], c["n"] = "sampled", _log(rng, 100, 20000)
            c["many"] = min(c["n"], _log(rng, 10, 1000))
        elif kind == "anchored":
            c["center"], c["n"], c["many"] = "first", _log(rng, 200, 50000), rng.choice([8, 8, 10, 12])
        elif kind == "pairs":
            c["n"], c["many"] = _log(rng, 50, 10000), _log(rng, 16, 60000)
        elif kind == "grad":
            c["n"], c["many"] = _log(rng, 100, 5000), _log(rng, 16, 256)
            c["median"] = min(median, 600)
            c["lo"], c["hi"] = min(c["lo"], c["median"]), min(c["hi"], 2000)
            c["ancestor"] = c["hi"]
        else:
            c["center"], c["n"] = "first", _log(rng, 40, 4500)
        c["lo"] = min(c["lo"], c["median"])
        # chains beyond the 16-bit cells cost more per cell; rows and traceback
        # codes are held three times over
        if _cost(c) * (3 if c["hi"] > 2900 else 1) <= most and c["hi"] <= 8000 and \
                c["n"] * c["median"] <= 45e6 and _cells_to_center(c) <= 1.2e11:
            return c


# ------------------------------------------------------------------ inputs

def _lengths(case, gen):
    x = torch.randn(case["n"], generator=gen, device=gen.device, dtype=torch.float64)
    L = torch.exp(math.log(case["median"]) + case["sigma"] * x)
    return L.round().clamp(case["lo"], case["hi"]).to(torch.int64)


def _make_set(case, seed):
    """(letters uint8 CUDA tensor, offsets int64 numpy, family int64 CUDA tensor)."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(1704 * 1000003 + int(seed))
    letters, M, _, _, bg = _protein() if case["alphabet"] == "protein" else _dna()
    k = len(bg)
    bgc = torch.tensor(np.cumsum(bg)[:-1], device=dev, dtype=torch.float32)

    def draw_residues(count):
        return torch.bucketize(torch.rand(count, generator=gen, device=dev), bgc, right=True)

    F, A, n = case["families"], case["ancestor"], case["n"]
    anc = draw_residues(F * A).reshape(F, A)
    L = torch.minimum(_lengths(case, gen), torch.tensor(A, device=dev))
    fam = torch.randint(0, F, (n,), generator=gen, device=dev)
    start = (torch.rand(n, generator=gen, device=dev) * (A - L + 1)).to(torch.int64)
    first = torch.cumsum(L, 0) - L
    seq = torch.repeat_interleave(torch.arange(n, device=dev), L)
    at = torch.arange(seq.numel(), device=dev) - first[seq] + start[seq]
    res = anc[fam[seq], at]
    total = res.numel()
    # substitutions: b != a with probability ~ p_b 2^(M[a][b] / 2)
    w = bg[None, :] * np.exp2(M[:k, :k].astype(np.float64) / 2.0)
    np.fill_diagonal(w, 0.0)
    cdf = torch.tensor(np.cumsum(w / w.sum(1, keepdims=True), 1)[:, :-1], device=dev, dtype=torch.float32)
    hit = (torch.rand(total, generator=gen, device=dev) < case["sub"]).nonzero()[:, 0]
    u = torch.rand(hit.numel(), generator=gen, device=dev)
    res[hit] = (cdf[res[hit]] <= u[:, None]).sum(1)
    # indels: an event is an insertion after its position or a deletion from
    # it on, one to three residues (the first residue of a sequence stays)
    ev = torch.rand(total, generator=gen, device=dev) < case["indel"]
    ins = torch.rand(total, generator=gen, device=dev) < 0.5
    size = torch.randint(1, 4, (total,), generator=gen, device=dev)
    count = torch.ones(total, dtype=torch.int64, device=dev)
    dele = torch.zeros(total, dtype=torch.bool, device=dev)
    for d in range(3):
        gone = ev & ~ins & (size > d)
        dele[d:] |= gone[:total - d] if d else gone
    dele[first] = False
    count[dele] = 0
    count += torch.where(ev & ins, size, torch.zeros_like(size))
    out = torch.repeat_interleave(res, count)
    where = torch.cumsum(count, 0) - count
    new = torch.ones(out.numel(), dtype=torch.bool, device=dev)
    new[where[~dele]] = False
    slots = new.nonzero()[:, 0]
    out[slots] = draw_residues(slots.numel())
    lens = torch.zeros(n, dtype=torch.int64, device=dev).index_add_(0, seq, count)
    if case["center"] == "ancestor":  # the unmutated precursor comes first
        out = torch.cat([anc[0], out])
        lens = torch.cat([torch.tensor([A], device=dev), lens])
        fam = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), fam])
    if int(lens.max()) > B.MSA_MAX_LEN:
        raise ValueError("a sequence beyond %d residues" % B.MSA_MAX_LEN)
    table = torch.tensor(np.frombuffer(letters.encode(), np.uint8).copy(), device=dev)
    offsets = np.zeros(lens.numel() + 1, np.int64)
    offsets[1:] = np.cumsum(lens.cpu().numpy())
    return table[out], offsets, fam


def _params(rng, alphabet):
    """The network's parameters, flat: per layer W [9][cin][cout] and bias."""
    parts = []
    for cin, cout, used, gain in ((32, 128, alphabet, 6.0), (128, 128, 128, 6.0),
                                  (128, 128, 128, 6.0), (128, 64, 128, 3.0)):
        a = math.sqrt(gain / (9 * used))
        W = rng.uniform(-a, a, (9, cin, cout)).astype(np.float32)
        W[:, used:] = 0.0
        parts += [W.ravel(), rng.uniform(-0.05, 0.05, cout).astype(np.float32)]
    return np.concatenate(parts)


def _pair_list(case, rng, n, fam):
    """Half within-family, half uniform pairs of different sequences."""
    m = case["many"]
    a = rng.integers(0, n, m)
    b = (a + rng.integers(1, n, m)) % n
    order = np.argsort(fam, kind="stable")
    lo = np.searchsorted(fam[order], fam[a])
    size = np.searchsorted(fam[order], fam[a], side="right") - lo
    near = order[lo + (rng.random(m) * size).astype(np.int64)]
    half = (np.arange(m) < m // 2) & (near != a)
    return np.stack([a, np.where(half, near, b)], 1).astype(np.int64)


def prepare(case, seed):
    letters, offsets, fam = _make_set(case, seed)
    alph, M, o, e, _ = _protein() if case["alphabet"] == "protein" else _dna()
    rng = np.random.default_rng([17, int(seed)])
    n = offsets.size - 1
    lens = np.diff(offsets)
    # small sets come from a user's host buffers, large ones are on the GPU
    if n <= 1000:
        letters = letters.cpu().numpy()
    s = dict(case=case, ctx=B.Context(M, alph, o, e), letters=letters, offsets=offsets, n=n,
             center=int(np.argmax(lens)) if case["center"] == "longest" else 0)
    h = s["ctx"].h
    if case["center"] == "sampled":
        s["refs"] = np.sort(rng.choice(n, case["many"], replace=False)).astype(np.int64)
    if case["center"] == "refined" or case["kind"] == "grad":
        s["params"] = _params(rng, M.shape[0])
        B.msa_selector_init(h, params=s["params"])
    if case["kind"] in ("pairs", "grad"):
        B.msa_load(h, letters, offsets)
        s["pairs"] = _pair_list(case, rng, n, fam.cpu().numpy())
        # distances of related and unrelated pairs at the trainer's scale (mean 50)
        s["targets"] = np.clip(rng.normal(50.0, 6.0, case["many"]), 0.0, None).astype(np.float32)
    if case["kind"] == "tree":
        B.msa_load(h, letters, offsets)
        B.msa_align_to_center(h, s["center"])
        B.msa_merge_gaps(h, want_rows=False)
    if case["kind"] in ("msa", "anchored"):
        s["rows"] = _row_buffer(s, n * _width_room(case))
    return s


def _width_room(case):
    """Columns of a row buffer that a user keeps for alignments like the case's:
    two flanks, and per center residue the longest of n rows' insertions (which
    grows with log n)."""
    longest = case["hi"] + case["hi"] // 8 + 64
    if case["center"] in ("ancestor", "longest"):
        longest = max(longest, case["ancestor"])
    return int(2 * longest + longest * (2 + 1.2 * math.log2(case["n"] + 1)))


def _row_buffer(s, size):
    """A flat buffer on the side that the letters come from: host or GPU."""
    if isinstance(s["letters"], np.ndarray):
        return np.zeros(size, np.uint8)
    return torch.zeros(size, dtype=torch.uint8, device="cuda")


def _rows(s):
    """(the buffer with the merged rows n x width in front, the width)."""
    h = s["ctx"].h
    _, W = B.msa_merge_gaps(h, want_rows=False)
    if s["n"] * W > len(s["rows"]):
        s["rows"] = _row_buffer(s, s["n"] * W)
    return B.msa_merge_gaps(h, out=s["rows"])


def run(s):
    case, h, n = s["case"], s["ctx"].h, s["n"]
    kind = case["kind"]
    if kind == "pairs":
        return {"scores": B.msa_pair_scores(h, s["pairs"])}
    if kind == "grad":
        loss, grad = B.msa_selector_grad(h, s["pairs"], s["targets"])
        return {"loss": loss, "grad": grad}
    if kind == "tree":
        joins, lengths = B.msa_nj_tree(h)
        return {"joins": joins, "lengths": lengths}
    B.msa_load(h, s["letters"], s["offsets"])
    scores = np.zeros(n, np.int32)
    if kind == "center":
        center, total = B.msa_select_center(h, B.MSA_CENTER_EXACT_SAMPLED, s["refs"])
        return {"center": center, "sum": total, "rowsums": B.msa_center_rowsums(h)}
    center, total = s["center"], 0
    if kind == "anchored":
        fallback = B.msa_align_anchored(h, center, case["many"], scores)
        rows, width = _rows(s)
        return {"fallback": fallback, "scores": scores, "rows": rows, "width": width, "sp": B.msa_sp_score(h)}
    if case["center"] == "exact":
        center, total = B.msa_select_center(h, B.MSA_CENTER_EXACT)
    elif case["center"] == "refined":
        center, total = B.msa_select_center_refined(h, case["many"])
    B.msa_align_to_center(h, center, scores)
    rows, width = _rows(s)
    return {"center": center, "sum": total, "scores": scores, "rows": rows, "width": width, "sp": B.msa_sp_score(h)}


# ------------------------------------------------------------------ work

def _mean_len(case):
    """(mean, mean of squares) of the clipped lognormal lengths."""
    if case["sigma"] == 0:
        return float(case["median"]), float(case["median"]) ** 2
    x = (np.arange(2000) + 0.5) / 2000
    z = torch.erfinv(torch.tensor(2 * x - 1)).numpy() * math.sqrt(2)
    L = np.clip(case["median"] * np.exp(case["sigma"] * z), case["lo"], min(case["hi"], case["ancestor"]))
    return float(L.mean()), float((L * L).mean())


def _cells_to_center(case):
    m, _ = _mean_len(case)
    Lc = case["ancestor"] if case["center"] in ("ancestor", "longest") else m
    return case["n"] * m * Lc if case["kind"] in ("msa", "tree") else 0.0


def work(case):
    """Residues in, results out; six integer operations per cell of the affine
    recurrence (two extensions, the diagonal's sum, three maxima), two
    operations per multiply-add of the network, one comparison per pair of
    residues of a tree's distances and one step per matrix entry it must read."""
    n, (m, _) = case["n"], _mean_len(case)
    total = n * m
    kind = case["kind"]
    if kind == "pairs":
        return {"bytes": total + 20 * case["many"], "flops": 6 * case["many"] * m * m}
    if kind == "grad":
        rows = min(n, 2 * case["many"]) * m
        taps = 9 * (32 * 128 + 2 * 128 * 128)
        par = 4 * (9 * (32 * 128 + 2 * 128 * 128 + 128 * 64) + 448)
        return {"bytes": rows + 2 * par, "flops": 6.0 * rows * taps}
    if kind == "tree":
        width = 2 * m  # the least columns the rows could have is about their mean length
        return {"bytes": n * width + 24 * n, "flops": n * n / 2 * m + n * n}
    if kind == "center":
        return {"bytes": total + 8 * n, "flops": 6 * total * case["many"] * m}
    if kind == "anchored":
        return {"bytes": total + n * 1.1 * m, "flops": 8 * total}
    cells = _cells_to_center(case)
    if case["center"] == "exact":
        cells += total * total / 2
    elif case["center"] == "refined":
        cells += total * case["many"] * m
    return {"bytes": total + n * 2 * m, "flops": 6 * cells}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


# ------------------------------------------------------------------ exact

def exact(case, seed):
    """The selector's loss and gradient in 64 bits (plain torch); the other
    kinds return whole numbers, bytes and correctly rounded divisions of whole
    numbers."""
    if case["kind"] != "grad":
        return None
    dev = torch.device("cuda")
    letters, offsets, fam = _make_set(case, seed)
    alph, M, _, _, _ = _protein()
    rng = np.random.default_rng([17, int(seed)])
    n = offsets.size - 1
    flat = _params(rng, M.shape[0])
    pairs = _pair_list(case, rng, n, fam.cpu().numpy())
    targets = np.clip(rng.normal(50.0, 6.0, case["many"]), 0.0, None).astype(np.float32)
    p = torch.tensor(flat, device=dev, dtype=torch.float64, requires_grad=True)
    lut = torch.zeros(256, dtype=torch.int64, device=dev)
    lut[torch.tensor(np.frombuffer(alph.encode(), np.uint8).copy(), device=dev).long()] = \
        torch.arange(len(alph), device=dev)
    code = lut[letters.long()]
    used, local = np.unique(pairs, return_inverse=True)
    local = torch.tensor(local.reshape(-1, 2), device=dev)
    lens = np.diff(offsets)[used]
    # sequences one after another, four zero rows before, between and after
    base = 4 + np.concatenate([[0], np.cumsum(lens + 4)[:-1]])
    T = int(base[-1] + lens[-1] + 4)
    row = torch.tensor(np.concatenate([np.arange(b, b + k) for b, k in zip(base, lens)]), device=dev)
    src = torch.tensor(np.concatenate([np.arange(offsets[u], offsets[u + 1]) for u in used]), device=dev)
    owner = torch.tensor(np.repeat(np.arange(used.size), lens), device=dev)
    x = torch.zeros(T, 32, dtype=torch.float64, device=dev)
    x[row, code[src]] = 1.0
    valid = torch.zeros(T, 1, dtype=torch.float64, device=dev)
    valid[row] = 1.0
    at = 0
    for layer, (cin, cout) in enumerate(((32, 128), (128, 128), (128, 128), (128, 64))):
        W = p[at:at + 9 * cin * cout].reshape(9, cin, cout)
        at += 9 * cin * cout
        b = p[at:at + cout]
        at += cout
        pad = torch.nn.functional.pad(x, (0, 0, 4, 4))
        y = b + sum(pad[t:t + T] @ W[t] for t in range(9))
        x = (torch.relu(y) if layer < 3 else y) * valid
    L = torch.tensor(lens, device=dev, dtype=torch.float64)
    emb = torch.zeros(used.size, 64, dtype=torch.float64, device=dev).index_add(0, owner, x[row])
    emb = emb / L.sqrt()[:, None]
    d = ((emb[local[:, 0]] - emb[local[:, 1]]) ** 2).sum(1)
    loss = ((d - torch.tensor(targets, device=dev, dtype=torch.float64)) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": p.grad.cpu().numpy()}
