"""The anchored alignment (the paper's trie path for similar nucleotides) on
the GPU against the oracle's: inserted-space rows, segments and the merged
MSA bit for bit, on the similar-DNA workload for several segment lengths,
with sequences sent to the local path (no match, a long unmatched stretch)
and on proteins."""
import numpy as np
import pytest

import oracle
from seqgen import dna_matrix, pack_sequences
from tests._gpu import binding, workload, make_ctx, oracle_problem

pytestmark = pytest.mark.gpu


def _check(b, h, prob, center, k, letters, offsets):
    scores = np.zeros(prob.n, np.int32)
    nf = b.msa_align_anchored(h, center, k, scores)
    seg, ins, occ = b.msa_alignment_info(h)
    rows, W = b.msa_merge_gaps(h)
    oseg, oins, oocc = oracle.anchored_all(prob, center, k)
    assert (ins == oins).all() and (occ == oocc).all()
    assert (seg == oseg).all() and (scores == oseg[:, 0]).all()
    oG, oW, orows = oracle.merge(prob, center, oins, oocc)
    assert W == oW and (rows == orows).all()
    return nf


@pytest.mark.parametrize("k", [8, 12, 16])
def test_similar_dna_matches_the_oracle(k):
    b = binding()
    letters, offsets, w, alph, M = workload("similar_dna_100k", n=300, seed=7)
    prob = oracle_problem(letters, offsets, alph, M, w.gap_open, w.gap_extend)
    with make_ctx(alph, M, w.gap_open, w.gap_extend) as h:
        b.msa_load(h, letters, offsets)
        nf = _check(b, h, prob, 0, k, letters, offsets)
    print("k", k, "sequences on the local path", nf)


def test_local_path_for_unanchored_and_long_stretches():
    """A random sequence (no match), one with a 120-residue foreign stretch
    between anchors (longer than the 80 a lane aligns), and similar ones."""
    b = binding()
    alph, M = dna_matrix(2, -3)
    rng = np.random.default_rng(3)
    bases = np.frombuffer(b"ACGT", np.uint8)
    center = bases[rng.integers(0, 4, 600)]
    seqs = [center.copy()]
    seqs.append(bases[rng.integers(0, 4, 300)])                          # unrelated
    seqs.append(np.concatenate([center[:200], bases[rng.integers(0, 4, 120)], center[320:]]))
    for _ in range(20):                                                   # similar
        s = center.copy()
        hit = rng.random(s.size) < 0.03
        s[hit] = bases[rng.integers(0, 4, int(hit.sum()))]
        seqs.append(s[int(rng.integers(0, 40)):s.size - int(rng.integers(0, 40))])
    letters, offsets = pack_sequences(seqs)
    prob = oracle_problem(letters, offsets, alph, M, 5, 2)
    with make_ctx(alph, M, 5, 2) as h:
        b.msa_load(h, letters, offsets)
        nf = _check(b, h, prob, 0, 12, letters, offsets)
    assert nf >= 2


def test_proteins_with_short_segments():
    b = binding()
    letters, offsets, w, alph, M = workload("plain_protein_200", n=60, seed=4)
    prob = oracle_problem(letters, offsets, alph, M, w.gap_open, w.gap_extend)
    with make_ctx(alph, M, w.gap_open, w.gap_extend) as h:
        b.msa_load(h, letters, offsets)
        _check(b, h, prob, 5, 4, letters, offsets)
        with pytest.raises(b.MSAError):
            b.msa_align_anchored(h, 5, 13)          # 13 x 5 bits > 64


@pytest.mark.parametrize("k", [4, 8, 10, 16])
def test_stretch_sizes_and_repeated_segments(k):
    """Unmatched stretches of every shape the aligners divide (one lane: 8 and
    16 center residues x 24; the warp: up to 80 a side), several in one
    sequence, beside centers with repeated segments (many matches per segment
    and position, chains decided by the tie rules)."""
    b = binding()
    alph, M = dna_matrix(2, -3)
    rng = np.random.default_rng(100 + k)
    bases = np.frombuffer(b"ACGT", np.uint8)
    rnd = lambda n: bases[rng.integers(0, 4, n)]  # noqa: E731
    for repeats in (False, True):
        center = rnd(63 * k)
        if repeats:
            unit = center[:2 * k].copy()
            for at in (6, 14, 15, 30, 31, 32, 50):
                center[at * k:at * k + 2 * k] = unit[:center.size - at * k][:2 * k]
        seqs = [center]
        for lc, lx in [(1, 1), (1, 7), (1, 24), (1, 25), (2, 3), (2, 16), (2, 24), (2, 30), (3, 20),
                       (0, 1), (0, 33), (1, 0), (4, 40), (5, 79), (6, 80), (6, 81)]:
            lc = min(lc, 80 // k) if lc else 0
            parts = [center[:10 * k]]
            for at in (10, 24, 40):
                parts += [rnd(lx), center[(at + lc) * k:(at + 14 if at < 40 else 63) * k if at != 24 else 40 * k]]
            seqs.append(np.concatenate(parts))
        for rate in (0.02, 0.1, 0.2):
            for _ in range(6):
                s = center.copy()
                hit = rng.random(s.size) < rate
                s[hit] = rnd(int(hit.sum()))
                cut = int(rng.integers(1, s.size - 1))
                seqs.append(np.concatenate([s[:cut], rnd(int(rng.integers(0, 30))), s[cut + int(rng.integers(0, 30)):]]))
        seqs.append(np.tile(center[:2 * k], 12))
        letters, offsets = pack_sequences(seqs)
        prob = oracle_problem(letters, offsets, alph, M, 5, 2)
        with make_ctx(alph, M, 5, 2) as h:
            b.msa_load(h, letters, offsets)
            _check(b, h, prob, 0, k, letters, offsets)


@pytest.mark.parametrize("segments", [1, 2, 3])
def test_segments_with_many_matches(segments):
    """A run of one residue over one to three center segments, longer in the
    subjects: 9 to 90 matches of each of them, around the 16 that one lane
    orders and the sizes of the warp's network; and runs so long that the
    subject goes to the local path after the ordering."""
    b = binding()
    alph, M = dna_matrix(2, -3)
    rng = np.random.default_rng(50 + segments)
    pool = np.frombuffer(b"ACGT", np.uint8)
    center = rng.choice(pool, size=1300)
    at = 640
    center[at:at + 8 * segments] = ord("A")
    center[at - 1] = center[at + 8 * segments] = ord("C")
    seqs = [center]
    for matches in (9, 15, 16, 17, 18, 31, 32, 33, 34, 63, 64, 65, 66, 80, 140):
        for _ in range(3):
            s = center.copy()
            hit = rng.random(s.size) < 0.02
            s[hit] = rng.choice(pool, size=int(hit.sum()))
            s[at:at + 8 * segments] = ord("A")
            s[at - 1] = s[at + 8 * segments] = ord("C")
            extra = max(0, matches + 7 - 8 * segments)
            seqs.append(np.concatenate([s[:at], np.full(extra, ord("A"), np.uint8), s[at:]]))
    letters, offsets = pack_sequences(seqs)
    prob = oracle_problem(letters, offsets, alph, M, 5, 2)
    with make_ctx(alph, M, 5, 2) as h:
        b.msa_load(h, letters, offsets)
        nf = _check(b, h, prob, 0, 8, letters, offsets)
    assert 3 <= nf <= 9
