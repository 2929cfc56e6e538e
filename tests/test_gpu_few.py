"""The few-subject alignment (one CTA per subject, fill and traceback in one
launch) against the oracle at the edges of its strips (128 center rows), rounds
of strips (2,048 rows), step chunks (16 columns) and traceback windows
(128 columns x 128 rows), with gap runs longer than a warp."""
import numpy as np
import pytest

import oracle
from seqgen import blosum62, dna_matrix, pack_sequences
from tests._gpu import binding, make_ctx, oracle_problem

pytestmark = pytest.mark.gpu


def related(rng, center, L, pool):
    """About L residues cut from the center, mutated, with an indel."""
    L = min(L, center.size)
    a = int(rng.integers(0, center.size - L + 1))
    s = center[a:a + L].copy()
    hit = rng.random(L) < 0.2
    s[hit] = rng.choice(pool, size=int(hit.sum()))
    k = int(rng.integers(0, L + 1))
    return np.concatenate([s[:k], rng.choice(pool, size=int(rng.integers(0, 4))), s[k:]])


def check(letters, offsets, alph, M, o, e, center):
    b = binding()
    prob = oracle_problem(letters, offsets, alph, M, o, e)
    oseg, oins, oocc, _, oW, orows = oracle.msa(prob, center)
    with make_ctx(alph, M, o, e) as h:
        b.msa_load(h, letters, offsets)
        scores = np.zeros(offsets.size - 1, np.int32)
        b.msa_align_to_center(h, center, scores)
        seg, ins, occ = b.msa_alignment_info(h)
        rows, W = b.msa_merge_gaps(h)
    assert (seg == oseg).all() and (scores == oseg[:, 0]).all()
    assert (ins == oins).all() and (occ == oocc).all()
    assert W == oW and (rows == orows).all()


@pytest.mark.parametrize("kind", ["protein", "dna"])
@pytest.mark.parametrize("lc", [1, 4, 5, 127, 128, 129, 300, 2047, 2048, 2049, 4200])
def test_few_subjects_at_the_strip_edges(kind, lc):
    rng = np.random.default_rng(lc)
    alph, M = blosum62() if kind == "protein" else dna_matrix()
    o, e = (11, 1) if kind == "protein" else (5, 2)
    pool = np.frombuffer(("ARNDCQEGHILKMFPSTWYV" if kind == "protein" else "ACGT").encode(), np.uint8)
    center = rng.choice(pool, size=lc)
    lens = [1, 2, 15, 16, 17, 33, 48, 49, 130, 500, 2200]
    seqs = [center] + [related(rng, center, L, pool) for L in lens] + [rng.choice(pool, size=L) for L in (1, 40, 700)]
    letters, offsets = pack_sequences(seqs)
    check(letters, offsets, alph, M, o, e, 0)


@pytest.mark.parametrize("o,e", [(2, 1), (5, 5), (1, 1)])
def test_few_subjects_long_gaps_ties_and_no_score(o, e):
    """Deleted and inserted blocks of 20 to 400 residues (gap runs across lanes
    and windows), repeats (tied paths), and a subject without a positive cell."""
    rng = np.random.default_rng(o * 10 + e)
    alph, M = dna_matrix()
    M = M.copy()
    np.fill_diagonal(M, 5)
    pool = np.frombuffer(b"ACG", np.uint8)
    center = rng.choice(pool, size=900)
    seqs = [center]
    for k in (20, 32, 33, 64, 130, 400):
        seqs.append(np.concatenate([center[:250], center[250 + k:]]))
        seqs.append(np.concatenate([center[:300], rng.choice(pool, size=k), center[300:]]))
    seqs.append(np.tile(np.frombuffer(b"ACGACG", np.uint8), 40))
    seqs.append(np.full(50, ord("T"), np.uint8))
    letters, offsets = pack_sequences(seqs)
    check(letters, offsets, alph, M, o, e, 0)


@pytest.mark.parametrize("lc", [2305, 4200])
def test_few_subjects_at_the_ring_s_wrap(lc):
    """Centers of several rounds of strips against subjects of 64 q + 1
    residues: the last column of a round and the first of the next share a
    ring slot."""
    rng = np.random.default_rng(lc)
    alph, M = blosum62()
    pool = np.frombuffer(b"ARNDCQEGHILKMFPSTWYV", np.uint8)
    center = rng.choice(pool, size=lc)
    seqs = [center] + [center[a:a + L] for L in (769, 833, 1025) for a in (0, 500, lc - L)]
    seqs += [rng.choice(pool, size=L) for L in (769, 833, 1025)]
    letters, offsets = pack_sequences(seqs)
    check(letters, offsets, alph, M, 11, 1, 0)


@pytest.mark.parametrize("precision", ["AUTO", "INT32"])
def test_many_subjects_keep_the_codes_kernels(precision):
    """12,000 subjects, where one CTA per subject would be the slower choice: the
    default alignment (a fill and a traceback) and the anchored path's left-over
    subjects (all of them: no segment matches) against the oracle."""
    b = binding()
    rng = np.random.default_rng(12)
    alph, M = dna_matrix()
    pool = np.frombuffer(b"ACGT", np.uint8)
    center = rng.choice(pool, size=150)
    seqs = [center] + [related(rng, center, int(L), pool) for L in rng.integers(100, 151, 12000)]
    letters, offsets = pack_sequences(seqs)
    n = len(seqs)
    prob = oracle_problem(letters, offsets, alph, M, 5, 2)
    oseg, oins, oocc, _, _, _ = oracle.msa(prob, 0)
    foreign = pack_sequences([center] + [rng.choice(pool, size=int(L)) for L in rng.integers(100, 151, 12000)])
    fprob = oracle_problem(*foreign, alph, M, 5, 2)
    fseg, fins, focc = oracle.anchored_all(fprob, 0, 24)
    with make_ctx(alph, M, 5, 2, precision=getattr(b, "MSA_" + precision)) as h:
        b.msa_load(h, letters, offsets)
        before = b.msa_stage_times(h)[1]["launches"]
        b.msa_align_to_center(h, 0)
        assert b.msa_stage_times(h)[1]["launches"] - before == 2
        seg, ins, occ = b.msa_alignment_info(h)
        assert (seg == oseg).all() and (ins == oins).all() and (occ == oocc).all()
        b.msa_load(h, *foreign)
        before = b.msa_stage_times(h)[1]["launches"]
        assert b.msa_align_anchored(h, 0, 24) == n - 1
        assert b.msa_stage_times(h)[1]["launches"] - before == 3
        seg, ins, occ = b.msa_alignment_info(h)
        assert (seg == fseg).all() and (ins == fins).all() and (occ == focc).all()
