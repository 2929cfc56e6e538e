"""Alignment of similar sequences, where the fill leaves out columns that no
best path can reach: against the oracle with shifts, long indels, repeats (tied
and off-diagonal paths) and unrelated subjects among similar ones, and against
the int32 kernels (which fill every column) over several subjects per warp."""
import numpy as np
import pytest

import oracle
from seqgen import blosum62, dna_matrix, pack_sequences
from tests._gpu import binding, make_ctx, oracle_problem

pytestmark = pytest.mark.gpu


def mutate(rng, s, p, pool):
    s = s.copy()
    hit = rng.random(s.size) < p
    s[hit] = rng.choice(pool, size=int(hit.sum()))
    return s


def variants(rng, center, pool):
    """Subjects of every kind a window can meet, similar ones first."""
    L = center.size
    seqs = [mutate(rng, center, p, pool) for p in (0.0, 0.0, 0.01, 0.03, 0.05, 0.08, 0.15)]
    for k in (3, 20, 90, 250):
        seqs.append(mutate(rng, np.concatenate([center[:L // 2], center[L // 2 + k:]]), 0.02, pool))
        seqs.append(mutate(rng, np.concatenate([center[:L // 3], rng.choice(pool, size=k), center[L // 3:]]), 0.02, pool))
        seqs.append(mutate(rng, center[k:], 0.02, pool))
        seqs.append(mutate(rng, center[:L - k], 0.02, pool))
        seqs.append(np.concatenate([rng.choice(pool, size=k), center, rng.choice(pool, size=2 * k)]))
    # a segment repeated, moved to the other end, and halves swapped
    seqs.append(np.concatenate([center[:200], center[:200], center]))
    seqs.append(np.concatenate([center[-150:], center]))
    seqs.append(np.concatenate([center[L // 2:], center[:L // 2]]))
    seqs.append(np.tile(center[:60], 12))
    seqs.append(rng.choice(pool, size=L))
    seqs.append(rng.choice(pool, size=70))
    seqs.append(center[100:140])
    return seqs


@pytest.mark.parametrize("kind, o, e", [("dna", 5, 2), ("dna", 2, 1), ("dna", 3, 3), ("protein", 11, 1)])
@pytest.mark.parametrize("lanes", [8, 16, 32])
def test_similar_subjects_match_the_oracle(kind, o, e, lanes):
    b = binding()
    rng = np.random.default_rng(o * 100 + lanes)
    alph, M = blosum62() if kind == "protein" else dna_matrix()
    pool = np.frombuffer(("ARNDCQEGHILKMFPSTWYV" if kind == "protein" else "ACGT").encode(), np.uint8)
    half = rng.choice(pool, size=330)
    for center in (rng.choice(pool, size=700), np.concatenate([half, mutate(rng, half, 0.03, pool)])):
        letters, offsets = pack_sequences([center] + variants(rng, center, pool))
        prob = oracle_problem(letters, offsets, alph, M, o, e)
        oseg, oins, oocc, _, _, _ = oracle.msa(prob, 0)
        with make_ctx(alph, M, o, e) as h:
            b.msa_load(h, letters, offsets)
            b.msa_set_align_group(h, lanes)
            b.msa_align_to_center(h, 0)
            seg, ins, occ = b.msa_alignment_info(h)
        assert (seg == oseg).all()
        assert (ins == oins).all() and (occ == oocc).all()


@pytest.mark.parametrize("odd_every", [0, 13, 2, 1])
def test_several_subjects_per_warp_match_full_columns(odd_every):
    """Guesses that come from a warp's previous subjects, too high ones
    included: subjects that are unrelated or half as long at a rate (too many of
    them, and every column is filled)."""
    b = binding()
    rng = np.random.default_rng(odd_every)
    alph, M = dna_matrix()
    pool = np.frombuffer(b"ACGT", np.uint8)
    center = rng.choice(pool, size=300)
    seqs = [center]
    for x in range(24000):
        if odd_every and x % odd_every == 0:
            seqs.append(rng.choice(pool, size=int(rng.integers(60, 310))) if x & 1 else center[:int(rng.integers(100, 200))])
            continue
        s = mutate(rng, center, (0.0, 0.02, 0.06)[x % 3], pool)
        a, k = int(rng.integers(0, 30)), int(rng.integers(30, 270))
        seqs.append(np.concatenate([s[a:k], s[k + int(rng.integers(0, 6)):]]))
    letters, offsets = pack_sequences(seqs)
    got = []
    for precision in (b.MSA_AUTO, b.MSA_INT32):
        with make_ctx(alph, M, 5, 2, precision=precision) as h:
            b.msa_load(h, letters, offsets)
            b.msa_set_align_group(h, 8)
            b.msa_align_to_center(h, 0)
            got.append(b.msa_alignment_info(h))
    for x, y in zip(*got):
        assert (x == y).all()


@pytest.mark.parametrize("n, nref, length", [(1000, 30, 900), (2500, 25, 600), (260, 0, 900)])
@pytest.mark.parametrize("odd_every", [0, 9, 2])
def test_center_of_similar_sequences_matches_full_columns(n, nref, length, odd_every):
    """Row sums of the bounded center kernel (every pair, and a sample of
    references) against the int32 kernels, with unrelated, repeated and short
    sequences among the similar ones; an odd number of references leaves one
    lane of the last pair empty."""
    b = binding()
    rng = np.random.default_rng(n + odd_every)
    alph, M = dna_matrix()
    pool = np.frombuffer(b"ACGT", np.uint8)
    center = rng.choice(pool, size=length)
    seqs = []
    for x in range(n):
        if odd_every and x % odd_every == 0:
            seqs.append((rng.choice(pool, size=int(rng.integers(50, length))), np.tile(center[:90], 7),
                         center[:int(rng.integers(100, length))])[x % 3])
            continue
        s = mutate(rng, center, (0.0, 0.02, 0.06)[x % 3], pool)
        a, k = int(rng.integers(0, length // 8)), int(rng.integers(length // 8, length))
        seqs.append(np.concatenate([s[a:k], s[k + int(rng.integers(0, 40)):]]))
    letters, offsets = pack_sequences(seqs)
    refs = np.sort(rng.choice(n, size=max(nref - 1 + n % 2, 1), replace=False))
    got = []
    for precision in (b.MSA_AUTO, b.MSA_INT32):
        with make_ctx(alph, M, 5, 2, precision=precision) as h:
            b.msa_load(h, letters, offsets)
            if nref:
                c = b.msa_select_center(h, b.MSA_CENTER_EXACT_SAMPLED, refs=refs)
            else:
                c = b.msa_select_center(h, b.MSA_CENTER_EXACT)
            got.append((c, b.msa_center_rowsums(h)))
    assert got[0][0] == got[1][0]
    assert (got[0][1] == got[1][1]).all()


def test_autotune_times_the_full_fill_of_similar_subjects():
    """Two launches (fill and traceback) per timed shape: the bounded fill, which
    has a shape of its own, stays out; the next alignment has it again, and the
    vote and it are two launches more."""
    b = binding()
    rng = np.random.default_rng(3)
    alph, M = dna_matrix()
    pool = np.frombuffer(b"ACGT", np.uint8)
    center = rng.choice(pool, size=1500)
    letters, offsets = pack_sequences([mutate(rng, center, 0.02, pool) for _ in range(1400)])  # 3.15e9 cells
    with make_ctx(alph, M, 5, 2) as h:
        b.msa_load(h, letters, offsets)
        count = lambda: b.msa_stage_times(h)[1]["launches"]  # noqa: E731
        before = count()
        rates, _ = b.msa_align_autotune(h, 0)
        shapes = int((rates > 0).sum())
        assert shapes == 15 and count() - before == 2 * 2 * shapes  # (each shape runs twice)
        b.msa_set_align_group(h, 8)
        before = count()
        b.msa_align_to_center(h, 0)
        assert count() - before == 4


@pytest.mark.parametrize("kind, o, e", [("dna", 5, 2), ("dna", 2, 1), ("dna", 3, 3), ("protein", 11, 1)])
@pytest.mark.parametrize("lanes", [8, 16, 32])
def test_variants_among_many_similar_subjects(kind, o, e, lanes):
    """The subjects of test_similar_subjects_match_the_oracle, and again as many
    close ones as make the set a similar one (unrelated ones are few)."""
    b = binding()
    rng = np.random.default_rng(o * 1000 + lanes)
    alph, M = blosum62() if kind == "protein" else dna_matrix()
    pool = np.frombuffer(("ARNDCQEGHILKMFPSTWYV" if kind == "protein" else "ACGT").encode(), np.uint8)
    half = rng.choice(pool, size=330)
    for center in (rng.choice(pool, size=700), np.concatenate([half, mutate(rng, half, 0.03, pool)])):
        seqs = variants(rng, center, pool)
        # spread over the lengths: the sample of the vote is taken in their order
        close = [mutate(rng, center[:center.size - int(k)], 0.02, pool) for k in rng.integers(0, 300, 6 * len(seqs))]
        letters, offsets = pack_sequences([center] + seqs + close)
        prob = oracle_problem(letters, offsets, alph, M, o, e)
        oseg, oins, oocc, _, _, _ = oracle.msa(prob, 0)
        with make_ctx(alph, M, o, e) as h:
            b.msa_load(h, letters, offsets)
            b.msa_set_align_group(h, lanes)
            b.msa_align_to_center(h, 0)
            seg, ins, occ = b.msa_alignment_info(h)
        assert (seg == oseg).all()
        assert (ins == oins).all() and (occ == oocc).all()


def similar_set(rng, n, length, odd_every, pool):
    """n sequences cut from variants of one, every odd_every-th one unrelated or
    a repeat of its start."""
    center = rng.choice(pool, size=length)
    seqs = [center]
    for x in range(1, n):
        if odd_every and x % odd_every == 0:
            seqs.append(rng.choice(pool, size=int(rng.integers(length // 2, length))) if x & 1
                        else np.tile(center[:90], length // 100))
            continue
        s = mutate(rng, center, (0.0, 0.02, 0.04)[x % 3], pool)
        a, k = int(rng.integers(0, length // 20)), int(rng.integers(length // 8, length))
        seqs.append(np.concatenate([s[a:k], s[k + int(rng.integers(0, 40)):]]))
    return pack_sequences(seqs)


@pytest.mark.parametrize("n, length, budget", [(20500, 420, 0), (20500, 420, 1 << 29), (40000, 300, 0), (1500, 1500, 0)])
@pytest.mark.parametrize("odd_every", [0, 40])
def test_narrower_bounded_groups_and_batches(n, length, budget, odd_every):
    """The default shapes from 3e9 cells on: the bounded fill's groups narrower
    than the full fill's (its codes then lie in a buffer laid out for the wider
    ones), in one batch of codes and in several, against int32 cells."""
    b = binding()
    rng = np.random.default_rng(n + odd_every)
    alph, M = dna_matrix()
    letters, offsets = similar_set(rng, n, length, odd_every, np.frombuffer(b"ACGT", np.uint8))
    got, launches = [], 0
    for precision in (b.MSA_INT32, b.MSA_AUTO):
        with make_ctx(alph, M, 5, 2, precision=precision) as h:
            b.msa_load(h, letters, offsets)
            if budget:
                b.msa_set_codes_budget(h, budget)
            before = b.msa_stage_times(h)[1]["launches"]
            b.msa_align_to_center(h, 0)
            launches = b.msa_stage_times(h)[1]["launches"] - before
            got.append(b.msa_alignment_info(h))
    # a vote, and per batch the two fills and the traceback
    assert launches % 3 == 1 and (launches > 4) == (budget > 0)
    for x, y in zip(*got):
        assert (x == y).all()


# queries of several passes of the full kernel, 2e10 cells and more; few groups
# (60 x 400) take the 16 x 16 shape, the others 8 x 20
@pytest.mark.parametrize("n, nref, length", [(1200, 41, 1500), (2600, 24, 1300), (400, 60, 2600), (420, 0, 1300)])
@pytest.mark.parametrize("odd_every", [0, 60])
def test_bounded_center_beside_the_full_one(n, nref, length, odd_every):
    """Row sums over a sample of references (an odd and an even number) and over
    every pair, where the bounded kernel takes every multi-pass query.  A context
    under a memory limit plans the full kernel alone, with fewer launches."""
    b = binding()
    rng = np.random.default_rng(n + odd_every)
    alph, M = dna_matrix()
    letters, offsets = similar_set(rng, n, length, odd_every, np.frombuffer(b"ACGT", np.uint8))
    refs = np.sort(rng.choice(n, size=max(nref, 1), replace=False))
    got, launches = [], []
    for precision, limit in ((b.MSA_AUTO, 0), (b.MSA_AUTO, 1 << 35), (b.MSA_INT32, 0)):
        with make_ctx(alph, M, 5, 2, precision=precision) as h:
            b.msa_set_memory_limit(h, limit)
            b.msa_load(h, letters, offsets)
            before = b.msa_stage_times(h)[1]["launches"]
            c = (b.msa_select_center(h, b.MSA_CENTER_EXACT_SAMPLED, refs=refs) if nref
                 else b.msa_select_center(h, b.MSA_CENTER_EXACT))
            launches.append(b.msa_stage_times(h)[1]["launches"] - before)
            got.append((c, b.msa_center_rowsums(h)))
    assert launches[0] >= launches[1] + 2  # the vote and the bounded launch
    for c, sums in got[:2]:
        assert c == got[2][0] and (sums == got[2][1]).all()
