"""The path at its documented size limits, bit for bit against the oracle:
sequences of the maximum length (MSA_MAX_LEN residues: the center kernels'
longest queries, int32 cells, the most passes of the alignment kernels), the
anchored path's longest sequences (one residue short of MSA_MAX_LEN) and the
tree of such an MSA."""
import numpy as np
import pytest

import oracle
from oracle import nj as T
from seqgen import blosum62, dna_matrix, pack_sequences, STANDARD_AA
from tests._gpu import binding, make_ctx, oracle_problem
from tests.test_gpu_anchored import _check as anchored_check
from tests.test_gpu_parity import run_pipeline, check_against_oracle

pytestmark = pytest.mark.gpu


def mutants(rng, ancestor, pool, lengths, rate):
    """Copies of the ancestor with substitutions at `rate`, cut to `lengths`
    (each from a random start)."""
    out = []
    for L in lengths:
        s = ancestor.copy()
        hit = rng.random(s.size) < rate
        s[hit] = pool[rng.integers(0, pool.size, int(hit.sum()))]
        start = int(rng.integers(0, ancestor.size - L + 1))
        out.append(s[start:start + L])
    return out


def test_maximum_length_proteins():
    b = binding()
    alph, M = blosum62()
    rng = np.random.default_rng(17)
    pool = np.frombuffer(STANDARD_AA.encode(), np.uint8)
    Lmax = b.MSA_MAX_LEN
    ancestor = pool[rng.integers(0, pool.size, Lmax)]
    seqs = mutants(rng, ancestor, pool, [Lmax, Lmax, 5000, 1, 777], 0.3)
    letters, offsets = pack_sequences(seqs)
    prob = oracle_problem(letters, offsets, alph, M, 11, 1)
    oc, orow = oracle.exact_center(prob)
    with make_ctx(alph, M, 11, 1) as h:
        b.msa_load(h, letters, offsets)
        c, _ = b.msa_select_center(h, b.MSA_CENTER_EXACT)
        assert c == oc and (b.msa_center_rowsums(h) == orow).all()
        for center in sorted({c, 0}):  # the exact center and a maximum-length one
            out = run_pipeline(b, h, letters, offsets, center)
            check_against_oracle(prob, center, *out)
        joins, lengths = b.msa_nj_tree(h)  # of the last MSA
    _, _, _, _, _, orows = oracle.msa(prob, center)
    oj, ol = T.nj(T.msa_distances(orows))
    assert (joins == oj).all() and (lengths == ol).all()


def test_anchored_path_at_its_longest_sequences():
    b = binding()
    alph, M = dna_matrix(2, -3)
    rng = np.random.default_rng(23)
    pool = np.frombuffer(b"ACGT", np.uint8)
    L = b.MSA_MAX_LEN - 1
    ancestor = pool[rng.integers(0, 4, L)]
    seqs = [ancestor.copy()] + mutants(rng, ancestor, pool, [L, L - 3, 4000, 9], 0.02)
    letters, offsets = pack_sequences(seqs)
    prob = oracle_problem(letters, offsets, alph, M, 5, 2)
    with make_ctx(alph, M, 5, 2) as h:
        b.msa_load(h, letters, offsets)
        anchored_check(b, h, prob, 0, 8, letters, offsets)
        # one residue longer is beyond the anchored path's positions
        seqs2 = seqs + [np.concatenate([ancestor, pool[:1]])]
        l2, o2 = pack_sequences(seqs2)
        b.msa_load(h, l2, o2)
        with pytest.raises(b.MSAError) as ei:
            b.msa_align_anchored(h, 0, 8)
        assert ei.value.code == b.MSA_ERANGE


ROWS_OF_6120 = """
import numpy as np
from seqgen import dna_matrix, pack_sequences
from tests._gpu import binding, make_ctx
b = binding()
alph, M = dna_matrix()
s = np.random.default_rng(1).choice(np.frombuffer(b"ACGT", np.uint8), size=6120)
letters, offsets = pack_sequences([s, s, s[:5000]])
with make_ctx(alph, M, 5, 2) as h:
    b.msa_load(h, letters, offsets)
    b.msa_align_to_center(h, 0)
    rows, W = b.msa_merge_gaps(h)
rows = np.asarray(rows).reshape(3, W)
assert W == 6120 and (rows[0] == s).all() and (rows[1] == s).all()
assert (rows[2] == np.concatenate([s[:5000], np.full(1120, ord("-"), np.uint8)])).all()
"""


def test_rows_whose_staging_fills_the_default_shared_memory():
    """Eight rows of 6,113 to 6,128 columns take exactly the 48 KB that a kernel
    gets by default, static shared memory not counted.  (In a process of its own:
    wider rows raise the limit for good.)"""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", ROWS_OF_6120], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr


@pytest.mark.parametrize("kind, n, length", [("protein", 130, 300), ("dna", 70, 500), ("protein", 40, 60)])
def test_tree_distances_in_no_more_than_their_matrix(kind, n, length):
    """A limit that leaves room for the n x n distances alone, and for a few
    kilobytes more: the same distances as without one."""
    from seqgen import blosum62
    b = binding()
    rng = np.random.default_rng(n)
    alph, M = blosum62() if kind == "protein" else dna_matrix()
    pool = np.frombuffer(alph[:20].encode(), np.uint8)
    base = rng.choice(pool, size=length)
    seqs = []
    for _ in range(n):
        s = base[:int(rng.integers(length // 2, length + 1))].copy()
        hit = rng.random(s.size) < 0.1
        s[hit] = rng.choice(pool, size=int(hit.sum()))
        seqs.append(s)
    letters, offsets = pack_sequences(seqs)
    with make_ctx(alph, M, 11, 1) as h:
        b.msa_load(h, letters, offsets)
        b.msa_align_to_center(h, 0)
        b.msa_merge_gaps(h, want_rows=False)
        want = b.msa_tree_distances(h)
        held = b.msa_memory(h)[0]
        for more in (0, 4096, 20000, 60000, 200000):
            b.msa_set_memory_limit(h, held + (8 * n * n + 255) // 256 * 256 + more)
            assert (b.msa_tree_distances(h) == want).all()
        b.msa_set_memory_limit(h, held + 8 * n * n - 4096)
        with pytest.raises(b.MSAError) as ei:
            b.msa_tree_distances(h)
        assert ei.value.code == b.MSA_ENOMEM
        # the alignment is still there, and another one starts from it
        b.msa_set_memory_limit(h, 0)
        before = b.msa_alignment_info(h)
        b.msa_align_to_center(h, 0)
        assert all((x == y).all() for x, y in zip(before, b.msa_alignment_info(h)))
