"""Pair scores of lists that take every width of the packed kernel and mix its
pairs with int32 ones, at the edges of the passes, against the oracle."""
import numpy as np
import pytest

import oracle
from seqgen import blosum62, dna_matrix, pack_sequences
from tests._gpu import binding, make_ctx, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npairs", [1, 2, 3, 17, 9729, 19457])
@pytest.mark.parametrize("kind,sat", [("protein", 0), ("protein", 300), ("dna", 0)])
def test_pair_lists(npairs, kind, sat):
    """1 pair to more than the widest group's limit; sat 300: only pairs whose
    shorter sequence is below 26 residues stay packed."""
    b = binding()
    rng = np.random.default_rng(npairs + sat)
    alph, M = blosum62() if kind == "protein" else dna_matrix()
    o, e = (11, 1) if kind == "protein" else (5, 2)
    pool = np.frombuffer(alph.encode(), dtype=np.uint8)
    lens = [1, 2, 15, 16, 25, 26, 27, 100, 127, 128, 129, 140]
    if npairs < 100:
        lens += [255, 256, 257, 511, 512, 513, 700, 1100]
    base = rng.choice(pool, size=max(lens))
    seqs = []
    for L in lens:
        s = base[:L].copy()
        hit = rng.random(L) < 0.3
        s[hit] = rng.choice(pool, size=int(hit.sum()))
        seqs += [s, rng.choice(pool, size=L)]
    letters, offsets = pack_sequences(seqs)
    prob = oracle_problem(letters, offsets, alph, M, o, e)
    n = len(seqs)
    pairs = rng.integers(0, n, size=(npairs, 2))
    if npairs == 17:
        pairs[:, 0], pairs[:, 1] = n - 2, np.arange(17)  # the longest against many
    with make_ctx(alph, M, o, e, sat_limit=sat) as h:
        b.msa_load(h, letters, offsets)
        got = b.msa_pair_scores(h, pairs)
    # (each of the n x n scores once)
    idx = np.array([(x, y) for x in range(n) for y in range(n)])
    want = oracle.pair_scores(prob, idx).reshape(n, n)
    assert (got == want[pairs[:, 0], pairs[:, 1]]).all()
