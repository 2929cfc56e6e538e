"""Self scores of the center selection: diagonal sums where the matrix allows
them, alignments for sequences with letters of negative diagonal score and for
matrices whose diagonal does not dominate -- always the oracle's row sums."""
import numpy as np
import pytest

import oracle
from seqgen import blosum62, pack_sequences
from tests._gpu import binding, make_ctx, oracle_problem

pytestmark = pytest.mark.gpu

# lengths around the 16-byte chunks and the 512-residue stride of a warp
LENGTHS = (1, 2, 15, 16, 17, 31, 33, 255, 511, 512, 513, 600)


@pytest.mark.parametrize("kind", ["plain", "negative_letters", "all_negative", "not_dominant"])
def test_row_sums_with_every_kind_of_self_score(kind):
    b = binding()
    rng = np.random.default_rng(31)
    alph, M = blosum62()
    M = M.copy()
    emit = "ARNDCQEGHILKMFPSTWYV"
    if kind == "negative_letters":
        emit = "ARNDCX*BZX"          # X scores -1 against itself
    if kind == "all_negative":
        emit = "X"
    if kind == "not_dominant":
        M[0, 4] = M[4, 0] = 11       # 2 s(A, C) > s(A, A) + s(C, C)
    pool = np.frombuffer(emit.encode(), dtype=np.uint8)
    letters, offsets = pack_sequences([rng.choice(pool, size=L) for L in LENGTHS])
    prob = oracle_problem(letters, offsets, alph, M, 11, 1)
    refs = np.array([0, 4, 9])
    with make_ctx(alph, M, 11, 1) as h:
        b.msa_load(h, letters, offsets)
        oc, orow = oracle.exact_center(prob)
        c, s = b.msa_select_center(h, b.MSA_CENTER_EXACT)
        assert (b.msa_center_rowsums(h) == orow).all()
        assert c == oc and s == orow[oc]
        oc, orow = oracle.exact_center(prob, refs=refs)
        c, s = b.msa_select_center(h, b.MSA_CENTER_EXACT_SAMPLED, refs=refs)
        assert (b.msa_center_rowsums(h) == orow).all()
        # the candidates' row sums over a reference view
        b.msa_selector_init(h, seed=3)
        c, s = b.msa_select_center_refined(h, len(LENGTHS), refs=refs)
        assert c == oc and s == orow[oc]
