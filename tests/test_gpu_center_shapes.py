"""Kernel shapes of the center selection: queries at the edges of every shape's
rows, sets from a few alignments (wide groups, several graph branches) to enough
for stacked pairs -- always the oracle's row sums."""
import numpy as np
import pytest

import oracle
from seqgen import blosum62, pack_sequences
from tests._gpu import binding, make_ctx, oracle_problem

pytestmark = pytest.mark.gpu


def _edges():
    # G*R rows of every shape, one less and one more, and two passes of the widest
    rows = (96, 160, 192, 224, 256, 320, 384, 448, 640, 896)
    return [r + d for r in rows for d in (-1, 0, 1)] + [1793]


@pytest.mark.parametrize("lengths, sampled", [
    ((256, 384), (0,)),
    (tuple(_edges()), (0, 7, 13, 14, 22, 30)),
    (tuple(range(225, 257, 2)) * 6 + tuple(range(321, 385, 4)) * 6, (0, 1, 90, 150, 191)),
    ((1,) * 400 + (250, 380, 381), (0, 400, 401, 402)),
])
def test_row_sums_of_every_shape(lengths, sampled):
    b = binding()
    rng = np.random.default_rng(len(lengths))
    alph, M = blosum62()
    pool = np.frombuffer(b"ARNDCQEGHILKMFPSTWYV", dtype=np.uint8)
    letters, offsets = pack_sequences([rng.choice(pool, size=L) for L in lengths])
    prob = oracle_problem(letters, offsets, alph, M, 11, 1)
    refs = np.array(sampled)
    with make_ctx(alph, M, 11, 1) as h:
        b.msa_load(h, letters, offsets)
        oc, orow = oracle.exact_center(prob)
        c, s = b.msa_select_center(h, b.MSA_CENTER_EXACT)
        assert (b.msa_center_rowsums(h) == orow).all()
        assert c == oc and s == orow[oc]
        oc, orow = oracle.exact_center(prob, refs=refs)
        c, s = b.msa_select_center(h, b.MSA_CENTER_EXACT_SAMPLED, refs=refs)
        assert (b.msa_center_rowsums(h) == orow).all()
        assert c == oc and s == orow[oc]
