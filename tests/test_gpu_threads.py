"""Two contexts of different sizes at work in two host threads: a kernel's
shared-memory limit is the process's, so neither call may depend on what the
other one needs."""
import threading

import numpy as np
import pytest

from seqgen import blosum62, dna_matrix, pack_sequences
from tests._gpu import binding, make_ctx

pytestmark = pytest.mark.gpu


def test_contexts_of_two_sizes_in_two_threads():
    b = binding()
    rng = np.random.default_rng(7)
    jobs = []
    for (alph, M), o, e, pool, length, n, reps in ((blosum62(), 11, 1, b"ARNDCQEGHILKMFPSTWYV", 1800, 10, 60),
                                                   (dna_matrix(), 5, 2, b"ACGT", 60, 12, 300)):
        pool = np.frombuffer(pool, np.uint8)
        base = rng.choice(pool, size=length)
        seqs = []
        for _ in range(n):
            s = base.copy()
            hit = rng.random(length) < 0.1
            s[hit] = rng.choice(pool, size=int(hit.sum()))
            seqs.append(s)
        letters, offsets = pack_sequences(seqs)
        pairs = np.array([[i, (i + 1) % n] for i in range(n)])
        jobs.append((alph, M, o, e, letters, offsets, pairs, reps))

    def once(h, pairs):
        b.msa_align_to_center(h, 0)
        seg, _, _ = b.msa_alignment_info(h)
        center, total = b.msa_select_center(h, b.MSA_CENTER_EXACT)
        return seg.tobytes(), np.asarray(b.msa_pair_scores(h, pairs)).tobytes(), center, total

    wanted, wrong = [], []
    for alph, M, o, e, letters, offsets, pairs, _ in jobs:
        with make_ctx(alph, M, o, e) as h:
            b.msa_load(h, letters, offsets)
            wanted.append(once(h, pairs))

    def work(job, want):
        alph, M, o, e, letters, offsets, pairs, reps = job
        try:
            with make_ctx(alph, M, o, e) as h:
                b.msa_load(h, letters, offsets)
                for _ in range(reps):
                    if once(h, pairs) != want:
                        wrong.append("another result")
                        return
        except Exception as x:  # noqa: BLE001 - reported by the test
            wrong.append(repr(x))

    threads = [threading.Thread(target=work, args=a) for a in zip(jobs, wanted)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
