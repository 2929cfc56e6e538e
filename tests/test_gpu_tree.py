"""The neighbour-joining tree on the GPU against the tree oracle, through the
C ABI: distances of the merged rows and every join (children and branch
lengths) bit for bit."""
import numpy as np
import pytest

import oracle
from oracle import nj as T
from tests._gpu import binding, workload, make_ctx, oracle_problem
from tests.test_oracle_nj import random_tree

pytestmark = pytest.mark.gpu


def any_ctx():
    from seqgen import dna_matrix
    alph, M = dna_matrix()
    return make_ctx(alph, M, 5, 2)


@pytest.mark.parametrize("n,seed", [(3, 1), (4, 2), (40, 3), (300, 4), (700, 5)])
def test_nj_of_additive_distances(n, seed):
    """Distances read off a random tree: the GPU joins equal the oracle's
    (which recovers the tree); 700 rows cross the packing of the matrix."""
    b = binding()
    tj, tl, D = random_tree(np.random.default_rng(seed), n)
    oj, ol = T.nj(D)
    with any_ctx() as h:
        joins, lengths = b.msa_nj(h, D)
    assert (joins == oj).all() and (lengths == ol).all()
    assert T.splits(joins, lengths, n) == T.splits(tj, tl, n)


def test_nj_ties_small_and_unbalanced():
    b = binding()
    cases = [np.zeros((1, 1), np.int64), np.array([[0, 7], [7, 0]], np.int64)]
    eq = np.full((9, 9), 2, np.int64)
    np.fill_diagonal(eq, 0)
    cases.append(eq)  # every Q ties at every join
    rng = np.random.default_rng(7)
    R = rng.integers(0, 1 << 20, size=(600, 600)).astype(np.int64)
    R = np.triu(R, 1)
    cases.append(R + R.T)  # no tree behind it: odd and negative updates floor
    with any_ctx() as h:
        for D in cases:
            oj, ol = T.nj(D)
            joins, lengths = b.msa_nj(h, D)
            assert (joins == oj).all() and (lengths == ol).all(), D.shape


def test_nj_from_device_memory_and_range_check():
    import torch
    b = binding()
    _, _, D = random_tree(np.random.default_rng(9), 50)
    oj, ol = T.nj(D)
    with any_ctx() as h:
        joins, lengths = b.msa_nj(h, torch.from_numpy(D).cuda())
        assert (joins == oj).all() and (lengths == ol).all()
        big = np.array([[0, 1 << 42, 1 << 42], [1 << 42, 0, 1 << 42], [1 << 42, 1 << 42, 0]],
                       np.int64)
        with pytest.raises(b.MSAError) as ei:
            b.msa_nj(h, big)
        assert ei.value.code == b.MSA_ERANGE
        joins, lengths = b.msa_nj(h, D)  # the context stays usable
        assert (joins == oj).all()


@pytest.mark.parametrize("name,n", [("plain_protein_200", 200), ("batched_uneven_10k", 700),
                                    ("similar_dna_100k", 120)])
def test_tree_of_the_msa(name, n):
    """The whole path to the tree: MSA rows, their distances and the joins
    equal the oracle's, computed from the oracle's own MSA."""
    b = binding()
    letters, offsets, w, alph, M = workload(name, n=n, seed=21)
    prob = oracle_problem(letters, offsets, alph, M, w.gap_open, w.gap_extend)
    center = int(np.argsort(np.diff(offsets), kind="stable")[n // 2])
    _, _, _, _, _, orows = oracle.msa(prob, center)
    od = T.msa_distances(orows)
    oj, ol = T.nj(od)
    with make_ctx(alph, M, w.gap_open, w.gap_extend) as h:
        b.msa_load(h, letters, offsets)
        with pytest.raises(b.MSAError):
            b.msa_tree_distances(h)  # before an alignment and merge
        b.msa_align_to_center(h, center)
        b.msa_merge_gaps(h, want_rows=False)
        d = b.msa_tree_distances(h)
        joins, lengths = b.msa_nj_tree(h)
    assert (d == od).all()
    assert (joins == oj).all() and (lengths == ol).all()


@pytest.mark.parametrize("name,n,frac,cap", [("batched_uneven_10k", 600, 0.1, 6),
                                             ("similar_dna_100k", 400, 0.1, 8),
                                             ("plain_protein_200", 200, 0.2, 5),
                                             ("plain_protein_200", 120, 0.1, 1)])
def test_clustered_tree_of_the_msa(name, n, frac, cap):
    """The clustered tree (sample tree cut into clusters, rows labelled, one
    outgroup-rooted tree per cluster, grafted back): joins, branch lengths and
    labels equal the oracle's on its own MSA."""
    b = binding()
    letters, offsets, w, alph, M = workload(name, n=n, seed=33)
    prob = oracle_problem(letters, offsets, alph, M, w.gap_open, w.gap_extend)
    center = int(np.argsort(np.diff(offsets), kind="stable")[n // 2])
    _, _, _, _, _, orows = oracle.msa(prob, center)
    sample = np.sort(np.random.default_rng(4).choice(n, max(2, int(frac * n)), replace=False))
    oj, ol, oc = T.cluster_tree(T.msa_distances(orows), sample, cap)
    with make_ctx(alph, M, w.gap_open, w.gap_extend) as h:
        b.msa_load(h, letters, offsets)
        with pytest.raises(b.MSAError):
            b.msa_nj_cluster_tree(h, sample, cap)  # before a merge
        b.msa_align_to_center(h, center)
        b.msa_merge_gaps(h, want_rows=False)
        joins, lengths, cluster = b.msa_nj_cluster_tree(h, sample, cap)
        with pytest.raises(b.MSAError):
            b.msa_nj_cluster_tree(h, [0, n], cap)  # a row out of range
    assert (cluster == oc).all()
    assert (joins == oj).all() and (lengths == ol).all()
    print(name, "clusters", int(cluster.max()) + 1)


def test_clustered_tree_degenerate_cuts():
    """One sample row (a single cluster: the NJ tree of all rows) and every
    row sampled with a cap above them (no cut): both equal the oracle's and,
    as unrooted trees, the plain NJ tree."""
    b = binding()
    letters, offsets, w, alph, M = workload("plain_protein_200", n=90, seed=8)
    prob = oracle_problem(letters, offsets, alph, M, w.gap_open, w.gap_extend)
    _, _, _, _, _, orows = oracle.msa(prob, 5)
    D = T.msa_distances(orows)
    nj_splits = T.splits(*T.nj(D), 90)
    with make_ctx(alph, M, w.gap_open, w.gap_extend) as h:
        b.msa_load(h, letters, offsets)
        b.msa_align_to_center(h, 5)
        b.msa_merge_gaps(h, want_rows=False)
        for sample, cap in (([17], 1), (np.arange(90), 90)):
            oj, ol, oc = T.cluster_tree(D, sample, cap)
            joins, lengths, cluster = b.msa_nj_cluster_tree(h, sample, cap)
            assert (joins == oj).all() and (lengths == ol).all() and (cluster == oc).all()
            assert T.splits(joins, lengths, 90) == nj_splits


@pytest.mark.parametrize("n", [5, 33, 511, 513, 1030])
@pytest.mark.parametrize("kind", ["ties", "negative", "star"])
def test_nj_around_the_launch_sizes(n, kind):
    """Matrices at the sizes where the joins move from one CTA to a grid of
    them and where the matrix is packed: small integers (almost every Q ties),
    entries of both signs, and near-equal distances."""
    if n > 600 and kind == "negative":
        pytest.skip("the oracle's time")
    b = binding()
    rng = np.random.default_rng(n)
    lo, hi = {"ties": (1, 4), "negative": (-(1 << 19), 1 << 19), "star": (500000, 540000)}[kind]
    D = np.triu(rng.integers(lo, hi, size=(n, n)).astype(np.int64), 1)
    D = D + D.T
    oj, ol = T.nj(D)
    with any_ctx() as h:
        joins, lengths = b.msa_nj(h, D)
    assert (joins == oj).all() and (lengths == ol).all()


@pytest.mark.parametrize("kind", ["protein", "dna"])
@pytest.mark.parametrize("n,length", [(3, 1), (64, 31), (65, 33), (130, 479), (5, 481), (66, 965)])
def test_distances_around_the_tile_sizes(kind, n, length):
    """Merged rows of about `length` columns (words of 32, steps of 480) and
    row counts around the 64-row tiles, with three and five symbol planes."""
    from seqgen import blosum62, dna_matrix, pack_sequences
    b = binding()
    rng = np.random.default_rng(length)
    alph, M = blosum62() if kind == "protein" else dna_matrix()
    pool = np.frombuffer(alph.encode(), dtype=np.uint8)
    letters, offsets = pack_sequences(
        [rng.choice(pool, size=max(1, length - int(rng.integers(0, 3)))) for _ in range(n)])
    with make_ctx(alph, M, 11, 1) as h:
        b.msa_load(h, letters, offsets)
        b.msa_align_to_center(h, 0)
        rows, _ = b.msa_merge_gaps(h)
        d = b.msa_tree_distances(h)
    assert (d == T.msa_distances(rows)).all()


def nj_matrix(rng, n, kind):
    lo, hi = {"ties": (1, 4), "star": (500000, 540000)}[kind]
    D = np.triu(rng.integers(lo, hi, size=(n, n)).astype(np.int64), 1)
    return D + D.T


@pytest.mark.parametrize("n", [127, 128, 129, 700])
@pytest.mark.parametrize("kind", ["ties", "star"])
def test_nj_in_every_launch_shape(n, kind):
    """One CTA and a cluster around the size where they change over, clusters of
    8 and 16, every CTA size, row sums in shared and in global memory, and one
    CTA with several rows per thread: all give the oracle's joins."""
    b = binding()
    D = nj_matrix(np.random.default_rng(n), n, kind)
    oj, ol = T.nj(D)
    with any_ctx() as h:
        for ctas, threads in ((0, 0), (1, 0), (8, 256), (8, 512), (8, 1024), (16, 256), (16, 512), (16, 1024)):
            for sums_global in (False, True):
                b.msa_debug_nj_shape(h, ctas, threads, sums_global)
                joins, lengths = b.msa_nj(h, D)
                assert (joins == oj).all() and (lengths == ol).all(), (ctas, threads, sums_global)
        for bad in ((2, 0), (16, 128)):
            with pytest.raises(b.MSAError) as ei:
                b.msa_debug_nj_shape(h, *bad)
            assert ei.value.code == b.MSA_EINVAL


def additive(rng, n):
    """Path lengths (int64[n, n] on the GPU) of a random binary tree over n leaves
    with even, distinct edge lengths, the leaves in random order."""
    import torch
    depth, meet = np.zeros(n, np.int64), np.zeros(n - 1, np.int64)  # of a leaf; where k and k + 1 part
    edge = iter(2 * rng.permutation(np.arange(1, 2 * n)))
    stack = [(0, n, 0)]
    while stack:
        lo, hi, d = stack.pop()
        if hi - lo == 1:
            depth[lo] = d
            continue
        cut = int(rng.integers(lo + 1, hi))
        meet[cut - 1] = d
        stack += [(lo, cut, d + int(next(edge))), (cut, hi, d + int(next(edge)))]
    h, g = torch.tensor(depth, device="cuda"), torch.tensor(meet, device="cuda")
    D = torch.zeros(n, n, dtype=torch.int64, device="cuda")
    cols = torch.arange(n - 1, device="cuda")
    for r0 in range(0, n - 1, 1024):  # two leaves part at the smallest depth between them
        r = torch.arange(r0, min(n - 1, r0 + 1024), device="cuda")[:, None]
        part = torch.where(cols[None] < r, 1 << 40, g[None].expand(r.numel(), -1)).cummin(1).values
        D[r0:r0 + r.numel(), 1:] = torch.where(cols[None] < r, 0, h[r] + h[None, 1:] - 2 * part)
    D += D.T.clone()
    order = torch.tensor(rng.permutation(n), device="cuda")
    return D[order][:, order].contiguous()


def path_sums(n, edges, root, probe):
    """Distance of every leaf from each probe leaf, along the tree's edges."""
    up = {c: (p, w) for p, c, w in edges}
    kids = {}
    for p, c, w in edges:
        kids.setdefault(p, []).append((c, w))
    out = []
    for leaf in probe:
        dist, v, d, came = {}, leaf, 0.0, None
        while True:
            stack = [(v, d)]
            while stack:
                u, du = stack.pop()
                if u < n:
                    dist[u] = du
                stack += [(c, du + w) for c, w in kids.get(u, []) if c != came]
            if v == root:
                break
            came, (v, w) = v, up[v]
            d += w
        out.append([dist[k] for k in range(n)])
    return np.array(out)


@pytest.mark.parametrize("n", [1536, 1537, 8193, 16500, 23000])
def test_nj_of_additive_distances_at_large_sizes(n):
    """Sizes where the default launch changes (threads at 1,537 and 8,193 rows,
    several rows per thread above 16,384, row sums in global memory above 22,800):
    the distances of a tree give that tree back, so its path lengths are the matrix."""
    import torch
    b = binding()
    D = additive(np.random.default_rng(n), n)
    probe = np.random.default_rng(1).choice(n, size=12, replace=False)
    rows = D[torch.tensor(probe, device="cuda")].cpu().numpy()
    with any_ctx() as h:
        joins, lengths = b.msa_nj(h, D)
    joins, lengths = np.asarray(joins).reshape(-1, 2), np.asarray(lengths).reshape(-1, 2)
    assert sorted(joins.ravel().tolist()) == list(range(2 * n - 2))
    edges = [(n + t, int(joins[t, s]), float(lengths[t, s])) for t in range(n - 1) for s in range(2)]
    assert (path_sums(n, edges, 2 * n - 2, probe.tolist()) == rows).all()
