"""Rows that the rounds read from the graph itself, at the edges of their bins.

A vertex of small degree keeps one bit per row entry instead of a rewritten list and is read in
32-byte chunks, so what can go wrong sits at the bin limits, at rows that need all their colors
(cliques), at every alignment of the adjacency array, and at its two ends.
"""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gcpkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1205_3809_gb300 as m
    m.library()
    return m


def _cliques(degree, seed):
    """Cliques with rows of `degree`, two of them with edges missing, and a sparse random graph
    around them; ids shuffled.  About 300 such rows at least, so that a task of one block's warps
    takes all the steps it may."""
    k = degree + 1
    u, v = np.triu_indices(k, 1)
    parts, n = [], 0
    for i in range(max(5, 300 // k + 1)):
        drop = 0 if i not in (3, 4) else 1 + i % max(1, u.size - 1)
        parts.append((u[drop:] + n, v[drop:] + n))
        n += k
    g = gg.gnm(400, 1200, seed)
    src = np.repeat(np.arange(g.n), g.degrees)
    parts.append((src + n, g.colidx.astype(np.int64) + n))
    n += g.n
    perm = gg.permutation(n, seed + 1)
    us, vs = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    return gg.from_edges(n, perm[us], perm[vs], name=f"cliques({degree})")


@pytest.mark.parametrize("degree", [1, 7, 8, 9, 10, 20, 21, 22, 24, 25, 26, 31, 32, 33, 56, 57, 58, 63, 120, 121, 122])
@pytest.mark.parametrize("keyed", [False, True])
def test_bin_edges(gcpkg, degree, keyed):
    g = _cliques(degree, 100 + degree)
    prio = (gg.draws(degree, 3, g.n) % np.uint64(5)).astype(np.uint32) if keyed else None
    want = oracle.iterative(g.rowptr, g.colidx, prio)
    rp = torch.from_numpy(g.rowptr).cuda()
    pr = torch.from_numpy(prio.view(np.int32)).cuda() if keyed else None
    # one block for all rounds, and a launch per round: few warps, so several steps a task
    few = ({"tail_volume": 1 << 30}, {"loop_mode": 1}, {"tail_volume": 1 << 30, "color_bits": 32})
    for shift in (0, 1, 6):  # the adjacency array at other alignments, its ends at other chunks
        buf = torch.full((g.nnz + 16,), 1 << 30, dtype=torch.int32, device="cuda")
        ci = buf[shift:shift + g.nnz]
        ci.copy_(torch.from_numpy(g.colidx))
        for options in (None, {"small_max_degree": 8}, {"medium_max_degree": 64}, {"color_bits": 32}) + few:
            got = gcpkg.color(rp, ci, pr, options=options, round_sizes=True)
            assert (got.ncolors, got.rounds) == (want.ncolors, want.rounds), (g.name, shift, options)
            assert np.array_equal(got.colors.cpu().numpy(), want.colors)
            assert np.array_equal(got.round_sizes, want.round_sizes)


def _reordered(g, order, seed):
    """The same graph with the entries of every row shuffled or descending."""
    ci = g.colidx.copy()
    rng = np.random.default_rng(seed)
    for v in range(g.n):
        row = ci[g.rowptr[v]:g.rowptr[v + 1]]
        row[:] = rng.permutation(row) if order == "shuffled" else row[::-1]
    return ci


@pytest.mark.parametrize("order", ["shuffled", "descending"])
@pytest.mark.parametrize("make", [
    lambda: _cliques(9, 3), lambda: gg.star(34, 0), lambda: gg.star(258, 257), lambda: gg.star(259, 0),
    lambda: gg.complete(257), lambda: gg.star(5000, 0), lambda: gg.rmat(13, 8, gg.RMAT_B, 3), lambda: gg.gnm(3000, 40000, 5),
    # whole warps of rows of one and of two chunks to append
    lambda: gg.complete(300), lambda: gg.complete_bipartite(1100, 270),
])
def test_rows_in_any_order(gcpkg, make, order):
    """Round 1 looks at a row's first chunk first: rows whose only preceding neighbour comes late, at
    every alignment, and rows longer than its limit, with index and key priority."""
    g = make()
    ci = _reordered(g, order, 11)
    keys = (gg.draws(5, 3, g.n) % np.uint64(7)).astype(np.uint32)
    rp = torch.from_numpy(g.rowptr).cuda()
    for prio in (None, keys):
        want = oracle.iterative(g.rowptr, ci, prio)
        pr = None if prio is None else torch.from_numpy(prio.view(np.int32)).cuda()
        for shift in (0, 3):
            buf = torch.full((g.nnz + 16,), 1 << 30, dtype=torch.int32, device="cuda")
            dev = buf[shift:shift + g.nnz]
            dev.copy_(torch.from_numpy(ci))
            got = gcpkg.color(rp, dev, pr, round_sizes=True)
            assert (got.ncolors, got.rounds) == (want.ncolors, want.rounds), (g.name, order, shift)
            assert np.array_equal(got.colors.cpu().numpy(), want.colors)
            assert np.array_equal(got.round_sizes, want.round_sizes)


def test_four_vertices_a_thread_in_round_1(gcpkg):
    """A graph large enough for round 1's wide form (1,024 vertices for every SM), not a multiple of
    its blocks: skewed, sparse and edgeless parts and long rows, entries shuffled in their rows, with
    and without keys, at two alignments."""
    parts = [gg.rmat(17, 8, gg.RMAT_B, 3), gg.gnm(70001, 250000, 4), gg.star(3000, 7), gg.star(300, 299), gg.edgeless(501)]
    n, us, vs = 0, [], []
    for g in parts:
        us.append(np.repeat(np.arange(g.n, dtype=np.int64), g.degrees) + n)
        vs.append(g.colidx.astype(np.int64) + n)
        n += g.n
    assert n >= 152 * 1024 and n % 1024
    perm = gg.permutation(n, 9)
    g = gg.from_edges(n, perm[np.concatenate(us)], perm[np.concatenate(vs)])
    row = np.repeat(np.arange(n), g.degrees)
    ci = g.colidx[np.lexsort((np.random.default_rng(5).random(g.nnz), row))]
    keys = (gg.draws(6, 3, n) % np.uint64(9)).astype(np.uint32)
    rp = torch.from_numpy(g.rowptr).cuda()
    for prio in (None, keys):
        want = oracle.iterative(g.rowptr, ci, prio)
        pr = None if prio is None else torch.from_numpy(prio.view(np.int32)).cuda()
        for shift in (0, 5):
            buf = torch.full((g.nnz + 16,), 1 << 30, dtype=torch.int32, device="cuda")
            dev = buf[shift:shift + g.nnz]
            dev.copy_(torch.from_numpy(ci))
            got = gcpkg.color(rp, dev, pr, round_sizes=True)
            assert (got.ncolors, got.rounds) == (want.ncolors, want.rounds)
            assert np.array_equal(got.colors.cpu().numpy(), want.colors)
            assert np.array_equal(got.round_sizes, want.round_sizes)
