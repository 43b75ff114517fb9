"""The checks of every adjacency entry: accepted graphs of every row shape, and one wrong entry
at the places where a warp's flat walk, its long-row loop or its last task could miss it."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gcpkg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1205_3809_gb300 as m
    m.library()
    return m


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _many_long_rows():
    """70 rows of 8,200 in a row, among enough empty ones that a warp takes 32 and a block 256."""
    g = gg.complete_bipartite(70, 8200)
    return gg.from_edges(310000, np.repeat(np.arange(g.n), g.degrees), g.colidx, name="70 rows of 8,200")


GRAPHS = [
    lambda: gg.path(2), lambda: gg.path(65), lambda: gg.grid2d(37, 53, 1), lambda: gg.gnm(5000, 40000, 2),
    lambda: gg.complete(256), lambda: gg.complete(257), lambda: gg.complete(258),  # rows of 255, 256, 257
    lambda: gg.star(3001, 17), lambda: gg.rmat(12, 16, gg.RMAT_B, 3),
    # 16, 2 and 1 rows a warp (32, 8 and 4 above), the last with rows on both sides of 256
    lambda: gg.gnm(999, 3900, 4), lambda: gg.gnm(1501, 37000, 5), lambda: gg.gnm(301, 38600, 6),
    # rows for the whole block: one of 8,193, two of 9,000, and more than a block notes down (64)
    lambda: gg.star(8194, 5), lambda: gg.complete_bipartite(2, 9000), lambda: _many_long_rows(),
]


@pytest.mark.parametrize("make", GRAPHS)
def test_one_wrong_entry(gcpkg, make):
    g = make()
    rp = _dev(g.rowptr)
    assert gcpkg.validate_csr(rp, _dev(g.colidx)) == gcpkg.GC_OK
    row = np.repeat(np.arange(g.n), g.degrees)
    longest = int(np.argmax(g.degrees))
    for at in {0, g.nnz - 1, int(g.rowptr[longest]), int(g.rowptr[longest + 1]) - 1, g.nnz // 2}:
        for wrong in (g.n, -1, -2 ** 31, int(row[at]), (int(g.colidx[at]) + 1) % g.n):
            ci = g.colidx.copy()
            ci[at] = wrong
            if wrong == g.colidx[at]:
                continue
            assert gcpkg.validate_csr(rp, _dev(ci)) == gcpkg.GC_ERR_BAD_GRAPH, (g.name, at, wrong)
            res = gcpkg.color(rp, _dev(ci), options={"validate": 1}, check=False)
            assert res.status == gcpkg.GC_ERR_BAD_GRAPH
    assert gcpkg.color(rp, _dev(g.colidx), options={"validate": 1}).status == gcpkg.GC_OK


def test_row_starts_are_checked_first(gcpkg):
    """Unusable row starts are refused without a look at the entries they would point to."""
    g = gg.gnm(1000, 4000, 5)
    for i, x in ((0, 1), (500, -7), (500, 1 << 30)):
        rp = g.rowptr.copy()
        rp[i] = x
        assert gcpkg.validate_csr(_dev(rp), _dev(g.colidx)) == gcpkg.GC_ERR_BAD_GRAPH
