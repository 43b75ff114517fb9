"""The network's kernels and the features at the edges of their tiles, grids and rows."""
import numpy as np
import pytest

import graphgen as gg
from oracle import learned as L

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


def _uniform(seed, stream, count, lo, hi):
    u = (gg.draws(seed, stream, count) >> np.uint64(11)).astype(np.float64) / float(1 << 53)
    return (lo + (hi - lo) * u).astype(np.float32)


# 256 threads a block, a block an SM (152 of them): one sample a thread up to 38,912, two up to
# 77,824, then four, and 155,648 in a turn of the grid
@pytest.mark.parametrize("n", [1, 2, 255, 257, 511, 512, 513, 1023, 1025, 38912, 38913, 77824, 77825, 155647, 155649])
def test_forward_sizes(gcpkg, n):
    p = _uniform(n, 7, L.N_PARAMS, -0.3, 0.3)
    x = _uniform(n + 1, 9, n * L.N_IN, -2.0, 24.0).reshape(n, L.N_IN)
    got = gcpkg.mlp_forward(_dev(p), _dev(x)).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), L.mlp_forward(p, x).view(np.uint32))


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, -0.0, 3.4e38, -3.4e38, 1e-41, -1e-39])
def test_forward_extreme_inputs(gcpkg, value):
    """The maximum with 0 taken after the rounding, of two units at a time: not a number gives 0,
    infinities and subnormal numbers pass through the rounding as they do one by one."""
    n = 1300
    p = _uniform(5, 7, L.N_PARAMS, -0.3, 0.3)
    x = _uniform(6, 9, n * L.N_IN, -2.0, 24.0).reshape(n, L.N_IN)
    x[np.arange(n), np.arange(n) % L.N_IN] = value
    x[::7] = value
    got = gcpkg.mlp_forward(_dev(p), _dev(x)).cpu().numpy()
    want = L.mlp_forward(p, x)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.array_equal(got[ok].view(np.uint32), want[ok].view(np.uint32))


# 128 samples a tile, two blocks an SM: 38,912 before a block takes a second tile
@pytest.mark.parametrize("n", [2, 31, 33, 127, 128, 129, 38911, 38913, 80000])
def test_gradient_sizes(gcpkg, n):
    p = _uniform(n, 7, L.N_PARAMS, -0.3, 0.3)
    x = _uniform(n + 1, 9, n * L.N_IN, 0.0, 16.0).reshape(n, L.N_IN)
    t = np.linspace(-1.0, 1.0, n).astype(np.float32)
    grad = torch.zeros(L.N_PARAMS, dtype=torch.float32, device="cuda")
    sse = torch.zeros(1, dtype=torch.float32, device="cuda")
    gcpkg.mlp_grad(_dev(p), _dev(x), _dev(t), 1.0 / n, grad, sse)
    want, want_sse = L.mlp_grad(p, x, t, 1.0 / n, rounding=True)
    got = grad.cpu().numpy().astype(np.float64)
    # the bound of test_gpu_learned.test_grad_matches_oracle: fp32 sums of n terms in another order
    assert np.all(np.abs(got - want) <= 1e-4 * np.abs(want).max() + 1e-5 * np.abs(want)), np.abs(got - want).max()
    assert abs(float(sse.item()) - want_sse) <= 1e-4 * want_sse + 1e-6


def _gradient_64bit(p, x, t, scale):
    """Gradient and squared error in 64 bits on the device, over the forward's own activations: its
    products of bf16 values are exact in 32 bits, so a 32-bit sum in input order has its bits."""
    W1, b1, W2, b2, W3, b3 = (p[a:b] for a, b in ((0, 192), (192, 224), (224, 1248), (1248, 1280), (1280, 1312), (1312, 1313)))
    half = lambda z: z.to(torch.bfloat16).float()
    W1, W2, W3 = half(W1).view(32, 6), half(W2).view(32, 32), half(W3)

    def chain(a, w):
        acc = torch.zeros(a.shape[0], w.shape[0], device=a.device)
        for k in range(a.shape[1]):
            acc = acc + a[:, k:k + 1] * w[:, k][None]
        return acc

    grad, sse = torch.zeros(L.N_PARAMS, dtype=torch.float64, device=p.device), 0.0
    for a0, tt in zip(half(x).split(1 << 20), t.split(1 << 20)):
        a1 = half(torch.relu(chain(a0, W1) + b1))
        a2 = half(torch.relu(chain(a1, W2) + b2))
        err = (chain(a2, W3[None])[:, 0] + b3) - tt
        dy = (2 * scale * err).double()
        d2 = dy[:, None] * W3.double()[None] * (a2 > 0)
        d1 = (d2 @ W2.double()) * (a1 > 0)
        grad += torch.cat([(d1.T @ a0.double()).reshape(-1), d1.sum(0), (d2.T @ a1.double()).reshape(-1), d2.sum(0),
                           dy @ a2.double(), dy.sum()[None]])
        sse += float((err.double() ** 2).sum())
    return grad, sse


# a warp's running sums are n / 1,216 terms long: 216, 3,449 and 13,798
@pytest.mark.parametrize("n, shift", [(262145, 0.0), (4194301, 0.0), (4194301, 50.0), (16777213, 0.0)])
def test_gradient_sums_of_many_samples(gcpkg, n, shift):
    """Each part of the gradient and the squared error against 64 bits.  The sums end in one atomic a
    block: 304 additions of 32 bits, each off by at most 2^-24 of the sum so far, which is half the
    end's on average: 304 / 2 * 2^-24 = 9e-6 of it at worst.  A chain of k terms in a warp is off by
    about sqrt(k / 3) * 2^-25 of its own sum, and 1,216 of them, independent, by 1/35 of that of the
    whole: 6e-8 for the longest here.  Measured: 1 to 5e-7, and 2 to 6e-7 with short chains and one
    sum a parameter."""
    g = torch.Generator(device="cuda").manual_seed(n)
    p = torch.randn(L.N_PARAMS, generator=g, device="cuda") * 0.25
    x = torch.rand(n, L.N_IN, generator=g, device="cuda") * 12
    t = torch.randn(n, generator=g, device="cuda") * 3 + shift
    want, want_sse = _gradient_64bit(p, x, t, 1.0 / n)
    grad, sse = torch.zeros(L.N_PARAMS, device="cuda"), torch.zeros(1, device="cuda")
    gcpkg.mlp_grad(p, x, t, 1.0 / n, grad, sse)
    for a, b in ((0, 192), (192, 224), (224, 1248), (1248, 1280), (1280, 1312), (1312, 1313)):
        assert float((grad.double() - want)[a:b].norm()) <= 9e-6 * float(want[a:b].norm()), (a, b)
    assert abs(float(sse) - want_sse) <= 9e-6 * want_sse


def _rows_of(degree, seed):
    """Vertices of exactly `degree` neighbours (stars), among a sparse random graph, ids shuffled."""
    parts, n = [], 0
    for _ in range(3):
        parts.append((np.full(degree, n), n + 1 + np.arange(degree)))
        n += degree + 1
    g = gg.gnm(300, 700, seed)
    parts.append((np.repeat(np.arange(g.n), g.degrees) + n, g.colidx.astype(np.int64) + n))
    n += g.n
    perm = gg.permutation(n, seed)
    u, v = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    return gg.from_edges(n, perm[u], perm[v])


# rows read by their own lane (up to 16), 4 lanes (up to 57), 16 lanes (up to 121) or the warp, at every
# alignment of both arrays
@pytest.mark.parametrize("degree", [1, 8, 16, 17, 25, 26, 57, 58, 120, 121, 122, 255, 257, 1000])
def test_feature_rows(gcpkg, degree):
    g = _rows_of(degree, 40 + degree)
    want = L.features(g.rowptr, g.colidx)
    for shift in range(8):
        rp = torch.full((g.n + 16,), -5, dtype=torch.int32, device="cuda")[shift % 4:][:g.n + 1]
        ci = torch.full((g.nnz + 16,), 1 << 30, dtype=torch.int32, device="cuda")[shift:][:g.nnz]
        rp.copy_(torch.from_numpy(g.rowptr))
        ci.copy_(torch.from_numpy(g.colidx))
        out = torch.empty(g.n * 6 + 1, dtype=torch.float32, device="cuda")[shift % 2:][:g.n * 6].view(g.n, 6)
        got = gcpkg.features(rp, ci, out=out).cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), (degree, shift)


# vertices a warp takes: 8 up to 58,368 vertices, 16 up to 116,736, then 32; 32 below 6 entries a row
@pytest.mark.parametrize("n", [1, 7, 9, 31, 33, 1000, 58367, 58368, 58369, 116736, 116737, 120001])
def test_feature_vertices(gcpkg, n):
    for edges in (2 * n, 3 * n, 5 * n):
        g = gg.gnm(n, min(edges, n * (n - 1) // 2), n)
        want = L.features(g.rowptr, g.colidx)
        got = gcpkg.features(_dev(g.rowptr), _dev(g.colidx)).cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), g.name


def test_feature_rows_of_every_kind_together(gcpkg):
    """Long, middle and short rows in one graph, in warps of 8, 16 and 32 vertices."""
    for scale, ef in ((11, 16), (16, 8), (17, 8)):
        g = gg.rmat(scale, ef, gg.RMAT_B, scale)
        want = L.features(g.rowptr, g.colidx)
        got = gcpkg.features(_dev(g.rowptr), _dev(g.colidx)).cpu().numpy()
        assert np.array_equal(got.view(np.uint32), want.view(np.uint32)), g.name
