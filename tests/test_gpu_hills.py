"""Hill sums at the sizes where their kernels change shape, against plain
numpy in FP64: the integer exponential over its whole argument range, the
nearest image of far hill centres, block and slice edges of the hill kernel,
the per-axis contraction (free-energy grids, fold) and the chunked
reweighting sums."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53  # one rounding, relative


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06873_gb300 import build
    build.build()
    d = torch.device("cuda:0")
    torch.cuda.set_stream(torch.cuda.Stream(d))
    return d


def _ctx(dev, n_cv, sigma, **kw):
    from paper_2510_06873_gb300 import metad
    return metad.Metad(metad.params_for(8, [23.0, 23.0, 23.0], n_cv=n_cv, sigma=sigma,
                                        stream=torch.cuda.current_stream(dev).cuda_stream, **kw))


def test_one_hill_over_the_whole_argument_range(dev):
    """V = exp(-e) of a single hill: the exponent takes six roundings
    (sigma^2, 1/2 over it, log2 e, its product, two squares), the exponential
    and the reference one each."""
    ctx = _ctx(dev, 1, (1.0,))
    ctx.load_hills([[0.0]], [1.0])
    s = np.concatenate([np.linspace(0.0, 2.0, 97), np.geomspace(1e-160, 37.6, 200), [37.2, 37.3, 38.5, 38.7, 40.0, 1e3]])
    for x in s:
        V, _ = ctx.bias_eval([x])
        e = 0.5 * x * x
        ref = math.exp(-e)
        # below the normal range the reference itself is a multiple of 2^-1074
        assert abs(V - ref) <= (6.0 * e + 3.0) * U * ref + 2.0 ** -1074, (x, V, ref)
    ctx.load_hills([[math.inf]], [1.0])
    assert ctx.bias_eval([0.0])[0] == 0.0


@pytest.mark.parametrize("n_cv", [1, 2])
@pytest.mark.parametrize("K", [1, 31, 255, 256, 257, 1023, 1025, 2500, 10000])
def test_hill_sum_block_edges(dev, n_cv, K):
    r = np.random.default_rng(K + n_cv)
    sig = np.array([0.05, 0.02])[:n_cv]
    ctr = np.array([2.0, 0.3])[:n_cv]
    c, w = ctr + sig * r.uniform(-6, 6, (K, n_cv)), r.uniform(0.1, 1.0, K)
    ctx = _ctx(dev, n_cv, sig)
    ctx.load_hills(c, w)
    V, g = ctx.bias_eval(ctr)
    d = ctr - c
    t = w * np.exp(-(d * d / (2 * sig**2)).sum(1))
    ref_g = -(t[:, None] * d / sig**2).sum(0)
    # each term within (6 e + 8) roundings with e <= 36, sums of K terms pairwise-like (<= 30 levels)
    tol = (6 * 36 + 8 + 30) * U
    assert abs(V - t.sum()) <= tol * t.sum()
    assert np.all(np.abs(g - ref_g) <= tol * (t[:, None] * np.abs(d) / sig**2).sum(0))


def test_far_periodic_centres_wrap_to_the_nearest_image(dev):
    from paper_2510_06873_gb300 import metad
    p = metad.params_for(22, [24.0] * 3, n_cv=2, sigma=(0.35, 0.6), cv_kind="torsion", biasfactor=math.inf,
                         stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = metad.Metad(p)
    ctx.set_cv_atoms([2, 3, 4, 5, 3, 4, 5, 6])
    r = np.random.default_rng(3)
    c, w = r.uniform(-16.0, 16.0, (3000, 2)), r.uniform(0.1, 1.0, 3000)
    ctx.load_hills(c, w)
    sig = np.array([0.35, 0.6])
    for s in r.uniform(-math.pi, math.pi, (20, 2)):
        V, g = ctx.bias_eval(s)
        d = s - c
        d -= 2 * math.pi * np.rint(d / (2 * math.pi))
        t = w * np.exp(-(d * d / (2 * sig**2)).sum(1))
        # an image shift leaves an absolute rounding of 16 U in d: 2 d 16 U / (2 sigma^2) in the exponent
        tol = (6 * 60 + 40 + 2 * math.pi * 16 / 0.35**2) * U
        assert abs(V - t.sum()) <= tol * t.sum()
        assert np.all(np.abs(g + (t[:, None] * d / sig**2).sum(0)) <= 4 * tol * (t[:, None] * np.abs(d) / sig**2).sum(0))


@pytest.mark.parametrize("n", [(7, 40), (8, 8), (16, 16), (17, 33), (101, 9), (300, 8)])
@pytest.mark.parametrize("K", [0, 1, 33, 65, 700])
def test_free_energy_grid_tile_edges(dev, n, K):
    r = np.random.default_rng(n[0] + K)
    sig, ctr = np.array([0.05, 0.02]), np.array([2.0, 0.3])
    c, w = ctr + sig * r.uniform(-6, 6, (K, 2)), r.uniform(0.1, 1.0, K)
    ctx = _ctx(dev, 2, sig)
    ctx.load_hills(c, w)
    lo, hi = ctr - 8 * sig, ctr + 7 * sig
    F = ctx.fes_grid(lo, hi, n)
    ax = [lo[d] + (np.arange(n[d]) + 0.5) * ((hi[d] - lo[d]) / n[d]) for d in range(2)]
    e = [(ax[d][:, None] - c[None, :, d]) ** 2 / (2 * sig[d] ** 2) for d in range(2)]
    V = (w * np.exp(-(e[0][:, None, :] + e[1][None, :, :]))).sum(2)
    ref = -(10.0 / 9.0) * V
    # every term within (6 e + 10) roundings, e <= 2 * 14^2 / 2, weighed by the whole sum
    assert np.abs(F - (ref - ref.min())).max() <= 2 * (6 * 196 + 10 + 40) * U * max(np.abs(ref).max(), 1e-300)
    assert F.min() == 0.0


@pytest.mark.parametrize("n", [(2, 2), (16, 17), (60, 35)])
@pytest.mark.parametrize("K", [1, 33, 600])
def test_fold_tile_edges(dev, n, K):
    """Node values, first and mixed derivatives of the folded hills, folded
    twice (the second fold adds to the first)."""
    r = np.random.default_rng(n[0] + K)
    sig, ctr = np.array([0.05, 0.02]), np.array([2.0, 0.3])
    lo, hi = ctr - 8 * sig, ctr + 8 * sig
    ctx = _ctx(dev, 2, sig, grid=(n, lo, hi))
    ref = np.zeros((*n, 4))
    scale = np.zeros((*n, 4))
    ax = [lo[d] + np.arange(n[d]) * ((hi[d] - lo[d]) / (n[d] - 1)) for d in range(2)]
    for _ in range(2):
        c, w = ctr + sig * r.uniform(-6, 6, (K, 2)), r.uniform(0.1, 1.0, K)
        ctx.load_hills(c, w)
        ctx.fold_hills()
        dx = [ax[d][:, None] - c[None, :, d] for d in range(2)]
        e = [dx[d] ** 2 / (2 * sig[d] ** 2) for d in range(2)]
        g = w * np.exp(-(e[0][:, None, :] + e[1][None, :, :]))
        u, v = (dx[0] / sig[0] ** 2)[:, None, :], (dx[1] / sig[1] ** 2)[None, :, :]
        for q, t in enumerate((g, -g * u, -g * v, g * u * v)):
            ref[..., q] += t.sum(2)
            scale[..., q] += np.abs(t).sum(2)
    G = ctx.get_grid()
    # (6 e + 10) roundings a term, e <= 2 * 14^2 / 2, and the sums; the node
    # positions differ by a rounding of 2.0, 16 sigma: e changes by 14 * 2 U 2.4 / sigma
    tol = (6 * 196 + 60 + 14 * 2 * 2.4 / 0.05 * 2) * U
    assert np.all(np.abs(G - ref) <= tol * scale + 1e-300)


@pytest.mark.parametrize("T", [1, 31, 33, 64, 65, 5000])
@pytest.mark.parametrize("n", [(1,), (20,), (9, 7)])
def test_reweight_chunk_edges(dev, T, n):
    k = len(n)
    r = np.random.default_rng(T + k)
    S = np.column_stack([r.normal(2.0, 0.1, T), r.normal(0.3, 0.03, T)])[:, :k]
    V = r.uniform(0.0, 15.0, T)
    lo, hi = np.array([1.8, 0.22])[:k], np.array([2.2, 0.38])[:k]
    ctx = _ctx(dev, k, (0.05, 0.02)[:k])
    F = ctx.fes_reweight(S, V, lo, hi, n)
    h = (hi - lo) / np.array(n)
    idx = np.floor((S - lo) / h).astype(int)
    ok = np.all((S >= lo) & (S < hi) & (idx < np.array(n)), axis=1)
    beta = 1.0 / (0.0083144626 * 300.0)
    acc = np.zeros(n)
    np.add.at(acc, tuple(idx[ok].T), np.exp(beta * (V[ok] - V.max())))
    assert np.array_equal(np.isinf(F), acc == 0.0)
    if acc.any():
        with np.errstate(divide="ignore"):
            ref = -np.log(acc / acc.sum()) / beta
        ref -= ref.min()
        fin = acc > 0
        assert np.allclose(F[fin], ref[fin], rtol=1e-11, atol=1e-11)


def _fold_sums(ax, c, w, sig):
    """Node sums of V, dV/dx, dV/dy, d2V/dxdy and of the terms' magnitudes."""
    ref, scale = (np.zeros((ax[0].size, ax[1].size, 4)) for _ in range(2))
    for k in range(0, len(w), 500):
        dx = [ax[d][:, None] - c[None, k:k + 500, d] for d in range(2)]
        e = [dx[d] ** 2 / (2 * sig[d] ** 2) for d in range(2)]
        g = w[k:k + 500] * np.exp(-(e[0][:, None, :] + e[1][None, :, :]))
        u, v = (dx[0] / sig[0] ** 2)[:, None, :], (dx[1] / sig[1] ** 2)[None, :, :]
        for q, t in enumerate((g, -g * u, -g * v, g * u * v)):
            ref[..., q] += t.sum(2)
            scale[..., q] += np.abs(t).sum(2)
    return ref, scale


@pytest.mark.parametrize("n,K", [((60, 35), 5505), ((60, 35), 11009), ((2, 600_000), 3)])
def test_fold_over_several_tables_and_node_by_node(dev, n, K):
    """One hill more than fits one table of factors, and two; a grid too long
    for the contraction's workspace."""
    r = np.random.default_rng(K)
    sig, ctr = np.array([0.05, 0.02]), np.array([2.0, 0.3])
    lo, hi = ctr - 8 * sig, ctr + 8 * sig
    ctx = _ctx(dev, 2, sig, grid=(n, lo, hi), hill_capacity=K)
    c, w = ctr + sig * r.uniform(-6, 6, (K, 2)), r.uniform(0.1, 1.0, K)
    ctx.load_hills(c, w)
    ctx.fold_hills()
    ref, scale = _fold_sums([lo[d] + np.arange(n[d]) * ((hi[d] - lo[d]) / (n[d] - 1)) for d in range(2)], c, w, sig)
    tol = (6 * 196 + 60 + 14 * 2 * 2.4 / 0.05 * 2) * U  # as test_fold_tile_edges
    assert np.all(np.abs(ctx.get_grid() - ref) <= tol * scale + 1e-300)


def test_fold_allocates_nothing_and_its_capture_outlives_other_calls(dev):
    """The fold's workspace is the context's own from creation on: a fold in
    the middle of a run allocates nothing, and a captured one can be replayed
    after calls that need a larger workspace."""
    sig, ctr = np.array([0.05, 0.02]), np.array([2.0, 0.3])
    lo, hi = ctr - 8 * sig, ctr + 8 * sig
    r = np.random.default_rng(5)
    c, w = ctr + sig * r.uniform(-6, 6, (300, 2)), r.uniform(0.1, 1.0, 300)
    kw = dict(grid=((40, 30), lo, hi), hill_capacity=500)
    a, b = _ctx(dev, 2, sig, **kw), _ctx(dev, 2, sig, **kw)
    held = a.device_bytes
    a.load_hills(c, w)
    a.fold_hills()
    assert a.device_bytes == held
    once = a.get_grid()
    a.load_hills(c, w)
    a.fold_hills()  # adds to the first
    b.load_hills(c, w)
    b.fes_grid(lo, hi, (16, 16))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.current_stream(dev)):
        b.fold_hills()
    assert not b.get_grid().any()  # captured, not run
    b.fes_grid(lo, hi, (900, 900))
    graph.replay()
    assert np.array_equal(b.get_grid(), once)
    graph.replay()
    assert np.array_equal(b.get_grid(), a.get_grid())


@pytest.mark.parametrize("K", [2753, 5600])
def test_free_energy_grid_over_several_tables(dev, K):
    """1,500 x 8 points: a table of factors holds 2,752 hills."""
    n = (1500, 8)
    r = np.random.default_rng(K)
    sig, ctr = np.array([0.05, 0.02]), np.array([2.0, 0.3])
    c, w = ctr + sig * r.uniform(-6, 6, (K, 2)), r.uniform(0.1, 1.0, K)
    ctx = _ctx(dev, 2, sig)
    ctx.load_hills(c, w)
    lo, hi = ctr - 8 * sig, ctr + 7 * sig
    F = ctx.fes_grid(lo, hi, n)
    ax = [lo[d] + (np.arange(n[d]) + 0.5) * ((hi[d] - lo[d]) / n[d]) for d in range(2)]
    ref = -(10.0 / 9.0) * _fold_sums(ax, c, w, sig)[0][..., 0]
    # as test_free_energy_grid_tile_edges
    assert np.abs(F - (ref - ref.min())).max() <= 2 * (6 * 196 + 10 + 40) * U * np.abs(ref).max()
    assert F.min() == 0.0


@pytest.mark.parametrize("T,n", [(140_000, (9, 7)), (5000, (2000, 1500)), (700, (3000, 3000))])
def test_reweight_with_few_or_long_chunks(dev, T, n):
    """More samples than 2,048 chunks of 64 hold; grids whose rows leave two
    chunks and one."""
    r = np.random.default_rng(T)
    S, V = np.column_stack([r.normal(2.0, 0.1, T), r.normal(0.3, 0.03, T)]), r.uniform(0.0, 15.0, T)
    lo, hi = np.array([1.8, 0.22]), np.array([2.2, 0.38])
    F = _ctx(dev, 2, (0.05, 0.02)).fes_reweight(S, V, lo, hi, n)
    idx = np.floor((S - lo) / ((hi - lo) / np.array(n))).astype(int)
    ok = np.all((S >= lo) & (S < hi) & (idx < np.array(n)), axis=1)
    beta = 1.0 / (0.0083144626 * 300.0)
    acc = np.zeros(n)
    np.add.at(acc, tuple(idx[ok].T), np.exp(beta * (V[ok] - V.max())))
    fin = acc > 0
    assert np.array_equal(np.isfinite(F), fin)
    ref = -np.log(acc[fin] / acc.sum()) / beta
    assert np.allclose(F[fin], ref - ref.min(), rtol=1e-11, atol=1e-11)


def test_reweight_without_memory_is_refused(dev):
    """A workspace no device has: METAD_ERR_OOM before any host array is read
    (no other order of summation stands in), and the context goes on."""
    from paper_2510_06873_gb300 import metad
    ctx = _ctx(dev, 2, (0.05, 0.02))
    S, V, F = np.full((1, 2), 2.0), np.zeros(1), np.zeros(64)
    lo, hi, n = np.array([1.8, 1.8]), np.array([2.2, 2.2]), np.array([8, 8], dtype=np.int32)
    call = lambda T: metad.lib().metad_fes_reweight(ctx.ctx, S.ctypes.data, V.ctypes.data, T, lo.ctypes.data,  # noqa: E731
                                                    hi.ctypes.data, n.ctypes.data, F.ctypes.data)
    assert call(1 << 40) == metad.METAD_ERR_OOM
    assert call(1) == metad.METAD_OK
    assert F.min() == 0.0 and np.isinf(F).sum() == 63
