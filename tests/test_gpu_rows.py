"""The row passes where their layout changes: atom counts around the slices of
eight and the blocks of 32 and 16 atoms (interleaved rows, four and eight lanes
an atom), rows at their capacity; cell grids around the sizes where the scan
takes none, one or two kernels; and the gradient written whole with its factor
read on the device, against the forces."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import check_bias, check_cv, check_forces, kbdt, setup_hills

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06873_gb300 import build
    build.build()
    d = torch.device("cuda:0")
    torch.cuda.set_stream(torch.cuda.Stream(d))
    return d


def _params(dev, n, box, mp, **kw):
    from paper_2510_06873_gb300 import metad
    return metad.params_for(n, box, n_cv=mp.n_cv, sigma=mp.sigma, stream=torch.cuda.current_stream(dev).cuda_stream,
                            hill_capacity=256, **kw)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 1031, 1047])
def test_step_at_slice_and_block_edges(dev, n, fp64):
    """The common tolerances against the oracle, with rows just long enough
    for the longest one."""
    from paper_2510_06873_gb300 import metad
    system = synth.wurtzite_system(n, cfg=93)
    mp = synth.MethodParams(n_cv=2)
    frame = synth.perturbed_frame(system, 2)
    p = oracle.params_from(mp, system.box)
    pairs = oracle.pairs_cells(frame, system.box, 3.5)
    longest = int(np.bincount(pairs.ravel(), minlength=n).max())
    c, _ = setup_hills(system, mp, 50, cfg=93)
    w = oracle.deposit_sequence(c, mp.sigma, mp.w0, kbdt(mp))
    ref = oracle.step(frame, p, c, w, mp.sigma)
    ctx = metad.Metad(_params(dev, n, system.box, mp, fp64=fp64, max_neighbors=longest))
    ctx.load_hills(c, w)
    F = torch.full((n + 1, 3), 7.0, dtype=torch.float32, device=dev)
    ctx.step(torch.from_numpy(frame).to(dev), F)
    s, V, dV = ctx.read_results()
    assert bool((F[n] == 7.0).all())
    check_cv(s, ref["s"])
    check_bias(V, dV, ref["V"], ref["dV"], mp)
    check_forces(F[:n].cpu().numpy(), ref["F"])
    ctx.close()


@pytest.mark.parametrize("kind,n_cv,fp64", [("coordination", 1, False), ("coordination", 1, True),
                                            ("coordination", 2, False), ("coordination", 2, True),
                                            ("torsion", 2, False)])
def test_gradient_is_the_scaled_force(dev, kind, n_cv, fp64):
    """bias_gradient with factor g equals bias_forces scaled by -g bit for bit,
    and writes 0 in the species column."""
    from paper_2510_06873_gb300 import metad
    system = synth.wurtzite_system(1001, cfg=94)
    mp = synth.MethodParams(n_cv=n_cv, sigma=(0.05, 0.02)[:n_cv])
    ctx = metad.Metad(_params(dev, system.n, system.box, mp, fp64=fp64, cv_kind=kind))
    if kind == "torsion":
        ctx.set_cv_atoms([0, 1, 2, 3, 1, 2, 3, 4])
    frame = synth.perturbed_frame(system, 0)
    pos = torch.from_numpy(frame).to(dev)
    ctx.build_neighbors(pos)
    s = ctx.cv_forward()
    ctx.load_hills([np.asarray(s) + 0.01], [1.0])
    ctx.bias_eval()
    F = torch.zeros((system.n, 3), dtype=torch.float32, device=dev)
    ctx.bias_forces(F, scale=-0.7)
    grad = torch.full((system.n, 4), 9.0, dtype=torch.float32, device=dev)
    g = torch.tensor(0.7, dtype=torch.float64, device=dev)
    metad.metad_bias_gradient(ctx.ctx, grad, g)
    V = torch.zeros((), dtype=torch.float64, device=dev)
    metad.metad_bias_value(ctx.ctx, V)
    _, V_host, _ = ctx.read_results()
    assert float(V) == V_host
    assert float(F.abs().max()) > 0.0
    assert torch.equal(grad[:, :3], F) and bool((grad[:, 3] == 0.0).all())
    ctx.close()


@pytest.mark.parametrize("cells", [(15, 16, 16), (16, 16, 16), (17, 16, 16), (48, 64, 64), (49, 64, 64)])
def test_cell_scan_edges(dev, cells):
    """Few atoms in pairs within rc, spread over grids of 4,096 cells and one
    layer fewer and more, and of 48 and 49 tiles of 4,096: exact pairs after a
    first build, and after a rebuild on moved positions."""
    from paper_2510_06873_gb300 import metad
    g = np.random.default_rng(sum(cells))
    box = np.array(cells) * (4.5 * 1.0002)
    mp = synth.MethodParams(n_cv=1, sigma=(0.05,))
    ctx = metad.Metad(_params(dev, 600, box, mp))
    for _ in range(2):
        a = g.uniform(0.0, 1.0, (300, 3)) * box
        xyz = np.concatenate([a, a + g.normal(0.0, 1.6, (300, 3))])
        pos = np.zeros((600, 4), np.float32)
        pos[:, :3] = synth.wrap_to_box(xyz, box)
        pos[::2, 3] = 1.0
        ctx.build_neighbors(torch.from_numpy(pos).to(dev))
        ref = oracle.pairs_brute(pos, box, 3.5)
        assert len(ref) > 100 and np.array_equal(ctx.export_neighbors(), ref)
    assert ctx.rebuild_count == 2
    ctx.close()


@pytest.mark.parametrize("n", [1023, 1025])
def test_one_cv_rows_on_demand(dev, n):
    """With one CV in FP32 the CV pass writes no rows: the export and the
    statistics make them, the CV pass before and after gives the same bits, and
    a row longer than its capacity is still refused."""
    from paper_2510_06873_gb300 import metad
    system = synth.wurtzite_system(n, cfg=92)
    mp = synth.MethodParams(n_cv=1, sigma=(0.05,))
    frame = synth.perturbed_frame(system, 1)
    pos = torch.from_numpy(frame).to(dev)
    pairs = oracle.pairs_cells(frame, system.box, 3.5)
    longest = int(np.bincount(pairs.ravel(), minlength=n).max())
    ctx = metad.Metad(_params(dev, n, system.box, mp, max_neighbors=longest))
    ctx.load_hills([[2.0]], [1.0])
    F = torch.zeros((n, 3), dtype=torch.float32, device=dev)
    ctx.step(pos, F)
    first = ctx.read_results()
    assert np.array_equal(ctx.export_neighbors(), pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))])
    assert ctx.neighbor_stats() == (2 * len(pairs), longest)
    again = ctx.cv_forward()
    check_cv(first[0], oracle.cv(frame, oracle.params_from(mp, system.box))[0])
    assert np.array_equal(first[0], again)
    ctx.close()
    short = metad.Metad(_params(dev, n, system.box, mp, max_neighbors=longest - 4 - longest % 4))
    with pytest.raises(metad.MetadError):
        short.step(pos, F)
        short.read_results()
    short.close()


def test_octant_edges_sort_alike_in_a_batch(dev):
    """Atoms within an ulp or two of their cell's middle: the single and the
    batched kernels put them into the same octants, so the rows have one order
    and a batched step gives the single step's bits."""
    from paper_2510_06873_gb300 import metad
    g = np.random.default_rng(8)
    edge, planes, side = 4.567, 9, 16
    box = np.array([planes * edge, 2.55 * side, 2.55 * side])
    k, a, b = np.meshgrid(np.arange(planes), np.arange(side), np.arange(side), indexing="ij")
    pos = np.zeros((k.size, 4), np.float32)
    mid = ((k.ravel() + 0.5) * edge).astype(np.float32)
    for ulps in (1, 2):
        mid = np.where(g.random(k.size) < 0.4, np.nextafter(mid, np.float32(g.choice([0.0, 99.0]))), mid)
    pos[:, 0] = mid
    pos[:, 1] = (a.ravel() + 0.5) * 2.55 + g.uniform(-0.3, 0.3, k.size)
    pos[:, 2] = (b.ravel() + 0.5) * 2.55 + g.uniform(-0.3, 0.3, k.size)
    pos[:, 3] = g.integers(0, 2, k.size)
    pos = torch.from_numpy(pos[g.permutation(k.size)]).to(dev)
    mp = synth.MethodParams(n_cv=2)
    s_ref, _, _ = oracle.cv(pos.cpu().numpy(), oracle.params_from(mp, box))
    ctxs = [metad.Metad(_params(dev, k.size, box, mp)) for _ in range(2)]
    F = [torch.zeros((k.size, 3), dtype=torch.float32, device=dev) for _ in range(2)]
    for ctx in ctxs:
        ctx.load_hills([s_ref + 0.01], [1.0])
    ctxs[0].step(pos, F[0])
    s0 = ctxs[0].read_results()
    batch = metad.Batch(ctxs[1:])
    batch.step([pos], F[1:])
    s1 = ctxs[1].read_results()
    assert np.array_equal(s0[0], s1[0]) and s0[1] == s1[1] and np.array_equal(s0[2], s1[2])
    assert torch.equal(F[0], F[1]) and float(F[0].abs().max()) > 0.0
    batch.close()
    for ctx in ctxs:
        ctx.close()


@pytest.mark.parametrize("n_cv", [1, 2])
def test_every_pair_enters_a_compensated_virial_sum(dev, n_cv):
    """Box gradient of rows of some 450 neighbours against FP64 sums, with
    factors that are exact in float32 (r0 a power of two, no stretch) and no
    force from the second CV, so that what is left is each pair's own rounding,
    unbiased, and the sums'.  The same arithmetic in numpy leaves 0.014 units of
    2^-24 (rms, relative, over boxes and axes) where the sums add nothing, and
    0.043 with plain float32 sums of a lane's share of a row."""
    from paper_2510_06873_gb300 import metad
    n, L, r0, rc = 1100, np.array([7.25, 7.5, 8.0]), 2.0, 3.5
    p = metad.params_for(n, L, n_cv=n_cv, sigma=(0.5, 0.02)[:n_cv], virial=True, max_neighbors=560, r0=r0, rc=rc,
                         stream=torch.cuda.current_stream(dev).cuda_stream, hill_capacity=4)
    p.stretch, p.cn_pairs = 0, 0
    ctx = metad.Metad(p)
    F = torch.zeros((n, 3), dtype=torch.float32, device=dev)
    rel = []
    for seed in range(24):
        r = np.random.default_rng(seed)
        g = (np.stack(np.meshgrid(*[np.arange(11)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) / 11
        x = (((g[r.permutation(1331)[:n]] + r.uniform(-0.3, 0.3, (n, 3)) / 11) % 1.0) * L).astype(np.float32)
        x = np.where(x >= L, np.float32(0.0), x)
        ctx.build_neighbors(torch.from_numpy(np.concatenate([x, np.zeros((n, 1), np.float32)], 1)).to(dev))
        s = np.asarray(ctx.cv_forward())
        c = s.copy()
        c[0] += 0.3
        ctx.load_hills([c], [1.0])
        _, dV = ctx.bias_eval()
        assert n_cv == 1 or dV[1] == 0.0
        ctx.bias_forces(F)
        d = x[None].astype(np.float64) - x[:, None].astype(np.float64)
        d -= L * np.rint(d / L)
        r2 = (d * d).sum(2)
        np.fill_diagonal(r2, rc * rc)
        d, rr = d[r2 < rc * rc], np.sqrt(r2[r2 < rc * rc])
        assert rr.size > 440 * n
        q = rr / r0
        dw = -6.0 * q**5 / (1.0 + q**6) ** 2 / r0
        ref = 0.5 * float(np.float32(dV[0] * 2.0 / n)) * ((dw / rr)[:, None] * d * d).sum(0) / L
        rel.append(ctx.box_gradient() / ref - 1.0)
    ctx.close()
    assert np.sqrt(np.mean(np.square(rel))) <= 0.025 * 2.0**-24


def test_gradient_factors_that_are_not_plain_memory(dev):
    """A factor that autograd negates lazily (through a conjugate) and one
    without memory (a zero tensor) give what their values say."""
    from paper_2510_06873_gb300 import autograd
    system = synth.wurtzite_system(1001, cfg=95)
    mp = synth.MethodParams(n_cv=2)
    ctx = autograd.BiasContext(_params(dev, system.n, system.box, mp))
    pos = torch.from_numpy(synth.perturbed_frame(system, 0)).to(dev).requires_grad_(True)
    ctx.build_neighbors(pos.detach())
    ctx.load_hills([np.asarray(ctx.cv_forward()) + 0.01], [1.0])
    grads, negated = [], []
    for wrap in (lambda V: V, lambda V: torch.complex(torch.zeros_like(V), V).conj().abs()):
        V = autograd.bias(pos, ctx)
        V.register_hook(lambda g: negated.append(g.is_neg()))
        grads += torch.autograd.grad(wrap(V), pos)  # V > 0: |V| has the gradient of V
    assert negated == [False, True]
    assert bool(grads[0].any()) and torch.equal(grads[0], grads[1])
    V = autograd.bias(pos, ctx)
    (zero,) = torch.autograd.grad(V, pos, torch._efficientzerotensor((), dtype=torch.float64, device=dev))
    assert not bool(zero.any())
    ctx.close()


def test_autograd_on_another_stream_than_the_context(dev):
    """Positions still being written on torch's current stream when the
    forward pass is called, and a context's stream that is behind when the
    gradient is read: both are waited for."""
    from paper_2510_06873_gb300 import autograd, metad
    system = synth.wurtzite_system(1001, cfg=96)
    mp = synth.MethodParams(n_cv=2)
    ctx = autograd.BiasContext(metad.params_for(system.n, system.box, n_cv=2, sigma=mp.sigma, hill_capacity=16))
    own = torch.cuda.ExternalStream(ctx.stream, device=dev)
    base = torch.from_numpy(synth.perturbed_frame(system, 0)).to(dev)
    torch.cuda.synchronize(dev)
    ctx.build_neighbors(base)
    ctx.load_hills([np.asarray(ctx.cv_forward()) + 0.01], [1.0])
    ref = base.clone().requires_grad_(True)
    torch.cuda.synchronize(dev)
    V_ref = autograd.bias(ref, ctx)
    V_ref.backward()
    torch.cuda.synchronize(dev)
    for _ in range(2):
        late = torch.zeros_like(base)
        torch.cuda.synchronize(dev)
        torch.cuda._sleep(20_000_000)  # some 10 ms
        late.copy_(base)
        late.requires_grad_(True)
        V = autograd.bias(late, ctx)
        with torch.cuda.stream(own):
            torch.cuda._sleep(20_000_000)
        (g,) = torch.autograd.grad(V, late)
        assert float(V.detach()) == float(V_ref.detach()) and torch.equal(g, ref.grad)
    ctx.close()


@pytest.mark.parametrize("n_cv", [1, 2])
@pytest.mark.parametrize("skin", [0.0, 1.0])
def test_fp64_geometry_from_compacted_rows(dev, skin, n_cv):
    """The FP64 filter forms its displacements from the row's compacted tags:
    long rows, the longest just fitting, of few and many candidates."""
    from paper_2510_06873_gb300 import metad
    n, L, rc = 1100, np.array([7.25, 7.5, 8.0]), 2.0
    r = np.random.default_rng(7)
    g = (np.stack(np.meshgrid(*[np.arange(11)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) / 11
    x = (((g[r.permutation(1331)[:n]] + r.uniform(-0.3, 0.3, (n, 3)) / 11) % 1.0) * L).astype(np.float32)
    frame = np.concatenate([np.where(x >= L, np.float32(0.0), x), r.integers(0, 2, (n, 1)).astype(np.float32)], 1)
    mp = synth.MethodParams(n_cv=n_cv, sigma=(0.05, 0.02)[:n_cv], rc=rc, r0=1.5)
    p = oracle.params_from(mp, L)
    pairs = oracle.pairs_cells(frame, L, rc)
    s0, _, _ = oracle.cv(frame, p)
    c = (np.asarray(s0)[:n_cv] + 0.01)[None]
    w = oracle.deposit_sequence(c, mp.sigma, mp.w0, kbdt(mp))
    ref = oracle.step(frame, p, c, w, mp.sigma)
    ctx = metad.Metad(_params(dev, n, L, mp, fp64=True, max_neighbors=int(np.bincount(pairs.ravel()).max()), rc=rc, r0=1.5,
                            skin=skin))
    ctx.load_hills(c, w)
    F = torch.zeros((n, 3), dtype=torch.float32, device=dev)
    pos = torch.from_numpy(frame).to(dev)
    ctx.step(pos, F)
    assert np.array_equal(ctx.export_neighbors(), pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))])
    s, V, dV = ctx.read_results()
    check_cv(s, ref["s"])
    check_bias(V, dV, ref["V"], ref["dV"], mp)
    check_forces(F.cpu().numpy(), ref["F"])
    ctx.close()


@pytest.mark.parametrize("n", [69_999, 70_000])
def test_fp64_pair_pass_where_its_chunks_change(dev, n):
    """Eight atoms a warp below 70,000 atoms, 32 from there on."""
    from paper_2510_06873_gb300 import metad
    system = synth.wurtzite_system(n, cfg=93)
    mp = synth.MethodParams(n_cv=2)
    frame = synth.perturbed_frame(system, 1)
    c, _ = setup_hills(system, mp, 20, cfg=93)
    w = oracle.deposit_sequence(c, mp.sigma, mp.w0, kbdt(mp))
    ref = oracle.step(frame, oracle.params_from(mp, system.box), c, w, mp.sigma)
    ctx = metad.Metad(_params(dev, n, system.box, mp, fp64=True))
    ctx.load_hills(c, w)
    F = torch.zeros((n, 3), dtype=torch.float32, device=dev)
    ctx.step(torch.from_numpy(frame).to(dev), F)
    s, V, dV = ctx.read_results()
    check_cv(s, ref["s"])
    check_bias(V, dV, ref["V"], ref["dV"], mp)
    check_forces(F.cpu().numpy(), ref["F"])
    ctx.close()


def test_one_cv_forces_do_not_depend_on_the_virial(dev):
    """The same bits with the virial asked for and without, and in a batch."""
    from paper_2510_06873_gb300 import metad
    system = synth.wurtzite_system(5003, cfg=97)
    mp = synth.MethodParams(n_cv=1, sigma=(0.05,))
    pos = torch.from_numpy(synth.perturbed_frame(system, 0)).to(dev)
    out = []
    for virial in (False, True):
        ctx = metad.Metad(_params(dev, system.n, system.box, mp, virial=virial))
        ctx.build_neighbors(pos)
        ctx.load_hills([np.asarray(ctx.cv_forward()) + 0.01], [1.0])
        batch = metad.Batch([ctx])
        for step in (lambda F: ctx.step(pos, F), lambda F: batch.step([pos], [F])):
            F = torch.zeros((system.n, 3), dtype=torch.float32, device=dev)
            step(F)
            s, V, _ = ctx.read_results()
            out.append((F, s[0], V))
        batch.close()
        ctx.close()
    for F, s, V in out[1:]:
        assert torch.equal(F, out[0][0]) and (s, V) == out[0][1:]
