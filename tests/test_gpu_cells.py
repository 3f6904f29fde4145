"""The located search of d <= 2 (the automatic form's tables of candidate points)
against the oracle, at the sizes where a table or a launch can go wrong: one-point
and two-point grids, patches and inline lists filled and overflowing, ties, samples
outside the tables' box, grids with no usable table, ragged tiles, both sample
precisions, Algorithm II.  Counts and cells are compared bit for bit.
"""
import os
import subprocess
import tempfile

import numpy as np
import pytest

import oracle
import qt_workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def B(gpu_lib):
    from paper_1101_3228_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _run_program(name, *flags):
    from paper_1101_3228_gb300.build import CSRC, _nvcc
    with tempfile.TemporaryDirectory() as tmp:
        exe = os.path.join(tmp, name)
        subprocess.run([_nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                        "--expt-relaxed-constexpr", "-I", CSRC, os.path.join(HERE, "cuda", name + ".cu"), "-o", exe],
                       check=True)
        return subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split()


def test_near_normals_within_their_bound():
    """The certificate allows 1.375 2^-20 of the radius, and radii up to 8.6."""
    out = _run_program("near_normals")
    val = {out[i]: float(out[i + 1]) for i in range(1, len(out), 2)}
    assert 0.0 < val["max_error"] < 1.0 and val["max_radius"] < 8.6 and val["max_radius_error"] < 1.0, val


def test_sampler_operations_are_the_ieee_ones():
    """Uniform, logarithm, radius, sine and cosine for all 2^23 FP32 uniforms, bit for bit."""
    out = _run_program("sampler_exact")
    assert [int(v) for v in out[3::2]] == [0] * 5, out


def _chain(d, n, Ns, M, scale=1.0, shift=0.0, seed=5):
    rng = np.random.default_rng(seed)
    A = np.repeat((0.9 * np.eye(d) + 0.05 * np.tri(d, k=-1).T)[None], n, 0)
    T = np.repeat((scale * 0.3 * (np.eye(d) + 0.2 * np.tri(d, k=-1)))[None], n, 0)
    L = np.concatenate([np.zeros((1, d, d)), np.repeat((scale * (np.eye(d) - 0.4 * np.tri(d, k=-1)))[None], n, 0)])
    m = np.full((n + 1, d), shift)
    b = np.repeat((shift - A[0] @ np.full(d, shift))[None], n, 0)
    N = np.array([1] + list(Ns), dtype=np.int64)
    g = np.concatenate([m[:1]] + [shift + scale * rng.standard_normal((k, d)) * 1.2 for k in Ns])
    return W.Model("chain", d, n, N, A, b, T, m, L, np.arange(n + 1.0), 0.0, "put_exp1d", 1.0, None, M, 99,
                   W.PREC_F32, "kmeans"), g


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("prec", [W.PREC_F32, W.PREC_F64])
@pytest.mark.parametrize("Ns,M", [((2, 3, 1, 64), 257), ((100, 101), 1025), ((500, 37), 20011), ((1023, 1024), 3001),
                                  ((1024, 1025), 777)])
def test_located_counts_bit_exact(ctx, B, d, prec, Ns, M):
    model, g = _chain(d, len(Ns), Ns, M)
    ref = oracle.transitions(model, g, M, model.seed, prec)
    for ct in (B.COUNTS_I64, B.COUNTS_U32):
        counts, st, dump = ctx.transitions(model, _dev(g), M, model.seed, B.options(prec=prec, counts_type=ct),
                                           dump_count=50, dump_stride=7)
        got = B.split_counts(model.N, counts.cpu().numpy().astype(np.int64))
        for k in range(model.n):
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")
        assert st.form_used == B.FORM_F32_RECHECK and st.device_status == 0
    off = model.offsets()
    ok = dump["i"][-1].cpu().numpy() >= 0
    X, Y = (dump[v][-1].cpu().numpy()[ok] for v in "XY")
    np.testing.assert_array_equal(dump["i"][-1].cpu().numpy()[ok], oracle.nearest(g[off[-3]:off[-2]], X))
    np.testing.assert_array_equal(dump["j"][-1].cpu().numpy()[ok], oracle.nearest(g[off[-2]:off[-1]], Y))


@pytest.mark.parametrize("prec", [W.PREC_F32, W.PREC_F64])
@pytest.mark.parametrize("scale,shift", [(1e-3, 5.0), (1e3, 0.0), (1e-6, 100.0)])
def test_located_counts_over_scales(ctx, B, prec, scale, shift):
    """Grids far from the origin: the last one leaves no usable table for FP32 samples
    (their spacing there is coarser than the bins)."""
    for d in (1, 2):
        model, g = _chain(d, 2, (150, 90), 4001, scale, shift)
        ref = oracle.transitions(model, g, model.M, model.seed, prec)
        counts, _, _ = ctx.transitions(model, _dev(g), model.M, model.seed, B.options(prec=prec))
        got = B.split_counts(model.N, counts.cpu().numpy())
        for k in range(model.n):
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"d {d} layer {k}")


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("kind", ["ties", "cluster", "line", "same", "outside"])
def test_located_cells_of_given_samples(ctx, B, d, kind):
    rng = np.random.default_rng(3)
    gA = rng.standard_normal((300, d))
    gB = 1.2 * rng.standard_normal((317, d))
    X, Y = rng.standard_normal((4001, d)), rng.standard_normal((4001, d))
    if kind == "ties":
        gA = np.round(gA * 8) / 8                    # dyadic: exact ties and duplicates
        X = np.round(X * 16) / 16
        Y[:2000] = W.boundary_samples(gB, 2000, seed=4, jitter=1e-9)
    elif kind == "cluster":
        gA[10:] = 1e-4 * gA[10:]                     # hundreds of points in one bin
        X[::2] *= 1e-4
        gB[5:] = gB[5] + 1e-9 * rng.standard_normal((312, d))
    elif kind == "line":
        gA[:, -1] = 0.25                             # no extent along the last axis
        X[::3, -1] = 0.25
    elif kind == "same":
        gA[:] = gA[0]
    else:
        X *= 50.0
        Y[7] = 1e30
        X[5] = -1e18
    for ct in (B.COUNTS_I64, B.COUNTS_U32):
        counts, st, ii, jj = ctx.counts_from_samples(_dev(gA), _dev(gB), _dev(X), _dev(Y), B.options(counts_type=ct),
                                                     want_cells=True)
        np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(gA, X))
        np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(gB, Y))
        np.testing.assert_array_equal(counts.cpu().numpy(), oracle.counts_from_samples(gA, gB, X, Y))
    if kind == "ties":
        assert st.rechecks > 100


@pytest.mark.parametrize("prec", [W.PREC_F32, W.PREC_F64])
@pytest.mark.parametrize("M", [1, 33, 20011, 300007])
def test_located_paths_bit_exact(ctx, B, prec, M):
    """Algorithm II: few paths (one per thread), several per thread, the Euler chain."""
    n = 3 if M > 10**5 else 5
    for d in (1, 2):
        model, g = _chain(d, n, [60, 1, 200, 33, 90][:n], M)
        for euler in (None, (np.full((n, d), 0.5), np.full((n, d), 0.3))):
            ref = oracle.pathwise(model, g, M, model.seed, prec, euler=euler)
            ref = ref[0] if isinstance(ref, tuple) else ref
            counts, _, _ = ctx.transitions_pathwise(model, _dev(g), M, model.seed, B.options(prec=prec), euler=euler)
            got = B.split_counts(model.N, counts.cpu().numpy())
            for k in range(n):
                np.testing.assert_array_equal(got[k], ref[k], err_msg=f"d {d} layer {k}")


def test_located_fused_price_and_timeouts(ctx, B):
    """One layer at a time (the fused price), a wait that gives up in either kernel, and
    alternating calls on one context (direct launches, then a captured step)."""
    model, g = _chain(2, 3, (80, 120, 60), 5003)
    phi = np.maximum(1.0 - np.exp(g.sum(1)), 0.0)
    ref = oracle.price(model.N, oracle.transitions(model, g, model.M, model.seed, W.PREC_F32), phi)
    other, g2 = _chain(1, 2, (70, 50), 3001, seed=8)
    phi2 = np.maximum(1.0 - np.exp(g2[:, 0]), 0.0)
    ref2 = oracle.price(other.N, oracle.transitions(other, g2, other.M, other.seed, W.PREC_F32), phi2)
    for flags in (0, B.FLAG_FUSED_BACKWARD, B.FLAG_NO_GRAPH, 0, 0, 0):
        for mdl, gr, ph, want in ((model, g, phi, ref), (other, g2, phi2, ref2)):
            for _ in range(3 if flags == 0 else 1):
                price, st = ctx.price(mdl, gr, mdl.M, mdl.seed, ph, B.options(flags=flags))
                assert abs(price - want) <= 1e-12 * max(abs(want), 1e-300)
    for call in (ctx.transitions, ctx.transitions_pathwise):
        with pytest.raises(B.QtError) as e:
            call(model, _dev(g), model.M, model.seed, B.options(spin_budget=-1))
        assert e.value.status == B.QT_ETIMEOUT
        call(model, _dev(g), model.M, model.seed)


def test_located_full_pool(ctx, B):
    """More long candidate lists than the pool holds: nearly every point of 40 grids in one
    bin's width, so that every bin of them keeps all of these points."""
    n, N, M = 40, 1024, 501
    rng = np.random.default_rng(9)
    model, _ = _chain(2, n, [N] * n, M)
    g = 1e-7 * rng.standard_normal((int(model.N.sum()), 2))
    g[1::N] += 1.0
    ref = oracle.transitions(model, g, M, model.seed, W.PREC_F32)
    counts, st, _ = ctx.transitions(model, _dev(g), M, model.seed)
    got = B.split_counts(model.N, counts.cpu().numpy())
    for k in range(n):
        np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")
    assert st.device_status == 0


@pytest.mark.parametrize("d", [1, 2])
def test_located_fp64_pairs_at_the_draws_own_rounding(ctx, B, d):
    """Scale 1e-9 about 100: the FP64 draw moves in steps of 1.4e-14, 10^-5 of the scale, so
    that some samples tie between two points exactly; the FP32 stand-in must not decide them."""
    M = 2 * 10**6
    model, _ = _chain(d, 2, (2, 3), M, 1e-9, 100.0)
    g = np.full((6, d), 100.0)
    g[1, 0] -= 2.0**-30
    g[2, 0] += 2.0**-30
    g[3, 0] -= 2.0**-29
    g[5, 0] += 2.0**-29
    ref = oracle.transitions(model, g, M, model.seed, W.PREC_F64)
    counts, st, _ = ctx.transitions(model, _dev(g), M, model.seed, B.options(prec=B.PREC_F64))
    got = B.split_counts(model.N, counts.cpu().numpy())
    for k in range(model.n):
        np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("spread", [1.0, 1e-5])
def test_located_fp64_pairs_off_the_next_mean(ctx, B, d, spread):
    """Marginal means that do not follow from each other (m_{k+1} != A m_k + b): the constant
    of the map is large against the normals' part, and its rounding does not shrink with
    their radius.  The grid of the next layer lies where the samples go."""
    M, n, N = 200003, 2, 60
    rng = np.random.default_rng(11)
    model, _ = _chain(d, n, (N, N), M, spread)
    m = model.m + np.array([0.0, 1.0, -0.7])[:, None]
    model = W.Model("off", d, n, model.N, model.A, model.b, model.T, m, model.L, model.t, 0.0, "put_exp1d", 1.0,
                    None, M, 99, W.PREC_F64, "kmeans")
    g = np.concatenate([m[:1], (model.A[0] @ m[0] + model.b[0]) + spread * 0.4 * rng.standard_normal((N, d)),
                        (model.A[1] @ m[1] + model.b[1]) + spread * rng.standard_normal((N, d))])
    ref = oracle.transitions(model, g, M, model.seed, W.PREC_F64)
    counts, _, _ = ctx.transitions(model, _dev(g), M, model.seed, B.options(prec=B.PREC_F64))
    got = B.split_counts(model.N, counts.cpu().numpy())
    for k in range(n):
        np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")


@pytest.mark.parametrize("d,N", [(1, 100), (1, 1000), (1, 1024), (2, 100), (2, 1000)])
@pytest.mark.parametrize("scale,shift", [(1.0, 0.0), (1e-3, 1.0), (1e4, 3e5), (1e-18, 0.0)])
@pytest.mark.parametrize("kind", ["normal", "cluster"])
def test_located_cells_at_cell_boundaries(ctx, B, d, N, scale, shift, kind):
    """What the tables leave out: samples on, and within 1e-15 to 1e-4 of, the boundary
    between two cells, on grids fine against the tables' bins and on grids far from the origin."""
    rng = np.random.default_rng(N + d)
    gA, gB = rng.standard_normal((N, d)), rng.standard_normal((N, d))
    if kind == "cluster":
        gA[::2] *= 1e-3
        gB[::3] = gB[0] + 1e-5 * gB[::3]
    M = 6000
    X, Y = W.boundary_samples(gA, M, seed=1), W.boundary_samples(gB, M, seed=2)
    jit = 10.0 ** rng.uniform(-15, -4, (2, M, 1)) * rng.standard_normal((2, M, d))
    X[M // 4:] += jit[0, M // 4:]
    Y[M // 4:] += jit[1, M // 4:]
    gA, gB, X, Y = (shift + scale * v for v in (gA, gB, X, Y))
    counts, st, ii, jj = ctx.counts_from_samples(_dev(gA), _dev(gB), _dev(X), _dev(Y), B.options(), want_cells=True)
    np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(gA, X))
    np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(gB, Y))
    assert st.device_status == 0 and st.rechecks > 1000


@pytest.mark.parametrize("kind", ["flat", "narrow", "off"])
def test_located_search_certifies_odd_grids(ctx, B, kind):
    """Grids with one point along an axis, with axes of very different extent, and far from the
    centre of the search still have tables and certificates: few searches need FP64.  On
    the flat grid, 500 points evenly over 8 and samples at most 4 beside it, the certificate
    asks for 4 sqrt(2) e sqrt(D) <= 1.4e-5, e = 2^-24 of 10 (the box's size), where second
    and best differ by up to the squared spacing, 2.6e-4: at most 6% are in doubt."""
    rng = np.random.default_rng(6)
    M, N, d = 20000, 500, 2
    g, X = rng.standard_normal((2, N, d)), np.clip(rng.standard_normal((2, M, d)), -4, 4)
    if kind == "flat":
        g[:, :, 0], g[:, :, 1] = np.linspace(-4, 4, N), 0.0
    elif kind == "narrow":
        g[:, :, 1] *= 1e-3
        X[:, :, 1] *= 1e-3
    else:
        d = 1
        g, X = 4.6 + 0.1 * g[:, :, :1], 4.6 + 0.1 * X[:, :, :1]
    counts, st, ii, jj = ctx.counts_from_samples(_dev(g[0]), _dev(g[1]), _dev(X[0]), _dev(X[1]), B.options(),
                                                 want_cells=True)
    np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(g[0], X[0]))
    np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(g[1], X[1]))
    assert st.rechecks < 0.15 * 2 * M


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("kind", ["flat0", "flat1", "point", "plain"])
def test_located_cells_far_beyond_the_box(ctx, B, d, kind):
    """Samples beside the tables, near and very far (1e-3 to 1e18 of the grid's width), where
    distances tie in FP64; grids with all points equal along an axis, whose table has one bin
    without an end there, and grids of one distinct point and another next to it."""
    rng = np.random.default_rng(8)
    N, M = 300, 40000
    g = rng.standard_normal((2, N, d))
    if kind == "point":
        g[0] = g[0, 0]
        g[1] = g[1, 0]
        g[1, 7] += 1e-12
    elif d == 2 and kind != "plain":
        g[:, :, int(kind[-1])] = 0.3
    X = rng.standard_normal((2, M, d)) * 10.0 ** rng.uniform(-3, 18, (2, M, 1))
    X[:, ::3, 0] = rng.standard_normal((2, len(X[0, ::3])))           # far along one axis only
    if d == 2:
        X[:, 1::3, 1] = rng.standard_normal((2, len(X[0, 1::3])))
    for k in range(2):
        tie = W.boundary_samples(g[k], 2000, seed=k) if kind != "point" else X[k, :2000]
        X[k, 2:6000:3] = tie
    counts, st, ii, jj = ctx.counts_from_samples(_dev(g[0]), _dev(g[1]), _dev(X[0]), _dev(X[1]), B.options(),
                                                 want_cells=True)
    np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(g[0], X[0]))
    np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(g[1], X[1]))
    assert st.device_status == 0


@pytest.mark.parametrize("d", [1, 2])
def test_located_search_centres_far_grids(ctx, B, d):
    """Given samples at 100 with a spread of 1e-4: FP32 coordinates about zero have steps of
    7.6e-6, about the grid's own middle 1e-11, so that few searches need FP64."""
    rng = np.random.default_rng(12)
    M, N = 20000, 400
    g, X = 100.0 + 1e-4 * rng.standard_normal((2, N, d)), 100.0 + 1e-4 * rng.standard_normal((2, M, d))
    counts, st, ii, jj = ctx.counts_from_samples(_dev(g[0]), _dev(g[1]), _dev(X[0]), _dev(X[1]), B.options(),
                                                 want_cells=True)
    np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(g[0], X[0]))
    np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(g[1], X[1]))
    assert st.rechecks < 0.15 * 2 * M


@pytest.mark.parametrize("d,prec", [(1, W.PREC_F32), (1, W.PREC_F64), (2, W.PREC_F32), (2, W.PREC_F64), (3, W.PREC_F32)])
@pytest.mark.parametrize("later", [0.0, np.nan])
def test_paths_read_the_first_mean_only(ctx, B, d, prec, later):
    """Algorithm II reads the model's mean for the first layer only: zero or undefined later
    ones change nothing."""
    M, n = 20011, 3
    model, g = _chain(d, n, (60, 200, 33), M, 0.1, 4.6)
    m = model.m.copy()
    m[1:] = later
    ref = oracle.pathwise(model, g, M, model.seed, prec)
    ref = ref[0] if isinstance(ref, tuple) else ref
    other = W.Model("m", d, n, model.N, model.A, model.b, model.T, m, model.L, model.t, 0.0, "put_exp1d", 1.0, None, M, 99,
                    prec, "kmeans")
    counts, st, _ = ctx.transitions_pathwise(other, _dev(g), M, model.seed, B.options(prec=prec))
    got = B.split_counts(model.N, counts.cpu().numpy())
    for k in range(n):
        np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")
    assert st.device_status == 0


@pytest.mark.parametrize("ratio", [1e-6, 1e-3, 0.01, 0.1, 0.4, 3.0, 30.0, 1e4])
@pytest.mark.parametrize("N", [2, 3, 17, 1024])
def test_located_cells_of_long_grids(ctx, B, ratio, N):
    """Grids much longer than high and the reverse: the table's bins follow the extents (8 bins
    at least along either axis)."""
    rng = np.random.default_rng(N)
    g, X = rng.standard_normal((2, N, 2)), 1.5 * rng.standard_normal((2, 9001, 2))
    g[:, :, 1] *= ratio
    X[:, :, 1] *= ratio
    X[0, ::3], X[1, ::3] = W.boundary_samples(g[0], 3001, 1, 1e-9), W.boundary_samples(g[1], 3001, 2, 1e-9)
    counts, st, ii, jj = ctx.counts_from_samples(_dev(g[0]), _dev(g[1]), _dev(X[0]), _dev(X[1]), B.options(),
                                                 want_cells=True)
    np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(g[0], X[0]))
    np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(g[1], X[1]))
    assert st.device_status == 0


@pytest.mark.parametrize("d,n,N,Ms", [(2, 80, 500, (60, 5000, 9000)), (2, 300, 100, (50, 1500, 4000)), (1, 300, 500, (40, 900, 3000))])
@pytest.mark.parametrize("prec", [W.PREC_F32, W.PREC_F64])
def test_located_and_brute_force_over_the_number_of_pairs(ctx, B, d, n, N, Ms, prec):
    """Few pairs a date do not pay for the tables of many dates: either side of the line, and
    the fused price, which takes one date at a time, give the oracle's counts."""
    model, g = _chain(d, n, [N] * n, max(Ms))
    G = _dev(g)
    for M in Ms:
        ref = np.concatenate([c.reshape(-1) for c in oracle.transitions(model, g, M, model.seed, prec)])
        counts, st, _ = ctx.transitions(model, G, M, model.seed, B.options(prec=prec))
        np.testing.assert_array_equal(counts.cpu().numpy(), ref)
        assert st.form_used == B.FORM_F32_RECHECK and st.device_status == 0
    phi = np.maximum(1.0 - np.exp(g.sum(1)), 0.0)
    blocks = oracle.transitions(model, g, Ms[0], model.seed, prec)
    price, _ = ctx.price(model, g, Ms[0], model.seed, phi, B.options(prec=prec, flags=B.FLAG_FUSED_BACKWARD))
    want = oracle.price(model.N, blocks, phi)
    assert abs(price - want) <= 1e-12 * max(abs(want), 1e-300)
