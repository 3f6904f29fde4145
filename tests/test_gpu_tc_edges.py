"""The tensor-core form at the sizes where its tiles, items and windows end, against
the oracle: grids of one point, one chunk, one operand tile and one point either side
of a tile, more tiles than the ring holds, samples either side of an item of 128, and
samples that tie within a chunk (exact distances to the chunk alone) or across chunks
(window search).  Counts and cells are compared bit for bit.
"""
import numpy as np
import pytest

import oracle
import qt_workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


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


@pytest.mark.parametrize("d", [3, 4, 6, 8, 10])
@pytest.mark.parametrize("NA,NB,M", [(1, 16, 1), (17, 127, 127), (128, 129, 128), (1, 1, 129), (255, 2, 300),
                                     (1500, 1, 513), (900, 1700, 1000)])
def test_cells_at_tile_edges(ctx, B, d, NA, NB, M):
    rng = np.random.default_rng(NA + 7 * NB + d)
    gA, gB = rng.standard_normal((NA, d)), 0.7 * rng.standard_normal((NB, d)) + 0.2
    X, Y = rng.standard_normal((M, d)), rng.standard_normal((M, d))
    # last points of the last chunk, and exact ties: duplicated points near and far in the grid
    if NA > 16:
        gA[-1] = gA[3]
        gA[5] = gA[4]
        X[::5] = gA[rng.integers(0, NA, len(X[::5]))]
    if NB > 16:
        gB[NB // 2] = gB[NB // 2 - 1]
        Y[::4] = gB[rng.integers(0, NB, len(Y[::4]))] + 1e-9 * rng.standard_normal((len(Y[::4]), d))
    for ct in (B.COUNTS_I64, B.COUNTS_U32):
        counts, st, ii, jj = ctx.counts_from_samples(_dev(gA), _dev(gB), _dev(X), _dev(Y),
                                                     B.options(form=B.FORM_TC_RECHECK, counts_type=ct), want_cells=True)
        np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(gA, X))
        np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(gB, Y))
        np.testing.assert_array_equal(counts.cpu().numpy(), oracle.counts_from_samples(gA, gB, X, Y))
        assert st.form_used == B.FORM_TC_RECHECK and st.device_status == 0


@pytest.mark.parametrize("chunk", [1, 3, 0])
def test_uneven_layers_over_windows(ctx, B, chunk):
    """Layers of very different grid sizes, a one-point grid in the middle, windows that
    end inside a layer; given draws of either layout option are the same step."""
    d, Ns = 4, [1, 300, 20, 1, 700, 129]
    rng = np.random.default_rng(2)
    n = len(Ns) - 1
    L = np.concatenate([np.zeros((1, d, d)), np.repeat((np.eye(d) - 0.3 * np.tri(d, k=-1))[None], n, 0)])
    A = np.repeat(0.9 * np.eye(d)[None], n, 0)
    T = np.repeat(0.4 * np.eye(d)[None], n, 0)
    model = W.Model("edge", d, n, np.array(Ns, dtype=np.int64), A, np.zeros((n, d)), T, np.zeros((n + 1, d)), L,
                    np.arange(n + 1.0), 0.0, "basket_put", 1.0, None, 700, 31, W.PREC_F32, "kmeans")
    g = np.concatenate([rng.standard_normal((k, d)) for k in Ns])
    for prec in (W.PREC_F32, W.PREC_F64):
        ref = oracle.transitions(model, g, model.M, model.seed, prec)
        for draw in (0, 1, 2):
            counts, st, _ = ctx.transitions(model, _dev(g), model.M, model.seed,
                                            B.options(prec=prec, tc_chunk_items=chunk, tc_draw=draw))
            got = B.split_counts(model.N, counts.cpu().numpy())
            for k in range(n):
                np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")
            assert st.device_status == 0


@pytest.mark.parametrize("d", [4, 10])
@pytest.mark.parametrize("Ns", [[1, 300, 200], [1, 1, 129, 1], [40, 700, 1, 1, 260]])
def test_few_items_take_their_grids_apart(ctx, B, d, Ns):
    """Up to twice as many items as SMs are screened grid by grid; item counts either side of
    the line, in one window and in windows of 7."""
    n = len(Ns) - 1
    rng = np.random.default_rng(2)
    L = np.concatenate([np.zeros((1, d, d)), np.repeat((np.eye(d) - 0.3 * np.tri(d, k=-1))[None], n, 0)])
    g = np.concatenate([rng.standard_normal((k, d)) for k in Ns])
    line = torch.cuda.get_device_properties(0).multi_processor_count * 2
    for items in (1, line // n, line // n + 1, line + 3):
        M = items * 128 - 5
        model = W.Model("few", d, n, np.array(Ns, dtype=np.int64), np.repeat(0.9 * np.eye(d)[None], n, 0), np.zeros((n, d)),
                        np.repeat(0.4 * np.eye(d)[None], n, 0), np.zeros((n + 1, d)), L, np.arange(n + 1.0), 0.0,
                        "basket_put", 1.0, None, M, 31, W.PREC_F32, "kmeans")
        ref = oracle.transitions(model, g, M, model.seed, W.PREC_F32)
        for chunk in (0, 7):
            counts, st, _ = ctx.transitions(model, _dev(g), M, model.seed, B.options(tc_chunk_items=chunk))
            got = B.split_counts(model.N, counts.cpu().numpy())
            for k in range(n):
                np.testing.assert_array_equal(got[k], ref[k], err_msg=f"items {items} layer {k}")
            assert st.device_status == 0 and st.form_used == B.FORM_TC_RECHECK


@pytest.mark.parametrize("Ns", [[1, 16, 16, 64, 17, 1, 40], [30, 34, 31, 33, 1024, 1, 1024]])
@pytest.mark.parametrize("chunk", [0, 40])
def test_small_layers_count_in_shared_memory(ctx, B, Ns, chunk):
    """Layers of up to 1024 entries (and one more) between larger ones, with many samples."""
    d, n, M = 4, len(Ns) - 1, 70001
    rng = np.random.default_rng(2)
    L = np.concatenate([np.zeros((1, d, d)), np.repeat((np.eye(d) - 0.3 * np.tri(d, k=-1))[None], n, 0)])
    g = np.concatenate([rng.standard_normal((k, d)) for k in Ns])
    model = W.Model("hist", d, n, np.array(Ns, dtype=np.int64), np.repeat(0.9 * np.eye(d)[None], n, 0), np.zeros((n, d)),
                    np.repeat(0.4 * np.eye(d)[None], n, 0), np.zeros((n + 1, d)), L, np.arange(n + 1.0), 0.0,
                    "basket_put", 1.0, None, M, 31, W.PREC_F32, "kmeans")
    ref = oracle.transitions(model, g, M, model.seed, W.PREC_F32)
    for ct in (B.COUNTS_I64, B.COUNTS_U32):
        for flags in (0, B.FLAG_GLOBAL_HIST):
            counts, st, _ = ctx.transitions(model, _dev(g), M, model.seed,
                                            B.options(counts_type=ct, flags=flags, tc_chunk_items=chunk))
            got = B.split_counts(model.N, counts.cpu().numpy())
            for k in range(n):
                np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")
            assert st.device_status == 0
