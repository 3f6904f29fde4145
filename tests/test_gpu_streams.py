"""One context called from several streams, and several times in a row, without waiting in
between: the workspace is handed from one step to the next on the device.  Results are
compared bit for bit with the same calls made one at a time (and those with the oracle in
the other tests).
"""
import ctypes

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


@pytest.fixture()
def ctx(B):
    c = B.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _samples_async(ctx, B, gA, gB, X, Y, counts, stream):
    """qt_counts_from_samples without statistics: it returns before the step has run."""
    o = B.options()
    ctx._check(ctx.lib.qt_counts_from_samples(ctx.h, gA.shape[1], gA.data_ptr(), gA.shape[0], gB.data_ptr(), gB.shape[0],
                                              X.data_ptr(), Y.data_ptr(), X.shape[0], ctypes.byref(o), counts.data_ptr(),
                                              None, None, None, stream.cuda_stream))


@pytest.mark.parametrize("d", [2, 4])
def test_given_samples_on_two_streams(ctx, B, d):
    """The second call's grids, of the same sizes, must not reach the first call's recheck: most
    of its samples tie between two points and are decided from the FP64 grids."""
    N, M = 900, 3000000
    rng = np.random.default_rng(d)
    pairs = []
    for k in range(2):
        gA, gB = rng.standard_normal((N, d)), rng.standard_normal((N, d))
        tie = W.boundary_samples(gA, 2000, seed=k), W.boundary_samples(gB, 2000, seed=7 + k)
        m = M if k == 0 else 2000
        pairs.append([_dev(gA), _dev(gB)] + [_dev(np.resize(t, (m, d))) for t in tie])
    want = []
    for gA, gB, X, Y in pairs:
        want.append(ctx.counts_from_samples(gA, gB, X, Y)[0])
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    for rep in range(3):
        got = [torch.empty_like(w) for w in want]
        torch.cuda.synchronize()
        for k in range(2):
            _samples_async(ctx, B, *pairs[k], got[k], s[k])
        torch.cuda.synchronize()
        for k in range(2):
            assert torch.equal(got[k], want[k]), (rep, k)


@pytest.mark.parametrize("d", [1, 2, 4])
def test_trees_on_two_streams(ctx, B, d):
    """Steps of different shapes alternate between two streams without a wait: uploads,
    tables and counts of one step are not another's (the third time round from a graph)."""
    rng = np.random.default_rng(3)
    cases = []
    for k, Ns in enumerate(((40, 300, 150), (700, 20), (100, 100, 100, 100))):
        n = len(Ns)
        A, T = np.repeat(0.9 * np.eye(d)[None], n, 0), np.repeat(0.3 * np.eye(d)[None], n, 0)
        L = np.concatenate([np.zeros((1, d, d)), np.repeat(np.eye(d)[None], n, 0)])
        model = W.Model("s", d, n, np.array((1,) + Ns, dtype=np.int64), A, np.zeros((n, d)), T, np.zeros((n + 1, d)), L,
                        np.arange(n + 1.0), 0.0, "put_exp1d", 1.0, None, 200000 + 777 * k, 5 + k, W.PREC_F32, "kmeans")
        g = np.concatenate([np.zeros((1, d))] + [rng.standard_normal((q, d)) for q in Ns])
        want = np.concatenate([c.reshape(-1) for c in oracle.transitions(model, g, model.M, model.seed, W.PREC_F32)])
        cases.append((model, _dev(g), torch.empty(len(want), dtype=torch.int64, device="cuda"), want))
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    for rep in range(4):
        for _, _, counts, _ in cases:
            counts.fill_(-1)
        torch.cuda.synchronize()
        for k, (model, g, counts, _) in enumerate(cases * 2):
            ctx.transitions(model, g, model.M, model.seed, counts=counts, want_stats=False, stream=s[k % 2])
        torch.cuda.synchronize()
        for k, (_, _, counts, want) in enumerate(cases):
            np.testing.assert_array_equal(counts.cpu().numpy(), want, err_msg=f"case {k}, round {rep}")


def test_backward_on_two_streams(ctx, B):
    """One-launch inductions of growing depth alternate between two streams while a long
    kernel holds the first: their layer tables are uploaded from pinned blocks that grow."""
    rng = np.random.default_rng(1)
    cases = []
    for n in (3, 8, 20, 60, 150, 400):
        N = np.array([1] + [40] * n, dtype=np.int64)
        counts = rng.integers(0, 50, int(np.sum(N[:-1] * N[1:])))
        phi = rng.random(int(N.sum()))
        off, want = np.concatenate([[0], np.cumsum(N)]), phi.copy()
        at = len(counts)
        for k in range(n - 1, -1, -1):
            c = counts[at - N[k] * N[k + 1]:at].reshape(N[k], N[k + 1]).astype(np.float64)
            at -= N[k] * N[k + 1]
            cont = c @ want[off[k + 1]:off[k + 2]] / c.sum(1)
            want[off[k]:off[k + 1]] = np.maximum(phi[off[k]:off[k + 1]], cont)
        cases.append((N, _dev(counts), _dev(phi), want))
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    busy = torch.empty(1 << 28, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s[0]):
        for _ in range(20):
            busy.add_(1.0)
    got = [ctx.backward(N, counts, phi, stream=s[k % 2]) for k, (N, counts, phi, _) in enumerate(cases)]
    torch.cuda.synchronize()
    for V, (_, _, _, want) in zip(got, cases):
        # 40 terms a row in either order, non-negative: (40 + 3) 2^-53 a layer, no growth
        np.testing.assert_allclose(V.cpu().numpy(), want, rtol=1e-13, atol=0)
