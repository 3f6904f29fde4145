"""Calls whose workspace does not fit (the library's allocations above a size fail under
QT_FAULT=alloc_above:B): the tensor-core form takes smaller windows, the located search gives
way to brute force, and the grid builder takes one size at a time.  Results are the same
bits, and no error message is left; a workspace without a smaller form is still refused.
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


def _model(d, n, N, M):
    rng = np.random.default_rng(0)
    A, T = np.repeat(0.9 * np.eye(d)[None], n, 0), np.repeat(0.3 * np.eye(d)[None], n, 0)
    L = np.concatenate([np.zeros((1, d, d)), np.repeat(np.eye(d)[None], n, 0)])
    model = W.Model("mem", d, n, np.array([1] + [N] * n, dtype=np.int64), A, np.zeros((n, d)), T, np.zeros((n + 1, d)), L,
                    np.arange(n + 1.0), 0.0, "put_exp1d", 1.0, None, M, 3, W.PREC_F32, "kmeans")
    return model, np.concatenate([np.zeros((1, d))] + [rng.standard_normal((N, d)) for _ in range(n)])


@pytest.mark.parametrize("d,n,N,M,limit", [(4, 3, 60, 400000, 30 << 20), (2, 60, 100, 6000, 600000), (1, 60, 60, 9000, 200000)])
@pytest.mark.parametrize("paths", [False, True])
def test_forward_step_with_little_memory(B, monkeypatch, d, n, N, M, limit, paths):
    model, g = _model(d, n, N, M)
    ctx = B.Context(0)
    G = torch.from_numpy(g).cuda()
    ref = oracle.pathwise(model, g, M, 3, W.PREC_F32) if paths else oracle.transitions(model, g, M, 3, W.PREC_F32)
    ref = ref[0] if isinstance(ref, tuple) else ref
    want = np.concatenate([c.reshape(-1) for c in ref])
    call = ctx.transitions_pathwise if paths else ctx.transitions
    monkeypatch.setenv("QT_FAULT", f"alloc_above:{limit}")
    for _ in range(3):
        counts, st, _ = call(model, G, M, 3)
        np.testing.assert_array_equal(counts.cpu().numpy(), want)
        assert st.device_status == 0 and ctx.lib.qt_last_error(ctx.h) == b""
    monkeypatch.setenv("QT_FAULT", "alloc_above:1000")
    other, g2 = _model(d, n, N + 500, M)
    with pytest.raises(B.QtError) as e:
        call(other, torch.from_numpy(g2).cuda(), M, 3)
    assert e.value.status == B.QT_ENOMEM
    monkeypatch.delenv("QT_FAULT")
    counts, _, _ = call(model, G, M, 3)
    np.testing.assert_array_equal(counts.cpu().numpy(), want)
    ctx.close()


def test_grid_builder_with_little_memory(B, monkeypatch):
    d, N = 3, [1, 40, 130, 90]
    n = len(N) - 1
    model, _ = _model(d, n, 1, 10)
    model.N = np.array(N, dtype=np.int64)
    ctx = B.Context(0)
    want = ctx.build_grids(model, B.GRID_KMEANS, samples=30000, iters=3, seed=5)
    ctx.close()
    ctx = B.Context(0)
    monkeypatch.setenv("QT_FAULT", f"alloc_above:{30000 * d * 4 + 20000}")
    got = ctx.build_grids(model, B.GRID_KMEANS, samples=30000, iters=3, seed=5)
    assert torch.equal(got, want) and ctx.lib.qt_last_error(ctx.h) == b""
    ctx.close()
