"""The one-launch backward induction's bounded waits: one that runs out (the library gives
up at once under QT_FAULT=timeout_tree) is reported, by qt_get_status after qt_backward and
by qt_price itself, and the context stays usable.
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


def _tree(d=2, n=5, N=300, M=20000):
    rng = np.random.default_rng(0)
    A, T = np.repeat(0.9 * np.eye(d)[None], n, 0), np.repeat(0.3 * np.eye(d)[None], n, 0)
    L = np.concatenate([np.zeros((1, d, d)), np.repeat(np.eye(d)[None], n, 0)])
    model = W.Model("t", d, n, np.array([1] + [N] * n, dtype=np.int64), A, np.zeros((n, d)), T, np.zeros((n + 1, d)), L,
                    np.arange(n + 1.0), 0.0, "put_exp1d", 1.0, None, M, 3, W.PREC_F32, "kmeans")
    g = np.concatenate([np.zeros((1, d))] + [rng.standard_normal((N, d)) for _ in range(n)])
    return model, g, np.maximum(1.0 - np.exp(g.sum(1)), 0.0)


@pytest.mark.parametrize("u32", [False, True])
def test_a_wait_that_runs_out_is_reported(B, monkeypatch, u32):
    model, g, phi = _tree()
    opts = B.options(counts_type=B.COUNTS_U32 if u32 else B.COUNTS_I64)
    ref = oracle.transitions(model, g, model.M, model.seed, W.PREC_F32)
    want = oracle.price(model.N, ref, phi)
    ctx = B.Context(0)
    G, PHI = torch.from_numpy(g).cuda(), torch.from_numpy(phi).cuda()
    counts, _, _ = ctx.transitions(model, G, model.M, model.seed, opts)
    assert ctx.status()[0] == B.QT_OK
    V = ctx.backward(model.N, counts, PHI, opts.counts_type)
    assert ctx.status()[0] == B.QT_OK
    assert abs(float(V[0]) - want) <= 1e-12 * abs(want)
    monkeypatch.setenv("QT_FAULT", "timeout_tree")
    ctx.backward(model.N, counts, PHI, opts.counts_type)
    assert ctx.status()[0] == B.QT_ETIMEOUT
    with pytest.raises(B.QtError) as e:
        ctx.price(model, g, model.M, model.seed, phi, opts)
    assert e.value.status == B.QT_ETIMEOUT
    monkeypatch.delenv("QT_FAULT")
    price, st = ctx.price(model, g, model.M, model.seed, phi, opts)
    assert st.device_status == 0 and abs(price - want) <= 1e-12 * abs(want)
    V = ctx.backward(model.N, counts, PHI, opts.counts_type)
    assert ctx.status()[0] == B.QT_OK and abs(float(V[0]) - want) <= 1e-12 * abs(want)
    # an error of the induction is not the next forward step's
    monkeypatch.setenv("QT_FAULT", "timeout_tree")
    ctx.backward(model.N, counts, PHI, opts.counts_type)
    monkeypatch.delenv("QT_FAULT")
    ctx.transitions(model, G, model.M, model.seed, opts)
    ctx.close()


def test_without_workspace_layer_by_layer(B, monkeypatch):
    """No memory for the one launch: the induction runs a launch per layer, succeeds, and
    leaves no message of the allocation that failed."""
    model, g, phi = _tree()
    ref = oracle.transitions(model, g, model.M, model.seed, W.PREC_F32)
    want = oracle.price(model.N, ref, phi)
    counts = torch.from_numpy(np.concatenate([c.reshape(-1) for c in ref]).astype(np.int64)).cuda()
    ctx = B.Context(0)
    monkeypatch.setenv("QT_FAULT", "alloc")
    V = ctx.backward(model.N, counts, torch.from_numpy(phi).cuda())
    monkeypatch.delenv("QT_FAULT")
    assert abs(float(V[0]) - want) <= 1e-12 * abs(want)
    assert ctx.lib.qt_last_error(ctx.h) == b""
    ctx.close()
