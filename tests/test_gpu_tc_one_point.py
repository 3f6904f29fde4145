"""The tensor-core form on layers whose two grids have one point each: their items need no
screen, and a CTA has many of them in a row before a layer that needs one.  The counts of
such a layer are M; the others are compared with the oracle bit for bit.
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


@pytest.mark.parametrize("d", [3, 8])
@pytest.mark.parametrize("Ns", [[1, 1, 300], [1, 1, 1], [1, 40, 1, 1, 1, 20], [1, 1, 17, 1, 1]])
def test_layers_of_one_point(B, d, Ns):
    n = len(Ns) - 1
    rng = np.random.default_rng(d)
    L = np.concatenate([np.zeros((1, d, d)), np.repeat((np.eye(d) - 0.3 * np.tri(d, k=-1))[None], n, 0)])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    big = 8 * 128 * 4 * sms + 77                         # more than eight items a CTA and layer
    g = np.concatenate([rng.standard_normal((k, d)) for k in Ns])
    ctx = B.Context(0)
    for M, chunk in ((big, 0), (big, 1000), (300, 0)):
        model = W.Model("one_point", d, n, np.array(Ns, dtype=np.int64), np.repeat(0.9 * np.eye(d)[None], n, 0),
                        np.zeros((n, d)), np.repeat(0.4 * np.eye(d)[None], n, 0), np.zeros((n + 1, d)), L,
                        np.arange(n + 1.0), 0.0, "basket_put", 1.0, None, M, 31, W.PREC_F32, "kmeans")
        counts, st, _ = ctx.transitions(model, torch.from_numpy(g).cuda(), M, model.seed,
                                        B.options(form=B.FORM_TC_RECHECK, tc_chunk_items=chunk))
        assert st.device_status == 0
        got = B.split_counts(model.N, counts.cpu().numpy())
        ref = oracle.transitions(model, g, M, model.seed, W.PREC_F32)
        for k in range(n):
            np.testing.assert_array_equal(got[k], ref[k], err_msg=f"layer {k}")
    ctx.close()
