"""Given samples so far from the grid that FP32 scores overflow, and samples that are not
finite: the window search has no finite window for them.  Far samples take the exact
FP64 argmin over the whole grid (compared bit for bit with the oracle, which evaluates
the same FP64 distances); a sample without a finite distance has no cell and is refused.
"""
import numpy as np
import pytest

import oracle

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


FORMS = [("FORM_AUTO", 1), ("FORM_AUTO", 2), ("FORM_F32_RECHECK", 1), ("FORM_F32_RECHECK", 2),
         ("FORM_F32_RECHECK", 12), ("FORM_TC_RECHECK", 3), ("FORM_TC_RECHECK", 8)]


@pytest.mark.parametrize("form,d", FORMS)
@pytest.mark.parametrize("NA,NB", [(2, 20), (33, 40), (64, 301)])
def test_far_samples(ctx, B, form, d, NA, NB):
    rng = np.random.default_rng(NA + d)
    gA, gB = rng.standard_normal((NA, d)), rng.standard_normal((NB, d)) + 0.5
    M = 400
    X, Y = rng.standard_normal((M, d)), rng.standard_normal((M, d))
    for k, e in enumerate((3, 9, 18, 19.5, 25, 37, 38.4, 60, 150)):
        X[k::23] *= 10.0 ** e
        Y[k + 1::29] *= 10.0 ** e
    counts, st, ii, jj = ctx.counts_from_samples(_dev(gA), _dev(gB), _dev(X), _dev(Y), B.options(form=getattr(B, form)),
                                                 want_cells=True)
    np.testing.assert_array_equal(ii.cpu().numpy(), oracle.nearest(gA, X))
    np.testing.assert_array_equal(jj.cpu().numpy(), oracle.nearest(gB, Y))
    np.testing.assert_array_equal(counts.cpu().numpy(), oracle.counts_from_samples(gA, gB, X, Y))
    assert st.device_status == 0


@pytest.mark.parametrize("form,d", FORMS)
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_undefined_samples_are_refused(ctx, B, form, d, bad):
    rng = np.random.default_rng(d)
    g = rng.standard_normal((40, d))
    X = rng.standard_normal((300, d))
    Y = X.copy()
    Y[200, d - 1] = bad
    with pytest.raises(B.QtError) as e:
        ctx.counts_from_samples(_dev(g), _dev(g), _dev(X), _dev(Y), B.options(form=getattr(B, form)))
    assert e.value.status == B.QT_EDEVICE
    # the context stays usable
    counts, _, _, _ = ctx.counts_from_samples(_dev(g), _dev(g), _dev(X), _dev(X), B.options(form=getattr(B, form)))
    np.testing.assert_array_equal(counts.cpu().numpy(), oracle.counts_from_samples(g, g, X, X))


def test_refusal_while_other_blocks_start(ctx, B):
    """Errors recorded by the first blocks of the tensor-core form's last kernel while others
    begin: every block takes one decision, and the call ends with the refusal, not a timeout."""
    d, M = 3, 400000
    rng = np.random.default_rng(5)
    g = rng.standard_normal((50, d))
    X = rng.standard_normal((M, d))
    X[::97, 0] = np.nan
    for _ in range(20):
        with pytest.raises(B.QtError) as e:
            ctx.counts_from_samples(_dev(g), _dev(g), _dev(X), _dev(X), B.options(form=B.FORM_TC_RECHECK))
        assert e.value.status == B.QT_EDEVICE
