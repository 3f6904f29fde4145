"""Backward induction and the swing recursion at the sizes where their kernels change:
one launch for a small tree (up to 1024 points, two rows a warp), a launch per layer
above, batches of 1024 columns, V or P in shared memory or not; empty rows, counts of
more than 27 bits, infinite and undefined obstacle values (a zero count times infinity
is undefined, as in the plain sum).

Reference: the recursion in numpy FP64.  Tolerance: at most 3000 products and sums per
row in either order, each with relative error 2^-53, on non-negative terms: (3000 + 3)
2^-53 < 1e-12 a layer; the recursion is a maximum of an exact value and a convex
combination, so it does not grow.
"""
import numpy as np
import pytest

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


def _tree(N, u32, density, seed, wide=False):
    rng = np.random.default_rng(seed)
    blocks = []
    for a, b in zip(N[:-1], N[1:]):
        c = rng.integers(1, 1000, (a, b)) * (rng.random((a, b)) < density)
        if a > 3:
            c[a // 2] = 0                                # an empty row
        if wide:
            c[-1, -1] = (1 << 31) + 5 if u32 else (1 << 40) + 3
        blocks.append(c.astype(np.int64))
    flat = np.concatenate([c.reshape(-1) for c in blocks])
    dev = torch.from_numpy(flat.astype(np.uint32).view(np.int32) if u32 else flat).cuda()
    return blocks, dev


def _backward(blocks, N, phi):
    off = np.concatenate([[0], np.cumsum(N)])
    V = phi.copy()
    for k in range(len(blocks) - 1, -1, -1):
        tot = blocks[k].sum(1)
        with np.errstate(all="ignore"):
            cont = (blocks[k].astype(np.float64) * V[off[k + 1]:off[k + 2]][None, :]).sum(1) / np.maximum(tot, 1)
        ph = phi[off[k]:off[k + 1]]
        V[off[k]:off[k + 1]] = np.where((tot > 0) & ~(ph > cont), cont, ph)
    return V


SIZES = [[1, 2], [1, 33, 5], [1, 500, 500, 500], [1, 1024, 1023, 1, 700], [1024, 609, 608, 1], [1, 1025, 40, 3],
         [5, 2049, 1500, 3000], [1, 1, 1, 1, 1, 1]]


@pytest.mark.parametrize("N", SIZES, ids=[str(s) for s in SIZES])
@pytest.mark.parametrize("u32", [False, True])
@pytest.mark.parametrize("density,wide", [(0.05, False), (1.0, False), (0.3, True)])
def test_backward_values(ctx, B, N, u32, density, wide):
    N = np.array(N, dtype=np.int64)
    blocks, dev = _tree(N, u32, density, 1, wide)
    phi = np.random.default_rng(4).random(int(N.sum())) * 10.0
    ct = B.COUNTS_U32 if u32 else B.COUNTS_I64
    ref = _backward(blocks, N, phi)
    for _ in range(2):
        V = ctx.backward(N, dev, torch.from_numpy(phi).cuda(), ct).cpu().numpy()
        assert np.max(np.abs(V - ref) / np.abs(ref)) < 1e-12


@pytest.mark.parametrize("N", [[1, 300, 200, 100], [1, 1500, 40]])
def test_backward_keeps_infinities_and_undefined_values(ctx, B, N):
    N = np.array(N, dtype=np.int64)
    blocks, dev = _tree(N, False, 0.1, 2)
    for where, value in ((-1, np.inf), (-3, np.nan), (int(N[0] + 7), np.inf), (-2, 1e300)):
        phi = np.random.default_rng(5).random(int(N.sum()))
        phi[where] = value
        ref = _backward(blocks, N, phi)
        V = ctx.backward(N, dev, torch.from_numpy(phi).cuda()).cpu().numpy()
        np.testing.assert_array_equal(np.isnan(V), np.isnan(ref))
        np.testing.assert_array_equal(np.isinf(V), np.isinf(ref))
        ok = np.isfinite(ref)
        assert np.max(np.abs(V[ok] - ref[ok]) / np.maximum(np.abs(ref[ok]), 1e-300)) < 1e-12


@pytest.mark.parametrize("N", [[1, 40, 33], [1, 500, 500, 500, 500], [3, 1100, 1500, 64], [1, 2300, 7]])
@pytest.mark.parametrize("Qmin,Qmax", [(0, 1), (0, 0), (2, 2), (1, 8), (0, 9), (1, 17)])
@pytest.mark.parametrize("u32", [False, True])
def test_swing_values(ctx, B, N, Qmin, Qmax, u32):
    N = np.array(N, dtype=np.int64)
    n = len(N) - 1
    blocks, dev = _tree(N, u32, 0.2, 3, wide=True)
    off = np.concatenate([[0], np.cumsum(N)])
    v = np.random.default_rng(6).random(int(N.sum())) * 5.0
    ok = lambda k, Q: Q <= Qmax and Q + n - k >= Qmin  # noqa: E731
    P = np.array([[0.0 if ok(n, Q) else -np.inf] * int(N[n]) for Q in range(Qmax + 1)])
    want = {n: P}
    for k in range(n - 1, -1, -1):
        tot = blocks[k].sum(1)
        C = {Q: np.where(tot > 0, blocks[k] @ P[Q] / np.maximum(tot, 1), 0.0) for Q in range(Qmax + 1) if ok(k + 1, Q)}
        new = np.full((Qmax + 1, int(N[k])), -np.inf)
        for Q in range(Qmax + 1):
            if Q in C:
                new[Q] = C[Q]
            if Q + 1 in C:
                new[Q] = np.maximum(new[Q], v[off[k]:off[k + 1]] + C[Q + 1])
        P = new
        want[k] = P
    ref = np.concatenate([want[k].reshape(-1) for k in range(n + 1)])
    got, _ = ctx.swing(N, dev, torch.from_numpy(v).cuda(), Qmin, Qmax, B.COUNTS_U32 if u32 else B.COUNTS_I64) \
        if Qmin <= n else (torch.from_numpy(ref), 0.0)
    got = got.cpu().numpy()
    np.testing.assert_array_equal(np.isinf(got), np.isinf(ref))
    fin = np.isfinite(ref)
    assert np.max(np.abs(got[fin] - ref[fin])) <= 1e-12 * max(1.0, np.max(np.abs(ref[fin])))


def test_root_value_of_many_rows(ctx, B):
    """A start distribution of more than 1024 points, and of one row longer than a CTA."""
    for N in ([1500, 20, 10], [1, 3000, 5]):
        N = np.array(N, dtype=np.int64)
        blocks, dev = _tree(N, False, 0.2, 9)
        v = np.random.default_rng(7).random(int(N.sum()))
        P, price = ctx.swing(N, dev, torch.from_numpy(v).cuda(), 0, 1)
        w = blocks[0].sum(1)
        P0 = P.cpu().numpy()[:int(N[0])]
        assert abs(price - (w * P0).sum() / w.sum()) <= 1e-12 * price


@pytest.mark.parametrize("N", [[3, 12289, 40], [1, 9, 13000, 64], [2, 30001, 2]])
@pytest.mark.parametrize("u32", [False, True])
@pytest.mark.parametrize("density,wide", [(0.02, False), (1.0, False), (0.3, True)])
def test_backward_values_beyond_shared_memory(ctx, B, N, u32, density, wide):
    """Layers of more than 12288 points: their values stay in device memory, the lists are the
    same, and so is the sum of 30001 terms: (30001 + 3) 2^-53 < 4e-12."""
    N = np.array(N, dtype=np.int64)
    blocks, dev = _tree(N, u32, density, 1, wide)
    phi = np.random.default_rng(4).random(int(N.sum())) * 10.0
    ct = B.COUNTS_U32 if u32 else B.COUNTS_I64
    for value in (None, np.inf, np.nan):
        if value is not None:
            phi[int(N[:2].sum()) - 5] = value
        ref = _backward(blocks, N, phi)
        V = ctx.backward(N, dev, torch.from_numpy(phi).cuda(), ct).cpu().numpy()
        np.testing.assert_array_equal(np.isnan(V), np.isnan(ref))
        np.testing.assert_array_equal(np.isinf(V), np.isinf(ref))
        ok = np.isfinite(ref)
        assert np.max(np.abs(V[ok] - ref[ok]) / np.abs(ref[ok])) < 4e-12
