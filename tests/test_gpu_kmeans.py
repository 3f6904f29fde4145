"""Sample Lloyd against numpy at the sizes where its kernels change: groups of 16
centres, tiles of 48 KB, draws per thread, dimension classes with padding, several
grid sizes in a launch, draws of different numbers.

Reference: one and two iterations on the same draws (the oracle's sampler, layer index
0xFFFF): the FP32 chain of fused multiply-adds in FP64 (a product of two FP32 is exact
there, and the sum's second rounding moves a distance for one in 2^29), the first
minimum, and whole-number sums at scale 2^36, so the centres are equal bit for bit.
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


def _lloyd(d, N, S, seed, iters):
    kseed = (seed ^ (0x9E3779B97F4A7C15 * N)) & 0xFFFFFFFFFFFFFFFF
    Z = np.asarray(oracle.normals(oracle.PREC_F32, kseed, 0xFFFF, 0, S, d)).astype(np.float32)
    C = Z[:N].copy()
    fixed = np.rint(Z.astype(np.float64) * 2.0**36).astype(np.int64)
    for _ in range(iters):
        idx = np.empty(S, dtype=np.int64)
        for a in range(0, S, 1000):
            acc = np.zeros((min(1000, S - a), N), dtype=np.float32)
            for l in range(d):
                df = Z[a:a + 1000, l, None] - C[None, :, l]
                acc = (df.astype(np.float64)**2 + acc).astype(np.float32)
            idx[a:a + 1000] = acc.argmin(1)
        cnt = np.bincount(idx, minlength=N)
        for l in range(d):
            s = np.zeros(N, dtype=np.int64)
            np.add.at(s, idx, fixed[:, l])
            C[cnt > 0, l] = ((s[cnt > 0] / 2.0**36) / cnt[cnt > 0]).astype(np.float32)
    return C


@pytest.mark.parametrize("d", [1, 2, 3, 4, 6, 7, 10, 11, 16])
@pytest.mark.parametrize("N,S,iters", [((2, 15, 16, 17), 129, 2), ((1, 48, 47, 48, 1000), 4097, 1), ((800, 3), 1023, 2),
                                       ((33,), 160001, 1)])
def test_centres_bit_exact(ctx, B, d, N, S, iters):
    if S > 100000 and d not in (2, 7):
        pytest.skip("the many-draw rule once for each half of the classes")
    n = len(N)
    eye = np.repeat(np.eye(d)[None], n + 1, 0)
    model = W.Model("chain", d, n, np.array((1,) + N, dtype=np.int64), 0.5 * eye[1:], np.zeros((n, d)), 0.1 * eye[1:],
                    np.zeros((n + 1, d)), eye, np.arange(n + 1.0), 0.0, "put_exp1d", 1.0, None, 1000, 99, W.PREC_F32,
                    "kmeans")
    g = ctx.build_grids(model, B.GRID_KMEANS, samples=S, iters=iters, seed=77).cpu().numpy().reshape(-1, d)
    off = model.offsets()
    for k in range(n + 1):
        Nk = int(model.N[k])
        ref = np.zeros((1, d)) if Nk == 1 else _lloyd(d, Nk, S, 77, iters)
        np.testing.assert_array_equal(g[off[k]:off[k + 1]].astype(np.float32), ref.astype(np.float32))
