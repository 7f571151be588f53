"""The dense Hessian's product at the edges of its tiles, slabs and token chunks, with chunk partials
in memory (few tiles) and in tensor memory (many), against fp64. Bar: 3xTF32 products lose about
2^-22 each and the tensor core's fp32 accumulation about 2^-23 per step of eight tokens within a
chunk of 1024, together below 3e-5 of sum_k |x_ka x_kb| / n."""
import numpy as np
import pytest

import paper_2412_09282_gb300 as P
from parity_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [(1, 8), (15, 128), (17, 136), (1023, 256), (1025, 264),
                                 (2048, 520), (33, 4904), (1040, 4872)])
def test_dense_hessian_edges(n, N):
    rng = np.random.default_rng(n + N)
    X = (rng.standard_normal((n, N)) * rng.lognormal(0.0, 0.5, N)).astype(np.float32)
    H, xsq, Hb, delta = [host(t).astype(np.float64) for t in P.crvq_hessian(dev(X), 0.01)]
    P.crvq_sync()
    X64 = X.astype(np.float64)
    S = X64.T @ X64 / n
    scale = np.abs(X64).T @ np.abs(X64) / n
    d = float(np.float32(0.01)) * np.diag(S).mean()
    assert abs(delta[0] - d) <= 4e-5 * d
    assert np.all(np.abs(xsq - np.diag(S)) <= 3e-5 * np.diag(S))
    assert np.array_equal(H, H.T)
    assert np.all(np.abs(H - S - d * np.eye(N)) <= 3e-5 * scale + 5e-5 * d * np.eye(N))
    G = N // 8
    i = np.arange(G)
    np.testing.assert_array_equal(Hb, H.reshape(G, 8, G, 8)[i, :, i, :])


@pytest.mark.parametrize("n,N", [(1, 8), (16, 128), (17, 136), (8000, 128), (8200, 128), (1024, 1016),
                                 (100, 1024), (100, 1032), (1025, 512), (1025, 520)])
def test_hessian_blocks_small_sizes(n, N):
    """On both sides of the line up to which one block sums, damps and writes the blocks (1024 channels,
    8192 terms): the same bits as the dense call, and as the blocks of the identity order."""
    rng = np.random.default_rng(n * N)
    X = dev((rng.standard_normal((n, N)) * rng.lognormal(0.0, 0.5, N)).astype(np.float32))
    _, xsq, Hb, delta = P.crvq_hessian(X, 0.01)
    Hb2, xsq2, delta2 = P.crvq_hessian_blocks(X, 0.01)
    P.crvq_sync()
    for a, b in ((xsq, xsq2), (Hb, Hb2), (delta, delta2)):
        np.testing.assert_array_equal(host(a), host(b))
    order = dev(np.arange(N, dtype=np.int32))
    np.testing.assert_array_equal(host(P.crvq_hessian_blocks(X, 0.01, perm=order)[0]), host(Hb2))
