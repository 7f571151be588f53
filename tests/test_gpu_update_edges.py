"""Edges of the codebook update's accumulation (four adjacent groups per block; sums in shared memory up
to 1024 codewords), of its solve (codewords per block by their number) and of the keep-if-better step
(only changed tuples are compared) against the fp64 oracle. Counts are exact;
codebooks agree to fp32 rounding of the solve (1e-4 of the largest value, the bar of the parity
tests); codes equal the oracle's up to fp64 near-ties."""
import numpy as np
import pytest

import paper_2412_09282_gb300 as P
from paper_2412_09282_gb300 import Codebook
from oracle import crvq_oracle as O
from parity_util import check_codes_with_ties, dev, host

pytestmark = pytest.mark.gpu

D = 8


def _blocks(rng, G, n=64):
    X = rng.standard_normal((n, G * D)) * rng.lognormal(0.0, 0.5, G * D)
    Xb = X.reshape(n, G, D).transpose(1, 0, 2)
    return (Xb.transpose(0, 2, 1) @ Xb / n + 0.05 * np.eye(D)).astype(np.float32)


@pytest.mark.parametrize("M,G,Gc,K", [
    (1, 1, 1, 3), (127, 3, 2, 256), (129, 4, 1, 256), (400, 5, 4, 257), (700, 9, 6, 100),
    # the larger shared sums, the global sums, and the solve's four and eight codewords per CTA
    (500, 6, 5, 305), (900, 7, 3, 611), (1300, 5, 5, 1024), (1300, 9, 2, 1025), (257, 4, 3, 4099)])
def test_update_over_group_quads(M, G, Gc, K):
    rng = np.random.default_rng(100 * G + K)
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    Hb = _blocks(rng, G)
    Cs = [(0.02 * rng.standard_normal((k, D))).astype(np.float32) for k in (K, 5)]
    codes = [rng.integers(0, k, (M, g)).astype(np.int32) for k, g in ((K, G), (5, Gc))]
    cbs = [Codebook(dev(C), dev(c), g) for C, c, g in zip(Cs, codes, (G, Gc))]
    ocbs = [O.Codebook(C, c, g) for C, c, g in zip(Cs, codes, (G, Gc))]
    for which in (0, 1):
        Cg, cnt = P.crvq_update_codebook(dev(W), D, dev(Hb), cbs, which)
        P.crvq_sync()
        Co, co = O.update_codebook(W, D, Hb, ocbs, which)
        np.testing.assert_array_equal(host(cnt), co)
        assert np.abs(host(Cg).astype(np.float64) - Co).max() <= 1e-4 * np.abs(Co).max()


@pytest.mark.parametrize("share", [0.0, 0.05, 1.0])
@pytest.mark.parametrize("M,G,Gc", [(1, 1, 1), (600, 5, 2)])
def test_keep_if_better_over_changed_tuples(M, G, Gc, share):
    """`share` of the old codes are random, the others the best ones: none, a few or all of the
    tuples change."""
    rng = np.random.default_rng(int(100 * share) + M)
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    Hb = _blocks(rng, G)
    Cs = [(0.02 * rng.standard_normal((k, D))).astype(np.float32) for k in (40, 7)]
    fresh = [O.Codebook(C, None, g) for C, g in zip(Cs, (G, Gc))]
    old, _ = O.encode_beam(W, D, Hb, fresh, 0, 4)
    for s, k in enumerate((40, 7)):
        r = rng.random(old[s].shape) < share
        old[s] = np.where(r, rng.integers(0, k, old[s].shape), old[s]).astype(np.int32)
    codes = [dev(c) for c in old]
    cbs = [Codebook(dev(C), c, g) for C, c, g in zip(Cs, codes, (G, Gc))]
    P.crvq_encode_beam(dev(W), D, dev(Hb), cbs, 0, 2, keep_if_better=True)
    P.crvq_sync()
    ocbs = [O.Codebook(C, c, g) for C, c, g in zip(Cs, old, (G, Gc))]
    oc, _ = O.encode_beam(W, D, Hb, ocbs, 0, 2, keep_if_better=True)
    check_codes_with_ties(W, D, Hb, ocbs, 0, [host(c) for c in codes], oc)
