"""Edges of the arg-min kernels against the fp64 oracle: codebook sizes around the 128-codeword
chunks and the 256-codeword limit between the resident and the streaming kernel, row counts around
the 128-row tiles and their pairs, shares that span several groups, rows left open by the certificate
(duplicate and nearly equal codewords, more of them than a CTA's list holds). Codes must be the fp64
arg-min, ties to the smaller index, except at fp64 near-ties (parity_util)."""
import numpy as np
import pytest
import torch

import paper_2412_09282_gb300 as P
from paper_2412_09282_gb300 import Codebook
from oracle import crvq_oracle as O
from parity_util import check_codes_with_ties, dev, host
from synthetic import LayerConfig

pytestmark = pytest.mark.gpu

D = 8


def _blocks(rng, G, n=64):
    X = rng.standard_normal((n, G * D)) * rng.lognormal(0.0, 0.5, G * D)
    Xb = X.reshape(n, G, D).transpose(1, 0, 2)
    return (Xb.transpose(0, 2, 1) @ Xb / n + 0.05 * np.eye(D)).astype(np.float32)


def _encode(W, Hb, C):
    M, G = W.shape[0], Hb.shape[0]
    codes = torch.full((M, G), -1, dtype=torch.int32, device="cuda")
    err = P.crvq_encode_beam(dev(W), D, dev(Hb), [Codebook(dev(C), codes, G)], 0, 1, want_err=True)
    P.crvq_sync()
    return host(codes), host(err)


def _check(W, Hb, C):
    codes, err = _encode(W, Hb, C)
    cb = [O.Codebook(C, None, Hb.shape[0])]
    oc, oerr = O.encode_beam(W, D, Hb, cb, 0, 1)
    check_codes_with_ties(W, D, Hb, cb, 0, [codes], oc)
    np.testing.assert_allclose(err, oerr, rtol=1e-5, atol=1e-12)
    return codes


@pytest.mark.parametrize("M,G,K", [
    (1, 1, 1), (127, 3, 2), (128, 2, 127), (129, 2, 128), (255, 5, 129), (256, 1, 255),
    (257, 7, 256), (300, 650, 16),                                   # shares over several groups
    (130, 2, 257), (1, 3, 384), (257, 2, 385), (129, 3, 1025), (64, 2, 3000),
    (300, 310, 257), (257, 210, 640), (130, 320, 1100)])             # a row tile per half of a block
def test_codebook_and_row_edges(M, G, K):
    rng = np.random.default_rng(M * 1000 + K)
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    C = (0.02 * rng.standard_normal((K, D))).astype(np.float32)
    _check(W, _blocks(rng, G), C)


def test_more_groups_than_one_sub_range():
    """K = 3000: the operand images of about 2760 groups fit a sub-range; the shared part of the
    images serves the second one too."""
    rng = np.random.default_rng(11)
    M, G, K = 2, 2800, 3000
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    C = (0.02 * rng.standard_normal((K, D))).astype(np.float32)
    _check(W, _blocks(rng, G), C)


@pytest.mark.parametrize("K", [15, 16, 17, 129, 200, 241])
def test_block_and_class_edges(K):
    """Codebook sizes around the 16-column blocks of the sweep, whose two smallest minima carry their
    block's number in their low bits; several groups per CTA and an odd number of row tiles."""
    rng = np.random.default_rng(K)
    M, G = 385, 260
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    C = (0.02 * rng.standard_normal((K, D))).astype(np.float32)
    _check(W, _blocks(rng, G), C)


@pytest.mark.parametrize("K", [64, 256, 600])
def test_rows_open_by_close_codewords(K):
    """Every codeword twice, the copy one unit in the last place off: no row is certified."""
    rng = np.random.default_rng(K)
    M, G = 700, 4
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    C = (0.02 * rng.standard_normal((K // 2, D))).astype(np.float32)
    near = np.nextafter(C, np.float32(1)).astype(np.float32)
    _check(W, _blocks(rng, G), np.concatenate([C, near]))
    # exact duplicates: the smaller index of every pair
    codes, _ = _encode(W, _blocks(rng, G), np.concatenate([C, C]))
    assert codes.max() < K // 2


@pytest.mark.parametrize("K", [200, 700])
def test_three_close_codewords_in_different_granules(K):
    """Triples of almost equal codewords spread over the codebook: more candidates than the two
    granules that the large pass keeps."""
    rng = np.random.default_rng(K + 1)
    M, G = 260, 3
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    base = (0.02 * rng.standard_normal((K // 4, D))).astype(np.float32)
    C = np.concatenate([base * (1 + 1e-7 * t) for t in range(4)]).astype(np.float32)
    _check(W, _blocks(rng, G), C)


@pytest.mark.parametrize("K", [64, 256])
def test_open_rows_more_than_a_list_holds(K):
    """1950 tile pairs in at most a few hundred blocks, every row open (the copies are one unit in the last
    place off): a block finds over a thousand open rows, four times what its list holds, so most are
    decided inside the running pipeline. The same codes as four groups at a time, where a block has one
    tile pair and its list holds every row; sampled groups against the oracle."""
    rng = np.random.default_rng(K)
    M, G = 700, 650
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    C = (0.02 * rng.standard_normal((K // 2, D))).astype(np.float32)
    C = np.concatenate([C, np.nextafter(C, np.float32(1))]).astype(np.float32)
    Hb = _blocks(rng, G)
    Wd, Hd, Cd = dev(W), dev(Hb), dev(C)

    def run(g0, n):
        codes = torch.full((M, n), -1, dtype=torch.int32, device="cuda")
        P.crvq_encode_beam(Wd[:, g0 * D:(g0 + n) * D], D, Hd[g0:g0 + n], [Codebook(Cd, codes, n)], 0, 1)
        P.crvq_sync()
        return host(codes)

    codes = run(0, G)
    parts = np.concatenate([run(g0, min(4, G - g0)) for g0 in range(0, G, 4)], axis=1)
    np.testing.assert_array_equal(codes, parts)
    for g in (0, 317, 649):
        T, cb = W[:, g * D:(g + 1) * D], [O.Codebook(C, None, 1)]
        oc, _ = O.encode_beam(T, D, Hb[g:g + 1], cb, 0, 1)
        check_codes_with_ties(T, D, Hb[g:g + 1], cb, 0, [codes[:, g:g + 1]], oc)


def test_lloyd_statistics_of_open_rows_more_than_a_list_holds():
    """A layer's base codebook after one Lloyd iteration from an initial codebook whose codewords come in
    pairs one unit in the last place apart: every row of its pass is open, far more per block than the list
    holds. Counts and sums of all of them: the same codebook and codes, bit for bit, as a separate
    encode, update and encode."""
    M, G, K = 700, 650, 64
    N = G * D
    rng = np.random.default_rng(9)
    cfg = LayerConfig("open_rows", M, N, 64, "plain", "lognormal", K_base=K, n_ext=0, B=1,
                      kmeans_iters=1, refine_rounds=0, importance_mode=2)
    X = dev(rng.standard_normal((64, N)).astype(np.float32))
    W = (0.02 * rng.standard_normal((M, N))).astype(np.float32)
    perm = P.crvq_quantize_layer(dev(W), X, cfg).perm  # the random order depends on the seed alone
    Ws = W[:, host(perm)].reshape(M * G, D)
    at = O.kmeans_sample_indices(M * G, K, O.phase_seed(cfg.seed, O.PHASE_BASE, 0))
    for a, b in zip(at[0::2], at[1::2]):
        Ws[b] = np.nextafter(Ws[a], np.float32(1))
    W[:, host(perm)] = Ws.reshape(M, N)
    out = P.crvq_quantize_layer(dev(W), X, cfg)
    assert torch.equal(out.perm, perm)
    assert out.report["flagged"] > M * G // 2

    T = dev(Ws.reshape(M, N))
    Hb, _, _ = P.crvq_hessian_blocks(X, cfg.damp_rel, perm=perm)
    C = P.crvq_kmeans_init(T, D, G, K, O.phase_seed(cfg.seed, O.PHASE_BASE, 0))
    codes = torch.empty((M, G), dtype=torch.int32, device="cuda")
    P.crvq_encode_beam(T, D, Hb, [Codebook(C, codes, G)], 0, 1)
    C, counts = P.crvq_update_codebook(T, D, Hb, [Codebook(C, codes, G)], 0)
    assert int(counts.sum()) == M * G
    P.crvq_encode_beam(T, D, Hb, [Codebook(C, codes, G)], 0, 1)
    P.crvq_sync()
    assert torch.equal(out.C_base, C)
    assert torch.equal(out.codes_base, codes)


@pytest.mark.parametrize("K,M", [(600, 300), (1100, 300), (1100, 40), (2500, 300)])
def test_open_rows_by_repeated_codewords_of_a_large_codebook(K, M):
    """Half of the vectors and of the codewords zero: thousands of rows open over most of the codebook
    (with 40 rows: hundreds, which blocks take instead of warps above 1024 codewords)."""
    rng = np.random.default_rng(K + M)
    G = 40
    W = (0.02 * rng.standard_normal((M, G, D))).astype(np.float32)
    W[rng.random((M, G)) < 0.5] = 0.0
    C = (0.02 * rng.standard_normal((K, D))).astype(np.float32)
    C[rng.random(K) < 0.5] = 0.0
    C[7] = 0.0
    codes = _check(W.reshape(M, G * D), _blocks(rng, G), C)
    assert codes[(W == 0).all(2)].max() <= 7


@pytest.mark.parametrize("K", [40, 256])
def test_repeated_codewords_do_not_open_rows(K):
    """Half of the vectors and of the codewords zero (of both signs), others repeated: the smallest index of
    equal codewords, and few rows that need an exact decision."""
    rng = np.random.default_rng(K)
    M, G = 300, 9
    W = (0.02 * rng.standard_normal((M, G, D))).astype(np.float32)
    W[rng.random((M, G)) < 0.5] = 0.0
    W = W.reshape(M, G * D)
    C = (0.02 * rng.standard_normal((K, D))).astype(np.float32)
    C[rng.random(K) < 0.5] = 0.0
    C[rng.random(K) < 0.2] *= -0.0
    C[K - 4:] = C[:4]
    codes = _check(W, _blocks(rng, G), C)
    first = np.array([np.nonzero((C == c).all(1))[0][0] for c in C])
    np.testing.assert_array_equal(first[codes], codes)

    cfg = LayerConfig("zeros", M, G * D, 64, "plain", "lognormal", K_base=K, n_ext=0, B=1,
                      kmeans_iters=2, refine_rounds=0)
    out = P.crvq_quantize_layer(dev(W), dev(rng.standard_normal((64, G * D)).astype(np.float32)), cfg)
    assert out.report["flagged"] < 0.1 * 6 * M * G  # six passes


def _tail_errs(T, C0s, H):
    """errs of one group that the searched codebook does not cover: T minus the fixed codebooks C0s (one
    codeword each), from crvq_encode_beam."""
    M = T.shape[0]
    W = np.concatenate([np.zeros((M, D), np.float32), T], axis=1)
    Hb = np.stack([np.eye(D, dtype=np.float32), H])
    zeros = torch.zeros((M, 2), dtype=torch.int32, device="cuda")
    cbs = [Codebook(dev(C.reshape(1, D)), zeros, 2) for C in C0s]
    cbs.append(Codebook(dev(np.zeros((1, D), np.float32)), torch.zeros_like(zeros[:, :1]), 1))
    err = P.crvq_encode_beam(dev(W), D, dev(Hb), cbs, len(C0s), 1, want_err=True)
    P.crvq_sync()
    r = T.astype(np.float64) - sum((C.astype(np.float64) for C in C0s), np.zeros(D))
    H = H.astype(np.float64)
    with np.errstate(over="ignore"):
        return host(err)[:, 1], np.einsum("md,de,me->m", r, H, r).astype(np.float32)


@pytest.mark.parametrize("scale", [1e20, 1.0, 1e-15, 1e-18, 1e-19, 3e-20, 1e-22])
def test_errs_beyond_the_range_of_fp32_pairs(scale):
    """Inf above fp32, and below 2^-100, where products of fp32 numbers lose their low parts, the fp64
    value rounded, denormal ones included (one unit in the last place: the order of the fp64 sums)."""
    rng = np.random.default_rng(3)
    T = (scale * rng.standard_normal((500, D))).astype(np.float32)
    err, want = _tail_errs(T, [], _blocks(rng, 1)[0])
    assert np.isinf(want).all() == (scale == 1e20) and not np.isnan(err).any()
    ok = np.abs(err.view(np.int32).astype(np.int64) - want.view(np.int32)) <= 1
    assert ok.all(), (err[~ok][:4], want[~ok][:4])


def test_errs_of_a_residual_that_is_the_rounding_of_its_terms():
    """t - c0 - c1 with t = c1 = 1 and a tiny c0: the fp32 residual is 0, the exact one -c0."""
    rng = np.random.default_rng(4)
    c0 = (1e-9 * rng.standard_normal(D)).astype(np.float32)
    one = np.ones(D, np.float32)
    err, want = _tail_errs(np.ones((5, D), np.float32), [c0, one], _blocks(rng, 1)[0])
    assert want.min() > 0
    np.testing.assert_allclose(err, want, rtol=1e-6)  # c0's part in fp32 pairs: 2^-24 of it each


def test_non_finite_codeword_and_target_are_reported_and_leave_the_rest():
    rng = np.random.default_rng(5)
    M, G, K = 200, 2, 100
    W = (0.02 * rng.standard_normal((M, G * D))).astype(np.float32)
    C = (0.02 * rng.standard_normal((K, D))).astype(np.float32)
    Hb = _blocks(rng, G)
    good, _ = _encode(W, Hb, C)
    W[7, 3] = np.nan
    codes = torch.zeros((M, G), dtype=torch.int32, device="cuda")
    P.crvq_encode_beam(dev(W), D, dev(Hb), [Codebook(dev(C), codes, G)], 0, 1)
    with pytest.raises(P.CrvqError) as e:
        P.crvq_sync()
    assert e.value.status == -6
    rest = np.arange(M) != 7
    np.testing.assert_array_equal(host(codes)[rest], good[rest])
