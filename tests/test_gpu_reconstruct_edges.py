"""Reconstruction of matrices large enough that the slices without extended codebooks run in a launch
of their own, and that a block takes several row blocks, against plain fp64 sums: reconstructions are
bit-exact, block losses within 1e-4 (the bar of the parity tests: fp32 terms). Sums that leave fp32's
range, for good or on the way, are those of fp64 rounded."""
import numpy as np
import pytest
import torch

import paper_2412_09282_gb300 as P
from paper_2412_09282_gb300 import Codebook
from parity_util import dev, host

pytestmark = pytest.mark.gpu

D = 8


@pytest.mark.parametrize("M,N,Gc", [(2600, 8192, 33), (5001, 4616, 5), (17, 9224, 2)])
def test_reconstruct_over_row_blocks_and_slices(M, N, Gc):
    rng = np.random.default_rng(M + N)
    G = N // D
    W = (0.02 * rng.standard_normal((M, N))).astype(np.float32)
    A = rng.standard_normal((G, 12, D))
    Hb = (A.transpose(0, 2, 1) @ A / 12 + 0.05 * np.eye(D)).astype(np.float32)
    perm = rng.permutation(N).astype(np.int32)
    Cs = [(0.02 * rng.standard_normal((k, D))).astype(np.float32) for k in (256, 16, 9)]
    codes = [rng.integers(0, k, (M, g)).astype(np.int32) for k, g in ((256, G), (16, Gc), (9, Gc))]
    cbs = [Codebook(dev(C), dev(c), c.shape[1]) for C, c in zip(Cs, codes)]
    Wh, lb, lc, lf = P.crvq_reconstruct_error(dev(W), D, dev(Hb), dev(perm), cbs, Gc)
    rec = Cs[0][codes[0]].astype(np.float64)
    for C, c in zip(Cs[1:], codes[1:]):
        rec[:, :Gc] += C[c]
    rec = rec.astype(np.float32).reshape(M, N)
    want = np.empty_like(rec)
    want[:, perm] = rec
    assert lf is None
    np.testing.assert_array_equal(host(Wh), want)
    d = (W - rec).astype(np.float64).reshape(M, G, D)
    per_group = np.einsum("mgi,gij,mgj->g", d, Hb.astype(np.float64), d, optimize=True)
    assert abs(lb - per_group.sum()) <= 1e-4 * per_group.sum()
    assert abs(lc - per_group[:Gc].sum()) <= 1e-4 * per_group[:Gc].sum()


def test_reconstruct_with_several_row_blocks_per_block():
    """158 row groups of 33 slices, more than sixteen blocks per SM: a block takes three or four row
    groups, the last ones ragged. Against fp64 on the device."""
    M, N, Gc = 20011, 8200, 40
    G = N // D
    g = torch.Generator(device="cuda").manual_seed(1)
    W = 0.02 * torch.randn((M, N), generator=g, device="cuda")
    A = torch.randn((G, 12, D), generator=g, device="cuda")
    Hb = (A.transpose(1, 2) @ A / 12 + 0.05 * torch.eye(D, device="cuda")).contiguous()
    perm = torch.randperm(N, generator=g, device="cuda").to(torch.int32)
    cbs = [Codebook(0.02 * torch.randn((k, D), generator=g, device="cuda"),
                    torch.randint(0, k, (M, c), generator=g, device="cuda", dtype=torch.int32), c)
           for k, c in ((256, G), (16, Gc), (9, Gc))]
    Wh, lb, lc, _ = P.crvq_reconstruct_error(W, D, Hb, perm, cbs, Gc)
    rec = cbs[0].C.double()[cbs[0].codes.long()]
    for cb in cbs[1:]:
        rec[:, :Gc] += cb.C.double()[cb.codes.long()]
    rec = rec.float().view(M, N)
    assert torch.equal(Wh[:, perm.long()], rec)
    d = (W - rec).double().view(M, G, D)
    per_group = torch.stack([((d[:, i] @ Hb[i].double()) * d[:, i]).sum() for i in range(G)])
    assert abs(lb - float(per_group.sum())) <= 1e-4 * float(per_group.sum())
    assert abs(lc - float(per_group[:Gc].sum())) <= 1e-4 * float(per_group[:Gc].sum())


@pytest.mark.parametrize("n_cb", [3, 6])
def test_reconstruct_sums_beyond_fp32(n_cb):
    """An infinite codeword gives an infinite element, and large terms of both signs their sum, whatever
    the partial sums did."""
    M, N = 40, 16
    G = N // D
    rng = np.random.default_rng(n_cb)
    Cs = [(0.02 * rng.standard_normal((4, D))).astype(np.float32) for _ in range(n_cb)]
    Cs[0][0, 3], Cs[1][1, 5] = np.inf, -np.inf
    for C, v in zip(Cs, (3e38, 3e38, -3e38)):
        C[2, 1] = v
        C[3, 6] = -v
    codes = [rng.integers(0, 2 if s < 3 else 4, (M, G)).astype(np.int32) for s in range(n_cb)]
    for c in codes[:3]:
        c[:10] = 2
        c[10:20] = 3
    codes[1][(codes[0] == 0) & (codes[1] == 1)] = 0
    cbs = [Codebook(dev(C), dev(c), G) for C, c in zip(Cs, codes)]
    W = np.zeros((M, N), np.float32)
    Hb = np.stack([np.eye(D, dtype=np.float32)] * G)
    Wh, _, _, _ = P.crvq_reconstruct_error(dev(W), D, dev(Hb), None, cbs, 0)
    rec = sum(C.astype(np.float64)[c] for C, c in zip(Cs, codes))
    with np.errstate(over="ignore"):
        want = rec.astype(np.float32).reshape(M, N)
    assert np.isinf(want).any() and not np.isnan(want).any() and (np.abs(want) > 1e38).any()
    np.testing.assert_array_equal(host(Wh), want)
