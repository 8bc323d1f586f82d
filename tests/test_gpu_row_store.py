"""Bins emptied and rows stored four at a time: row lengths, strides and alignments that allow it and that do not."""
import pytest
import torch

import paper_2505_18976_b200 as G

pytestmark = pytest.mark.gpu


# n: a thread block per row (160), a cluster per row (5); k: below, at and off a multiple of four; off, pad: a result that begins off a
# 16-byte boundary or whose rows do
@pytest.mark.parametrize("out_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,k,off,pad", [(160, 3, 0, 1), (160, 4, 0, 0), (160, 2_048, 0, 0), (160, 2_050, 0, 2), (160, 1_024, 2, 6),
                                         (160, 1_024, 4, 3), (5, 2_048, 0, 4), (5, 1_023, 1, 0)])
def test_rows_of_any_length_and_alignment(n, k, off, pad, out_dtype):
    p, kprime = 20_000, 8_192
    gen = torch.Generator("cuda").manual_seed(k + n)
    g = torch.randn((n, p), generator=gen, device="cuda")
    idx = G.mask_to_device(G.grass_random_mask_host(p, kprime, 3))
    wide = torch.full((n, off + k + pad), 7.0, device="cuda", dtype=out_dtype)
    out = G.grass_compress(g, idx, k, 1, 99, out=wide[:, off:off + k]).double()
    assert (wide[:, :off] == 7.0).all() and (wide[:, off + k:] == 7.0).all()
    bucket, sign = G.grass_sjlt_table(k, 1, 99, kprime)
    x = g[:, idx.long()].double()
    ref = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x * sign.double())
    absum = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x.abs())
    # sums of at most `load` fp32 terms, each addition off by 2^-24 of a partial sum; bf16 rounds once more
    load = int(torch.bincount(bucket.long(), minlength=k).max())
    tol = 2.0 * load ** 0.5 * 2.0 ** -24 * absum + 2.0 ** -24 * ref.abs()
    if out_dtype == torch.bfloat16:
        tol = tol + 2.0 ** -8 * ref.abs()
    assert ((out - ref).abs() <= tol).all()


# grass_fim stores four entries at a time in whole tiles off the diagonal: tiles at the edge, few tiles and many (added up by several
# clusters), rows that begin off a 16-byte boundary
@pytest.mark.parametrize("n,k,pad", [(300, 256, 0), (300, 256, 1), (300, 257, 3), (5_000, 1_024, 0), (5_000, 1_024, 2), (5_000, 900, 4)])
def test_fim_rows_of_any_alignment(n, k, pad):
    gen = torch.Generator("cuda").manual_seed(n + k)
    X = torch.randn((n, k), generator=gen, device="cuda")
    wide = torch.full((k, k + pad), 7.0, device="cuda")
    F = G.grass_fim(X, out=wide[:, :k]).double()
    assert (wide[:, k:] == 7.0).all()
    Xd = X.double()
    ref, absum = Xd.T @ Xd / n, Xd.abs().T @ Xd.abs() / n
    # six bf16 products keep each product to 2^-23; accumulators are truncated once per 16 samples
    assert ((F - ref).abs() <= 2.0 ** -22 * absum + 2.0 * (n / 16 + 64) ** 0.5 * 2.0 ** -23 * absum).all()
