"""Plain SJLT through the table of the projection (grass_compress_ws) against the dense projection matrix."""
import pytest
import torch

import paper_2505_18976_b200 as G

pytestmark = pytest.mark.gpu


# p: below one group of 128, one chunk, a chunk and one position, several chunks; n: a single row, an odd last one, rows
# shared by two blocks, more rows than blocks; k: copies of few bins, one and two rows per unit, the largest bucket; rows
# that start off a 16-byte boundary
@pytest.mark.parametrize("n,p,k,off,ld,dtype,out_dtype", [
    (1, 1, 1, 0, 1, torch.float32, torch.float32), (3, 5, 7, 0, 5, torch.bfloat16, torch.float32),
    (5, 127, 600, 0, 127, torch.float32, torch.float32), (2, 6_400, 4_096, 0, 6_400, torch.float32, torch.float32),
    (7, 6_401, 2_048, 1, 6_404, torch.float32, torch.float32), (301, 7_937, 1_024, 0, 7_937, torch.bfloat16, torch.float32),
    (33, 40_003, 1_361, 3, 40_011, torch.bfloat16, torch.bfloat16), (9, 20_000, 16_384, 0, 20_000, torch.float32, torch.float32),
    (4, 9_999, 32_768, 2, 10_003, torch.float32, torch.bfloat16), (149, 30_000, 100, 0, 30_000, torch.float32, torch.float32)])
def test_table_parity(tune, n, p, k, off, ld, dtype, out_dtype):
    gen = torch.Generator("cuda").manual_seed(n + p)
    wide = torch.full((n, ld + off), float("nan"), device="cuda", dtype=dtype)
    g = wide[:, off:off + p]
    x = torch.randn((n, p), generator=gen, device="cuda")
    g.copy_(x * (torch.rand((n, p), generator=gen, device="cuda") < 0.4))
    tune(compress_dense=2)
    out = G.grass_compress(g, None, k, 1, 99, out=torch.full((n, k), 3.0, device="cuda", dtype=out_dtype)).double()
    bucket, sign = G.grass_sjlt_table(k, 1, 99, p)
    gd = g.double()
    ref = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), gd * sign.double())
    absum = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), gd.abs())
    # a sum of at most `load` fp32 terms, every addition rounds by 2^-24 of a partial sum; bf16 rows are rounded once more
    load = int(torch.bincount(bucket.long(), minlength=k).max())
    tol = 2.0 * load ** 0.5 * 2.0 ** -24 * absum + 2.0 ** -24 * ref.abs()
    if out_dtype == torch.bfloat16:
        tol = tol + 2.0 ** -8 * ref.abs()
    assert ((out - ref).abs() <= tol).all()
    assert (out[absum == 0] == 0).all()


def test_non_finite_values_propagate(tune):
    g = torch.zeros((3, 9_000), device="cuda")
    g[1, 4_000], g[2, 8_999] = float("inf"), float("nan")
    tune(compress_dense=2)
    out = G.grass_compress(g, None, 512, 1, 5)
    assert (out[0] == 0).all() and torch.isinf(out[1]).sum() == 1 and torch.isnan(out[2]).sum() == 1
    assert torch.isfinite(out).sum() == 3 * 512 - 2
