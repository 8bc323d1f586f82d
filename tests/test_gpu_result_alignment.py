"""Results stored four at a time where their place allows it: grass_fim with whole tiles of one thread block, and FactGraSS clusters whose
result begins off a 16-byte (fp32) or 8-byte (bf16) boundary."""
import pytest
import torch

import paper_2505_18976_b200 as G

pytestmark = pytest.mark.gpu


# one thread block per tile: few samples, or more tiles than two per SM
@pytest.mark.parametrize("n,k,off,pad", [(200, 900, 0, 0), (200, 900, 4, 4), (200, 901, 0, 0), (300, 2_304, 0, 0), (300, 2_304, 0, 1), (300, 2_306, 1, 1)])
def test_fim_whole_tiles(n, k, off, pad):
    gen = torch.Generator("cuda").manual_seed(n + k)
    X = torch.randn((n, k), generator=gen, device="cuda")
    wide = torch.full((k, off + k + pad), 7.0, device="cuda")
    F = G.grass_fim(X, out=wide[:, off:off + k]).double()
    assert (wide[:, :off] == 7.0).all() and (wide[:, off + k:] == 7.0).all()
    Xd = X.double()
    ref, absum = Xd.T @ Xd / n, Xd.abs().T @ Xd.abs() / n
    # six bf16 products keep each product to 2^-23; accumulators are truncated once per 16 samples
    assert ((F - ref).abs() <= 2.0 ** -22 * absum + 2.0 * (n / 16 + 64) ** 0.5 * 2.0 ** -23 * absum).all()


# k whose slices are whole groups of four and k whose are not; an odd base, an odd row stride, neither
@pytest.mark.parametrize("out_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("k,off,pad", [(1_024, 0, 0), (1_024, 1, 3), (1_024, 2, 2), (1_024, 4, 4), (1_024, 4, 1), (1_026, 1, 1), (64, 3, 1)])
def test_factgrass_cluster_result_anywhere(k, off, pad, out_dtype):
    B, T, d_in, d_out = 3, 96, 200, 300
    gen = torch.Generator("cuda").manual_seed(k)
    A = torch.randn((B, T, d_in), generator=gen, device="cuda").to(torch.bfloat16)
    D = torch.randn((B, T, d_out), generator=gen, device="cuda").to(torch.bfloat16)
    mi, mo = (G.mask_to_device(G.grass_random_mask_host(d, m, d)) for d, m in ((d_in, 64), (d_out, 48)))
    wide = torch.full((B, off + k + pad), 7.0, device="cuda", dtype=out_dtype)
    layers = G.GroupedLayers([dict(A=A, G=D, mask_in=mi, mask_out=mo, k=k, s=1, seed=99, out_offset=0)])
    ws = torch.empty(G.factgrass_grouped_workspace_bytes(1), dtype=torch.uint8, device="cuda")
    with G.tuning(factgrass_path=1):
        out = G.factgrass_compress_grouped(layers, wide[:, off:off + k], ws).double()
    assert (wide[:, :off] == 7.0).all() and (wide[:, off + k:] == 7.0).all()
    a, d = A[:, :, mi.long()].double(), D[:, :, mo.long()].double()
    bucket, sign = G.grass_sjlt_table(k, 1, 99, a.shape[2] * d.shape[2])

    def project(x, signs):
        return torch.zeros((B, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x.reshape(B, -1) * signs)

    ref, absum = project(a.transpose(1, 2) @ d, sign.double()), project(a.abs().transpose(1, 2) @ d.abs(), 1.0)
    # products of bf16 are exact in fp32; T of them and then `load` blocks are added, each addition off by at most 2^-23 of a partial sum
    load = int(torch.bincount(bucket.long(), minlength=k).max())
    tol = (T + load + 8) * 2.0 ** -23 * absum
    if out_dtype == torch.bfloat16:
        tol = tol + 2.0 ** -8 * (ref.abs() + tol)
    assert ((out - ref).abs() <= tol).all()
