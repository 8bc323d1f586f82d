"""grass_compress by its forms of launch (a block per row, stored four at a time or one by one; a cluster per row; many blocks): remainders of rows and
masks, several draws, no mask, and what rows that rule out 16-byte stores cost."""
import pytest
import torch

import paper_2505_18976_b200 as G

pytestmark = pytest.mark.gpu


def _check(n, p, kprime, k, s, off, pad, dtype, out_dtype):
    gen = torch.Generator("cuda").manual_seed(k + n)
    g = torch.randn((n, p), generator=gen, device="cuda").to(dtype)
    idx = G.mask_to_device(G.grass_random_mask_host(p, kprime, 3)) if kprime else None
    wide = torch.full((n, off + k + pad), 7.0, device="cuda", dtype=out_dtype)
    out = G.grass_compress(g, idx, k, s, 99, out=wide[:, off:off + k]).double()
    assert (wide[:, :off] == 7.0).all() and (wide[:, off + k:] == 7.0).all()
    x = (g[:, idx.long()] if kprime else g).double().repeat_interleave(s, 1) / s ** 0.5
    bucket, sign = G.grass_sjlt_table(k, s, 99, x.shape[1] // s)
    ref = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x * sign.double())
    absum = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x.abs())
    # at most `load` additions in any order, each off by 2^-24 of a partial sum; the scale and its product off by 2^-24 each
    load = int(torch.bincount(bucket.long(), minlength=k).max())
    tol = (load + (2 if s > 1 else 0)) * 2.0 ** -24 * absum
    if out_dtype == torch.bfloat16:
        tol = tol + 2.0 ** -8 * (ref.abs() + tol)
    assert ((out - ref).abs() <= tol).all()


# n, p, k', k, s, off, pad: whole rows by 256, 512 and 1,024 threads, one past a round, of every position, bins at the limit of shared
# memory and of a length off four; off = 4, pad = 4: 16-byte stores between columns that are not theirs; clusters of 2 to 8
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("out_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,p,kprime,k,s,off,pad", [
    (160, 20_000, 2_047, 512, 1, 4, 4), (160, 20_000, 2_049, 1_024, 2, 4, 4), (160, 20_000, 4_097, 16_384, 1, 0, 1), (160, 20_000, 8_192, 16_384, 1, 4, 4),
    (150, 20_000, 8_191, 51_199, 1, 0, 0), (150, 20_000, 8_191, 51_200, 3, 0, 0), (149, 20_000, 1, 4, 1, 4, 4), (160, 3_001, 0, 1_000, 1, 4, 4),
    (160, 20_000, 8_193, 1_001, 1, 1, 2), (700, 20_000, 12_289, 2_048, 1, 4, 4), (1, 20_000, 8_192, 2_048, 2, 3, 0), (5, 70_000, 8_195, 1_001, 1, 4, 4), (40, 90_000, 44_531, 3_000, 1, 4, 4)])
def test_forms(n, p, kprime, k, s, off, pad, dtype, out_dtype):
    _check(n, p, kprime, k, s, off, pad, dtype, out_dtype)


def _time(pad, k, g, idx):
    outs = [torch.empty((g[0].shape[0], k + pad), device="cuda")[:, :k] for _ in g]
    times = []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for i in range(32):
            G.grass_compress(g[i % len(g)], idx, k, 1, 99, out=outs[i % len(g)])
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return min(times)


# A row of odd stride is stored by lanes on consecutive elements.  (Lanes four elements apart, as they once were: 22 and 49 % slower than
# rows that take 16-byte stores, where this is 3 and 7 %.)
@pytest.mark.parametrize("k", [16_384, 40_000])
def test_cost_of_rows_off_a_boundary(k):
    g = [torch.randn((256, 65_536), device="cuda") for _ in range(5)]
    idx = G.mask_to_device(G.grass_random_mask_host(65_536, 8_192, 3))
    _time(0, k, g, idx)
    assert _time(1, k, g, idx) < 1.15 * _time(0, k, g, idx)


# few rows under long masks: more blocks than a cluster has, adding into a zeroed row (fp32 only: a bf16 row is rounded once)
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,p,kprime,k,s,off,pad", [(2, 300_001, 209_525, 752, 1, 3, 1), (7, 200_000, 131_073, 2_267, 1, 4, 4), (3, 150_000, 0, 3_000, 2, 0, 1)])
def test_wide_splits(n, p, kprime, k, s, off, pad, dtype):
    _check(n, p, kprime, k, s, off, pad, dtype, torch.float32)
