"""grass_compress where its shared memory is at the 48 KB that a launch has without asking for more.  The limit, once raised, stays raised
for a kernel, so the calls are the first of a process of their own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALLS = """
import sys
import torch
import paper_2505_18976_b200 as G

n, p, kprime, k = map(int, sys.argv[1:])
gen = torch.Generator("cuda").manual_seed(k)
g = torch.randn((n, p), generator=gen, device="cuda")
idx = G.mask_to_device(G.grass_random_mask_host(p, kprime, 3)) if kprime else None
out = G.grass_compress(g, idx, k, 1, 99).double()
x = (g[:, idx.long()] if kprime else g).double()
bucket, sign = G.grass_sjlt_table(k, 1, 99, x.shape[1])
ref = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x * sign.double())
absum = torch.zeros((n, k), device="cuda", dtype=torch.float64).index_add_(1, bucket.long(), x.abs())
load = int(torch.bincount(bucket.long(), minlength=k).max())
assert ((out - ref).abs() <= load * 2.0 ** -24 * absum).all()      # at most `load` additions, each off by 2^-24 of a partial sum
"""


# bins alone (k = 12,288), bins and index list (4,096 and 8,192 entries), bins of two rows and the queues (2 x 5,376)
@pytest.mark.parametrize("n,p,kprime,k", [(5, 20_000, 8_192, 12_288), (160, 20_000, 8_192, 4_096), (64, 8_192, 0, 5_376)])
def test_first_call_at_the_limit(n, p, kprime, k):
    r = subprocess.run([sys.executable, "-c", CALLS, str(n), str(p), str(kprime), str(k)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
