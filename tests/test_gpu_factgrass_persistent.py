"""GPU parity of the persistent FactGraSS kernel against the CPU oracle, where its shares of work can go wrong: remainders of
a 32-token step and of the 128 x 128 block, samples cut between thread blocks, samples without tokens, accumulators of more
than 8,192 tokens.  Tolerance: the rule of parity.py, with the longest chain of additions as in the other FactGraSS tests."""
import numpy as np
import pytest
import torch

from parity import check_close, max_bin_load

pytestmark = pytest.mark.gpu

# d_in, d_out, kin, kout, k
LAYERS = [(300, 200, 128, 128, 4096), (96, 160, 65, 100, 97), (129, 128, 1, 128, 14_336), (64, 500, 33, 7, 300)]


def _compare(layers, dtype, B, T, lens, path):
    import oracle
    import paper_2505_18976_b200 as G
    from paper_2505_18976_b200 import workloads as W
    lengths = np.full(B, T, dtype=np.int32) if lens is None else np.array(lens, dtype=np.int32)
    begin = (np.cumsum(lengths) - lengths).astype(np.int64)
    rows = int(lengths.sum())
    name = "f32" if dtype == torch.float32 else "bf16"
    dicts, keep, off = [], [], 0
    for n, (d_in, d_out, kin, kout, k) in enumerate(layers):
        gen = torch.Generator(device="cuda").manual_seed(n)
        A = torch.randn((rows, d_in), device="cuda", generator=gen).to(dtype)
        Gr = torch.randn((rows, d_out), device="cuda", generator=gen).to(dtype)
        mi, mo = oracle.random_mask(d_in, kin, n + 1), oracle.random_mask(d_out, kout, n + 20)
        shape = (lambda t, d: t) if lens is not None else (lambda t, d: t.view(B, T, d))
        dicts.append(dict(A=shape(A, d_in), G=shape(Gr, d_out), mask_in=G.mask_to_device(mi), mask_out=G.mask_to_device(mo), k=k,
                          s=1, seed=n + 5, out_offset=off))
        keep.append((A, Gr, mi, mo, kin, kout, k, off))
        off += k
    out = torch.full((B, off), float("nan"), device="cuda")
    ws = torch.full((G.factgrass_grouped_workspace_bytes(len(layers)),), 0xA5, dtype=torch.uint8, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    with G.tuning(factgrass_path=path):
        if lens is None:
            G.factgrass_compress_grouped(G.GroupedLayers(dicts), out, ws, dev_status=st)
        else:
            G.factgrass_compress_grouped_varlen(G.GroupedLayers(dicts), out, ws, B, T, tok_begin=torch.tensor(begin).cuda(),
                                                tok_count=torch.tensor(lengths).cuda(), dev_status=st)
        torch.cuda.synchronize()
    assert int(st.item()) == 0
    # this kernel, and no other, writes the tables of the projections: 128 x 128 entries of 16 bits per layer, behind the descriptors
    tables = ws[ws.numel() - len(layers) * 2 * 128 * 128:].view(len(layers), -1)
    assert (tables != 0xA5).any(dim=1).all(), "another kernel took the call"
    host = out.cpu().numpy()
    for n, (A, Gr, mi, mo, kin, kout, k, o) in enumerate(keep):
        ref, absum = oracle.factgrass_varlen(W.bits_of(A), W.bits_of(Gr), mi, mo, k, 1, n + 5, begin, lengths, dtype=name)
        ob, _ = oracle.sjlt_table(k, 1, n + 5, kin * kout)
        check_close(host[:, o:o + k], ref, absum, 1e-4 if name == "f32" else 2e-2, int(lengths.max()) + max_bin_load(ob, k) + 64,
                    eps=2.0 ** -23, what=f"layer {n} {name} B={B} T={T}")


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("layers,B,T,lens,path", [
    (LAYERS, 1, 1, None, 2),                                     # fewer steps than SMs
    (LAYERS, 3, 33, None, 2),
    (LAYERS, 9, 300, None, 2),                                   # shares that end inside samples, several samples per share
    (LAYERS[:1], 5, 1024, None, 2),                              # 32 steps a sample in even shares
    (LAYERS[:2], 7, 500, [500, 0, 1, 32, 33, 499, 64], 2),
    (LAYERS, 40, 33, None, None),                                # by its own rule: an item for every SM
    (LAYERS[:2], 90, 64, list(range(64, 1, -1)) + [0] * 27, None),
    ([(8, 8, 3, 2, 7)], 4, 310_000, None, 2),                    # more than 8,192 tokens for one thread block
])
def test_persistent(layers, B, T, lens, path, dtype):
    _compare(layers, dtype, B, T, lens, path)
