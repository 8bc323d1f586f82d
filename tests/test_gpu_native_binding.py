"""The compiled marshalling of the binding against the ctypes code it stands in for: same results, same exceptions,
and no verdict of its own on operands that are out of the ordinary."""
import ctypes

import pytest
import torch

import paper_2505_18976_b200 as G
from paper_2505_18976_b200 import binding as B

pytestmark = pytest.mark.gpu


class _Declines:
    """A stand-in for the extension that leaves every call to the ctypes code."""

    def __getattr__(self, name):
        return lambda *a: None


def _calls(n=5, p=300, k=64, T=40):
    gen = torch.Generator("cuda").manual_seed(7)
    r = lambda *s: torch.randn(s, generator=gen, device="cuda")       # noqa: E731
    idx = G.mask_to_device(G.grass_random_mask_host(p, 37, 1))
    mi, mo = (G.mask_to_device(G.grass_random_mask_host(48, 16, s)) for s in (2, 3))
    A, Gr = r(n, T, 48).bfloat16(), r(n, T, 48).bfloat16()
    g = r(n, p)
    count = torch.tensor([T, 0, 3, T - 1, 7], dtype=torch.int32, device="cuda")
    layers = [dict(A=A, G=Gr, mask_in=mi, mask_out=mo, k=k, s=1, seed=5 + l, out_offset=l * k) for l in range(3)]
    ws = torch.empty(G.factgrass_grouped_workspace_bytes(3), dtype=torch.uint8, device="cuda")
    out = lambda: torch.full((n, 3 * k), float("nan"), device="cuda")  # noqa: E731
    tr, te = r(9, 64), r(5, 64)
    return {
        "mask": lambda: G.grass_compress(g, idx, k, 1, 9),
        "identity": lambda: G.grass_compress(g[:, :296], None, k, 2, (1 << 64) + 9),
        "p": lambda: G.grass_compress(g, G.mask_to_device(G.grass_random_mask_host(200, 37, 1)), k, 1, 9, p=200),
        "bf16_out": lambda: G.grass_compress(g, idx, k, 1, 9, out_dtype=torch.bfloat16),
        "one_row_out": lambda: G.grass_compress(g[:1], idx, k, 1, 9, out=torch.empty((1, k), device="cuda")),
        "layer": lambda: G.factgrass_compress(A, Gr, mi, mo, k, 1, 9),
        "varlen": lambda: G.factgrass_compress_varlen(A, Gr, mi, mo, k, 1, 9, n, T, None, count),
        "grouped": lambda: G.factgrass_compress_grouped(G.GroupedLayers(layers), out(), ws),
        "grouped_varlen": lambda: G.factgrass_compress_grouped_varlen(G.GroupedLayers(layers), out(), ws, n, T, None, count),
        "score": lambda: G.grass_score(tr, te),
        "score_bf16": lambda: G.grass_score_bf16(tr.bfloat16(), te.bfloat16()),
    }


@pytest.mark.parametrize("name", ["mask", "identity", "p", "bf16_out", "one_row_out", "layer", "varlen", "grouped",
                                  "grouped_varlen", "score", "score_bf16"])
def test_same_as_ctypes(name, monkeypatch):
    call = _calls()[name]
    fast = call()
    monkeypatch.setattr(B, "_fast", lambda: _Declines())
    slow = call()
    # the order of floating-point atomics is free: a bin of at most a few dozen fp32 terms, a few ulps
    assert fast.dtype == slow.dtype and fast.shape == slow.shape
    tol = 2.0 ** -7 if fast.dtype == torch.bfloat16 else 1e-5
    assert torch.allclose(fast.float(), slow.float(), rtol=tol, atol=tol)


def test_errors_come_from_the_same_place():
    g = torch.zeros((4, 64), device="cuda")
    idx = G.mask_to_device(G.grass_random_mask_host(64, 8, 1))
    with pytest.raises(G.GrassError) as e:
        G.grass_compress(g, idx, 0, 1, 0)                      # k == 0: the library's verdict
    assert e.value.code == 1
    with pytest.raises(TypeError):
        G.grass_compress(g, idx.to(torch.int64), 16, 1, 0)     # index list of the wrong width
    with pytest.raises(ValueError):
        G.grass_compress(g.cpu(), idx, 16, 1, 0)               # pageable host memory
    with pytest.raises(TypeError):
        G.grass_compress(g.double(), idx, 16, 1, 0)
    with pytest.raises(AssertionError):
        G.grass_score(g, torch.zeros((4, 32), device="cuda"))  # different contraction lengths
    layers = [dict(A=g.view(2, 2, 64), G=g.view(2, 2, 64), mask_in=idx, mask_out=idx, k=8, s=1, seed=0, out_offset=-1)]
    with pytest.raises(ValueError):
        G.GroupedLayers(layers)


@pytest.fixture
def no_more_memory():
    """Call it, and the allocator gives out nothing that it does not hold already."""
    def close():
        torch.cuda.empty_cache()
        torch.cuda.set_per_process_memory_fraction(0.0)
    yield close
    torch.cuda.set_per_process_memory_fraction(1.0)


def test_out_of_memory_is_torchs_exception(no_more_memory):
    g, x = torch.zeros((1 << 16, 8), device="cuda"), torch.zeros((1 << 13, 8), device="cuda")
    A = torch.zeros((1 << 15, 1, 8), device="cuda")
    m = G.mask_to_device(G.grass_random_mask_host(8, 4, 1))
    no_more_memory()
    for call in (lambda: G.grass_compress(g, None, 4_096, 1, 0), lambda: G.factgrass_compress(A, A, m, m, 8_192, 1, 0),
                 lambda: G.grass_score(g, x)):
        with pytest.raises(torch.OutOfMemoryError):
            call()


def test_calls_do_without_the_scratch_that_they_cannot_have(no_more_memory):
    """Plain SJLT of a batch wants a table of 2 bytes per position; with `out` given it needs no memory at all."""
    n, p, k = 32, 1 << 24, 256
    g = torch.zeros((n, p), device="cuda")
    g[:, ::4_097] = 1.0
    want, out = G.grass_compress(g, None, k, 1, 0), torch.empty((n, k), device="cuda")
    no_more_memory()
    assert G.grass_compress(g, None, k, 1, 0, out=out) is out
    assert torch.equal(out, want)      # sums of ones, exact in any order


@pytest.mark.parametrize("n,T", [(150, 40), (40, 500)])
def test_single_fp32_layers_get_the_table_where_the_library_would_use_it(n, T, monkeypatch):
    """An item for every SM, and steps for every SM; against the ctypes code, which hands over no scratch."""
    gen = torch.Generator("cuda").manual_seed(2)
    A, Gr = (torch.randn((n, T, d), generator=gen, device="cuda") for d in (200, 150))
    mi, mo = (G.mask_to_device(G.grass_random_mask_host(d, 100, s)) for d, s in ((200, 2), (150, 3)))
    spec = B.SjltSpec(4_096, 1, 9)
    scratch = lambda rows: G.lib().factgrass_compress_workspace_bytes(B.F32, rows, T, 100, 100, ctypes.byref(spec))  # noqa: E731
    assert scratch(n) > 0 and scratch(4) == 0
    fast = G.factgrass_compress(A, Gr, mi, mo, 4_096, 1, 9)
    monkeypatch.setattr(B, "_fast", lambda: _Declines())
    slow = G.factgrass_compress(A, Gr, mi, mo, 4_096, 1, 9)
    # sums of T products of two unit normals, 10,000 / 4,096 of them per bin, in two orders of fp32 additions
    assert (fast - slow).abs().max() <= 64 * 2.0 ** -24 * T ** 0.5 * float(slow.abs().max())
