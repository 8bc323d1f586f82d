"""Kernels that start while the kernel before them still runs: what that one writes is read complete, and what it reads is not
overwritten; on a stream, and recorded into a graph behind every kind of node."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import paper_2505_18976_b200 as g
    g.lib()
    return g


def _calls(G):
    """Each writes its input, runs a call on it and returns the result; the second argument counts up."""
    g = torch.randn((64, 65_536), device="cuda")
    idx = G.mask_to_device(G.grass_random_mask_host(65_536, 8_192, 3))
    few = G.mask_to_device(G.grass_random_mask_host(65_536, 1_024, 4))
    A = torch.randn((4, 96, 200), device="cuda").to(torch.bfloat16)
    Gr = torch.randn((4, 96, 300), device="cuda").to(torch.bfloat16)
    wide_g = torch.randn((2, 600_001), device="cuda")
    wide_idx = G.mask_to_device(G.grass_random_mask_host(600_001, 110_000, 6))
    mi, mo = (G.mask_to_device(G.grass_random_mask_host(d, 64, d)) for d in (200, 300))

    def clusters():
        g.neg_()
        return G.grass_compress(g[:3], idx, 2_048, 1, 5)

    def rows():
        g.neg_()
        return G.grass_compress(g, few, 512, 1, 5)

    def wide():                # zeroed by a memset, then added into by more blocks than a cluster has
        wide_g.neg_()
        return G.grass_compress(wide_g, wide_idx, 1_024, 1, 5)

    def dense():
        g.neg_()
        return G.grass_compress(g[:4], None, 2_048, 1, 5)

    def layer():
        A.neg_()
        return G.factgrass_compress(A, Gr, mi, mo, 1_024, 1, 5)

    train, test = torch.randn((300, 520), device="cuda"), torch.randn((40, 520), device="cuda")

    def score():
        train.neg_()
        return G.grass_score(train, test)

    def score_bf16():
        train.neg_()
        return G.grass_score_bf16(train.to(torch.bfloat16), test.to(torch.bfloat16))

    return dict(clusters=clusters, rows=rows, wide=wide, dense=dense, layer=layer, score=score, score_bf16=score_bf16)


# sums in another order: at most some tens of fp32 additions per value
def _same(a, b):
    return (a - b).abs().max() <= 2.0 ** -18 * b.abs().max()


@pytest.mark.parametrize("name", ["clusters", "rows", "wide", "dense", "layer", "score", "score_bf16"])
def test_chained_calls_read_finished_inputs(G, name):
    call = _calls(G)[name]
    outs = [call() for _ in range(60)]
    torch.cuda.synchronize()
    for i, o in enumerate(outs):
        assert _same(o if i % 2 == 0 else -o, outs[0]), i


@pytest.mark.parametrize("before", ["nothing", "kernel", "copy", "download", "fill", "join", "call"])
def test_recorded_behind_any_node(G, before):
    g = torch.randn((64, 65_536), device="cuda")
    idx = G.mask_to_device(G.grass_random_mask_host(65_536, 8_192, 3))
    ref = G.grass_compress(g, idx, 2_048, 1, 5)
    x, y, host = torch.zeros(1_000, device="cuda"), torch.empty(1_000, device="cuda"), torch.empty(1_000).pin_memory()
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        if before == "kernel":
            x.add_(1)
        elif before == "copy":
            y.copy_(x)
        elif before == "download":
            host.copy_(x, non_blocking=True)
        elif before == "fill":
            x.zero_()
        elif before == "join":
            side.wait_stream(main)
            with torch.cuda.stream(side):
                x.add_(1)
            y.add_(1)
            main.wait_stream(side)
        elif before == "call":
            G.grass_compress(g, idx, 2_048, 1, 5)
        out = G.grass_compress(g, idx, 2_048, 1, 5)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert _same(out, ref)


@pytest.mark.parametrize("name", ["clusters", "wide", "dense", "layer", "score", "score_bf16"])
def test_recorded_calls(G, name):
    call = _calls(G)[name]
    ref = call()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        outs = [call(), call()]
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert _same(outs[1], ref) and _same(-outs[0], ref)


# calls that take tensor memory, on two streams at once: clusters of the layer's blocks beside pairs of the score's
@pytest.mark.parametrize("M", [96, 192, 400])
def test_layers_beside_scores(G, M):
    A = torch.randn((3, 200, 200), device="cuda").to(torch.bfloat16)
    Gr = torch.randn((3, 200, 300), device="cuda").to(torch.bfloat16)
    mi, mo = (G.mask_to_device(G.grass_random_mask_host(d, 64, d)) for d in (200, 300))
    train = torch.randn((900, 1_024), device="cuda").to(torch.bfloat16)
    test = torch.randn((M, 1_024), device="cuda").to(torch.bfloat16)
    layer = lambda: G.factgrass_compress(A, Gr, mi, mo, 512, 1, 5)
    score = lambda: G.grass_score_bf16(train, test)
    ref_l, ref_s = layer(), score()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [], []
    for _ in range(40):
        for call, stream, out in zip((layer, score), streams, outs):
            with torch.cuda.stream(stream):
                out.append(call())
    torch.cuda.synchronize()
    assert all(_same(o, ref_l) for o in outs[0]) and all(_same(o, ref_s) for o in outs[1])
