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


# Calls that follow one another with nothing in between, the first long and on few thread blocks, so that the second's wait
# beside it.  Each writes what the next one reads (alternating inputs: what the pass before left there is wrong), or writes where
# the one before reads or writes.

def _pairs(G):
    """name -> (two inputs, the first call on one of them, the second call, whose result is compared)"""
    g = [torch.randn((3, 500_000), device="cuda") for _ in range(2)]
    gh = [x.to(torch.bfloat16) for x in g]
    long = G.mask_to_device(G.grass_random_mask_host(500_000, 200_000, 3))
    short = G.mask_to_device(G.grass_random_mask_host(2_048, 700, 4))
    A = [torch.randn((2, 2_000, 200), device="cuda").to(torch.bfloat16) for _ in range(2)]
    Gr = torch.randn((2, 2_000, 300), device="cuda").to(torch.bfloat16)
    mi, mo = (G.mask_to_device(G.grass_random_mask_host(d, 64, d)) for d in (200, 300))
    test = torch.randn((40, 2_048), device="cuda")
    test_h, test_l = test.to(torch.bfloat16), torch.randn((40, 512), device="cuda")
    test_lh = test_l.to(torch.bfloat16)
    train = [torch.randn((100, 16_000), device="cuda") for _ in range(2)]
    train_h = [x.to(torch.bfloat16) for x in train]
    wide, wide_h = train[0][:40].clone(), train_h[0][:40].clone()
    c, ch, cl = torch.empty((3, 2_048), device="cuda"), torch.empty((3, 2_048), device="cuda", dtype=torch.bfloat16), torch.empty((2, 512), device="cuda")
    chl = cl.to(torch.bfloat16)
    ws = torch.empty(G.factgrass_grouped_workspace_bytes(1), dtype=torch.uint8, device="cuda")
    s = torch.empty((100, 40), device="cuda")
    few = G.mask_to_device(G.grass_random_mask_host(40, 16, 4))
    t40 = torch.randn((8, 40), device="cuda")

    def layer_bf16(a):
        one = G.GroupedLayers([dict(A=a, G=Gr, mask_in=mi, mask_out=mo, k=512, s=1, seed=5, out_offset=0)])
        return G.factgrass_compress_grouped(one, chl, ws)

    def layer(a):
        return G.factgrass_compress(a, Gr, mi, mo, 512, 1, 5, out=cl)

    return {
        "compress, score": (g, lambda x: G.grass_compress(x, long, 2_048, 1, 5, out=c), lambda x: G.grass_score(c, test)),
        "compress, score_bf16": (gh, lambda x: G.grass_compress(x, long, 2_048, 1, 5, out=ch), lambda x: G.grass_score_bf16(ch, test_h)),
        "compress, compress": (g, lambda x: G.grass_compress(x, long, 2_048, 1, 5, out=c), lambda x: G.grass_compress(c, short, 512, 1, 6)),
        "compress, plain": (g, lambda x: G.grass_compress(x, long, 2_048, 1, 5, out=c), lambda x: G.grass_compress(c, None, 512, 1, 6)),
        "layer, score": (A, layer, lambda x: G.grass_score(cl, test_l)),
        "layer, score_bf16": (A, layer_bf16, lambda x: G.grass_score_bf16(chl, test_lh)),
        "layer, compress": (A, layer, lambda x: G.grass_compress(cl, None, 256, 1, 6)),
        "score, score": (train, lambda x: G.grass_score(x, wide, out=s), lambda x: G.grass_score(s, t40)),
        "score, compress": (train, lambda x: G.grass_score(x, wide, out=s), lambda x: G.grass_compress(s, few, 16, 1, 6)),
        "score_bf16, score": (train_h, lambda x: G.grass_score_bf16(x, wide_h, out=s), lambda x: G.grass_score(s, t40)),
        # the second call's results take the place of the first's
        "compress over compress": (g, lambda x: G.grass_compress(x, long, 2_048, 1, 5, out=c), lambda x: G.grass_compress(x[:, :2_048], short, 2_048, 1, 6, out=c)),
        "score over compress": (g, lambda x: G.grass_compress(x, long, 2_048, 1, 5, out=c), lambda x: G.grass_score(x[:, :2_048], test, out=c[:, :40])),
    }


PAIRS = ["compress, score", "compress, score_bf16", "compress, compress", "compress, plain", "layer, score", "layer, score_bf16",
         "layer, compress", "score, score", "score, compress", "score_bf16, score", "compress over compress", "score over compress"]


# fp32: the first call's values differ by what _same allows and carry that into the second's sums, which differ by as much again.
# bf16 results of the first call: a value whose sum (in another order) falls to the other side of a rounding boundary differs by
# 2^-8 of itself, and of sums of 512 values and more a handful of such differences are below 2^-9.
def _close(a, b, name):
    tol = 2.0 ** -16 if "bf16" not in name else 2.0 ** -9
    return (a - b).abs().max() <= tol * b.abs().max()


@pytest.mark.parametrize("recorded", [False, True])
@pytest.mark.parametrize("name", PAIRS)
def test_calls_wait_for_the_call_before(G, tune, name, recorded):
    # one thread block per row; no zero-fill between the calls
    tune(compress_jsplit=1, compress_dense=1, score_splits=1)
    inputs, first, second = _pairs(G)[name]
    refs = []
    for x in inputs:
        first(x)
        torch.cuda.synchronize()
        refs.append(second(x).clone())
        torch.cuda.synchronize()
    assert not _close(refs[0], refs[1], name)
    outs = []
    if recorded:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for i in range(6):
                first(inputs[i % 2])
                outs.append(second(inputs[i % 2]))
        for _ in range(5):
            graph.replay()
    else:
        for i in range(30):
            first(inputs[i % 2])
            outs.append(second(inputs[i % 2]))
    torch.cuda.synchronize()
    if " over " in name:                           # one buffer: the last call's results
        assert _close(outs[-1], refs[1], name)
    else:
        for i, o in enumerate(outs):
            assert _close(o, refs[i % 2], name), i


@pytest.mark.parametrize("name", ["compress", "layer", "score"])
def test_inputs_are_read_before_the_next_call_overwrites_them(G, tune, name):
    tune(compress_jsplit=1, compress_dense=1, score_splits=1)
    short = G.mask_to_device(G.grass_random_mask_host(2_048, 700, 4))
    src = torch.randn((3, 2_048), device="cuda")
    if name == "compress":
        x = torch.randn((3, 500_000), device="cuda")
        long = G.mask_to_device(G.grass_random_mask_host(500_000, 200_000, 3))
        first, target = lambda: G.grass_compress(x, long, 2_048, 1, 5), x[:, -2_048:]
    elif name == "layer":
        x = torch.randn((2, 2_000, 256), device="cuda").to(torch.bfloat16)
        Gr = torch.randn((2, 2_000, 300), device="cuda").to(torch.bfloat16)
        mi, mo = (G.mask_to_device(G.grass_random_mask_host(d, 64, d)) for d in (256, 300))
        first, target = lambda: G.factgrass_compress(x, Gr, mi, mo, 512, 1, 5), x.view(-1).view(torch.float32)[-3 * 2_048:].view(3, 2_048)
    else:
        x, test = torch.randn((100, 16_000), device="cuda"), torch.randn((40, 16_000), device="cuda")
        first, target = lambda: G.grass_score(x, test), x[:3, -2_048:]
    saved = x.clone()
    ref = first()
    torch.cuda.synchronize()
    for _ in range(20):
        x.copy_(saved)
        got = first()
        G.grass_compress(src, short, 2_048, 1, 6, out=target)
        torch.cuda.synchronize()
        assert _close(got, ref, name)
    assert not torch.equal(x, saved)
