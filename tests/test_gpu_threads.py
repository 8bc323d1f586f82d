"""Two threads with problems of different sizes, each on its own stream: the launch of one must not depend on what the other has
asked the runtime for in between (the calls release the interpreter's lock around the library)."""
import threading

import pytest
import torch

import paper_2505_18976_b200 as G

pytestmark = pytest.mark.gpu


def _calls(name):
    """The same kernel with much shared memory and with less, both above what needs no permission."""
    gen = torch.Generator("cuda").manual_seed(1)
    r = lambda *s: torch.randn(s, generator=gen, device="cuda")       # noqa: E731
    if name in ("mask", "sjlt"):
        g = r(40, 4_000)
        idx = G.mask_to_device(G.grass_random_mask_host(4_000, 900, 1)) if name == "mask" else None
        sizes = (40_000, 14_000) if name == "mask" else (32_768, 17_000)
        return [lambda k=k: G.grass_compress(g, idx, k, 1, 3) for k in sizes]
    if name == "layer":
        A = r(3, 40, 100)
        m = G.mask_to_device(G.grass_random_mask_host(100, 30, 1))
        return [lambda k=k: G.factgrass_compress(A, A, m, m, k, 1, 3) for k in (30_000, 5_000)]
    out = []
    for k in (1_500, 100):
        X = r(2 * k, k)
        L, b = G.grass_fim_factor(G.grass_fim(X), 0.1), r(1, k)
        out.append(lambda L=L, b=b: G.grass_fim_apply(L, b.clone()))
    return out


@pytest.mark.parametrize("name", ["mask", "sjlt", "layer", "solve"])
def test_two_threads_two_sizes(tune, name):
    if name == "sjlt":
        tune(compress_dense=2)      # the table's kernel whatever the size
    calls = _calls(name)
    want = [c() for c in calls]
    torch.cuda.synchronize()
    failed, got = [], [None, None]
    start = threading.Barrier(2)

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(1_500):
                    got[i] = calls[i]()
                torch.cuda.current_stream().synchronize()
        except Exception as e:      # noqa: BLE001  (reported by the main thread)
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for w, g in zip(want, got):
        assert torch.allclose(w, g, rtol=1e-4, atol=1e-4 * float(w.abs().max()))
