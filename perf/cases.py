"""Timed cases of the compression and attribution path, through the public Python calls.

A case is a dict of plain values; ``op`` says which call it stands for:

    grass    grass_compress: dense per-sample gradients, Random Mask or identity mask, SJLT
    layer    factgrass_compress: one linear layer
    grouped  factgrass_compress_grouped: every linear layer of a transformer in one call
    varlen   factgrass_compress_grouped_varlen: the same for a packed batch of samples of their own lengths
    score    grass_score / grass_score_bf16: all-pair inner products of compressed vectors
    fim      grass_fim, grass_fim_factor, grass_fim_apply, grass_score: preconditioned scores of one layer block

``prepare`` draws the inputs on the GPU with the generators of ``workloads`` (the value distributions and zero
patterns of the five benchmark configurations); masks and the projection's seed belong to the program and are the
same for every batch, as in a real run.  Byte counts in ``work`` are what the call cannot do without: the 32-byte
memory sectors that hold a masked element (expected number for a uniform mask), every other input and every output
once.
"""
from __future__ import annotations

import math

import torch

import paper_2505_18976_b200 as G
from paper_2505_18976_b200 import workloads as W

HASH_SEED = 0x5EED
MASK_SEED = 3
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f32": 4, "bf16": 2}
LAYERS = {"gpt2s": W._gpt2_small_layers, "llama3_8b": W._llama3_8b_layers}


def listed():
    return [
        # one sample at a time (a loop that takes one gradient per backward pass) from an MLP of 0.11 M parameters:
        # the smallest call, its cost is the call itself
        dict(name="grass_one_sample", op="grass", n=1, p=109_386, kprime=8_192, k=2_048, dtype="f32", out="f32",
             zero_prob=0.9, dist="normal"),
        # a batch of gradients of a small model; benchmark configuration 1
        dict(name="grass_256x64k", op="grass", n=256, p=65_536, kprime=8_192, k=2_048, dtype="f32", out="f32",
             zero_prob=0.9, dist="normal"),
        # a ragged batch of ResNet-9-sized gradients (4.83 M parameters, an odd row length, k' = 4 k) kept in bf16,
        # compressed into a bf16 cache
        dict(name="grass_bf16_61x4.8M", op="grass", n=61, p=4_825_157, kprime=32_768, k=8_192, dtype="bf16",
             out="bf16", zero_prob=0.7, dist="student_t3"),
        # a full batch of the large dense configuration (configuration 2)
        dict(name="grass_512x4M", op="grass", n=512, p=4_194_304, kprime=65_536, k=4_096, dtype="f32", out="f32",
             zero_prob=0.7, dist="student_t3"),
        # plain SJLT without a mask at p = 131,072 (the shape of the projection benchmark)
        dict(name="sjlt_1024x128k", op="grass", n=1_024, p=131_072, kprime=0, k=4_096, dtype="f32", out="f32",
             zero_prob=0.7, dist="normal"),
        # one linear layer from a backward hook, padded batch; configuration 3
        dict(name="layer_768x3072", op="layer", B=32, T=512, d_in=768, d_out=3_072, kin=128, kout=128, k=4_096,
             dtype="bf16", pad=0.05),
        # all 48 linear layers of GPT-2-small after one backward pass (configuration 4); the activations are new
        # tensors in every pass, so the descriptor table is built in every pass too
        dict(name="gpt2s_16x1024", op="grouped", layers="gpt2s", blocks=12, B=16, T=1_024, kin=64, kout=64, k=1_024,
             dtype="bf16", handle=False),
        # all 224 linear layers of a Llama-3-8B-shaped model (configuration 5), activations in buffers that the
        # program reuses, so that it keeps the descriptor table
        dict(name="llama3_8b_4x2048", op="grouped", layers="llama3_8b", blocks=32, B=4, T=2_048, kin=64, kout=64,
             k=4_096, dtype="bf16", handle=True),
        # fp32 activations of three GPT-2-small blocks, seven sequences of their own lengths packed without padding,
        # factor masks of 128 for k_l = 4,096 (the ratio of the published comparison)
        dict(name="varlen_f32_7x1024", op="varlen", layers="gpt2s", blocks=3, B=7, T=1_024, kin=128, kout=128,
             k=4_096, dtype="f32"),
        # attribution: 16,384 compressed training gradients against 256 test gradients (configuration 5)
        dict(name="score_f32_16384x256", op="score", N=16_384, M=256, D=4_096, dtype="f32"),
        # attribution over a bf16 cache of all 48 layers of GPT-2-small (48 x 1,024), 4,656 training samples, a test
        # set that is no multiple of any tile
        dict(name="score_bf16_4656x300", op="score", N=4_656, M=300, D=49_152, dtype="bf16"),
        # one layer block of preconditioned attribution: projected FIM of 4,656 samples, damped factor, the test
        # rows solved against it, scores
        dict(name="fim_4656x1024", op="fim", n=4_656, k=1_024, M=256),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(("grass", "grass", "sjlt", "layer", "grouped", "varlen", "score", "fim"))
    dt = rng.choice(("f32", "bf16"))
    if op == "grass":
        p = _log_int(rng, 16_384, 6_000_000)
        n = _log_int(rng, 1, min(512, max(1, (1 << 31) // p)))
        kprime = max(512, int(p / math.exp(rng.uniform(math.log(4), math.log(128)))))
        return dict(op="grass", n=n, p=p, kprime=kprime, k=_log_int(rng, 512, 8_192), dtype=dt,
                    out=rng.choice(("f32", "f32", "bf16")), zero_prob=rng.choice((0.5, 0.7, 0.9, 0.95)),
                    dist=rng.choice(("normal", "student_t3")))
    if op == "sjlt":
        p = _log_int(rng, 16_384, 524_288)
        n = _log_int(rng, 32, min(2_048, (1 << 27) // p))
        return dict(op="grass", n=n, p=p, kprime=0, k=_log_int(rng, 512, 32_768), dtype=dt, out="f32",
                    zero_prob=rng.choice((0.0, 0.5, 0.7, 0.9, 0.99)), dist="normal")
    if op == "layer":
        return dict(op="layer", B=_log_int(rng, 1, 32), T=_log_int(rng, 32, 2_048),
                    d_in=rng.choice((768, 1_000, 2_048, 3_072, 4_096)), d_out=rng.choice((768, 1_000, 2_304, 3_072, 4_096)),
                    kin=rng.randint(32, 128), kout=rng.randint(32, 128), k=_log_int(rng, 256, 4_096), dtype=dt,
                    pad=rng.choice((0.0, 0.05)))
    if op == "grouped":
        kk = rng.choice((32, 48, 64, 96, 128))
        if rng.random() < 0.5:
            return dict(op="grouped", layers="gpt2s", blocks=rng.randint(1, 12), B=rng.randint(1, 16),
                        T=_log_int(rng, 64, 1_024), kin=kk, kout=kk, k=_log_int(rng, 256, 4_096), dtype=dt,
                        handle=rng.random() < 0.5)
        return dict(op="grouped", layers="llama3_8b", blocks=rng.randint(1, 8), B=rng.randint(1, 4),
                    T=_log_int(rng, 256, 2_048), kin=kk, kout=kk, k=_log_int(rng, 256, 4_096), dtype=dt,
                    handle=rng.random() < 0.5)
    if op == "varlen":
        kk = rng.choice((32, 64, 128))
        return dict(op="varlen", layers="gpt2s", blocks=rng.randint(1, 6), B=rng.randint(1, 24), T=_log_int(rng, 64, 1_024),
                    kin=kk, kout=kk, k=_log_int(rng, 256, 4_096), dtype=dt)
    if op == "score":
        D = 8 * _log_int(rng, 64, 8_192)
        return dict(op="score", N=_log_int(rng, 256, min(32_768, (1 << 28) // D)), M=_log_int(rng, 1, 1_024), D=D, dtype=dt)
    return dict(op="fim", n=_log_int(rng, 512, 16_384), k=_log_int(rng, 256, 4_096), M=_log_int(rng, 1, 512))


# ------------------------------------------------------------------------------------------------ inputs

def _mask(p, kprime, seed):
    return G.mask_to_device(G.grass_random_mask_host(p, kprime, seed))


def _workload(case, layers, seed):
    return W.FactGrassWorkload("case", tuple(layers), B=case["B"], T=case["T"], kin=case["kin"], kout=case["kout"],
                               k=case["k"], g_dist="laplace", g_scale=1e-3, pad_frac=case.get("pad", 0.0),
                               data_seed=seed, mask_seed=MASK_SEED, hash_seed=HASH_SEED)


def _layer_dicts(case, layers, seed, rows=None):
    """The layers as the grouped calls take them; rows: tokens of a packed batch (all layers share its layout)."""
    wl = _workload(case, layers, seed)
    out = []
    for l, lay in enumerate(layers):
        mi, mo = W.layer_mask_seeds(wl, l)
        A, Gr = W.layer_io(wl, l, "cuda", DTYPE[case["dtype"]])
        if rows is not None:
            A, Gr = A.view(-1, lay.d_in)[:rows], Gr.view(-1, lay.d_out)[:rows]
        out.append(dict(A=A, G=Gr, mask_in=_mask(lay.d_in, case["kin"], mi), mask_out=_mask(lay.d_out, case["kout"], mo),
                        k=case["k"], s=1, seed=W.layer_hash_seed(wl, l), out_offset=l * case["k"]))
    return out


def prepare(case, seed):
    op = case["op"]
    st = dict(case)
    if op == "grass":
        st["g"] = W.dense_gradients(case["n"], case["p"], case["zero_prob"], case["dist"], 1e-2, seed, "cuda",
                                    DTYPE[case["dtype"]])
        st["idx"] = _mask(case["p"], case["kprime"], MASK_SEED) if case["kprime"] else None
    elif op == "layer":
        st.update(_layer_dicts(case, [W.LinearLayer("layer", case["d_in"], case["d_out"])], seed)[0])
    elif op in ("grouped", "varlen"):
        layers = LAYERS[case["layers"]](case["blocks"])
        B, rows = case["B"], None
        if op == "varlen":
            gen = torch.Generator().manual_seed(seed)
            count = torch.randint(case["T"] // 4, case["T"] + 1, (B,), generator=gen)
            begin = torch.cumsum(count, 0) - count
            rows = int(count.sum())
            st["tok_count"], st["tok_begin"] = count.to(torch.int32).cuda(), begin.to(torch.int64).cuda()
        st["dicts"] = _layer_dicts(case, layers, seed, rows)
        st["out"] = torch.empty((B, case["k"] * len(layers)), dtype=torch.float32, device="cuda")
        st["workspace"] = torch.empty(G.factgrass_grouped_workspace_bytes(len(layers)), dtype=torch.uint8, device="cuda")
        if case.get("handle"):
            st["group"] = G.GroupedLayers(st["dicts"])
    elif op == "score":
        train, test = W.score_vectors(case["N"], case["M"], case["D"], seed, "cuda")
        st["train"], st["test"] = train.to(DTYPE[case["dtype"]]), test.to(DTYPE[case["dtype"]])
    else:
        st["train"], st["test"] = W.score_vectors(case["n"], case["M"], case["k"], seed, "cuda")
        st["lam"] = 0.1
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------------------------------------ one pass

def run(st):
    op = st["op"]
    if op == "grass":
        return G.grass_compress(st["g"], st["idx"], st["k"], 1, HASH_SEED, out_dtype=DTYPE[st["out"]])
    if op == "layer":
        return G.factgrass_compress(st["A"], st["G"], st["mask_in"], st["mask_out"], st["k"], st["s"], st["seed"])
    if op == "grouped":
        group = st["group"] if st["handle"] else G.GroupedLayers(st["dicts"])
        return G.factgrass_compress_grouped(group, st["out"], st["workspace"])
    if op == "varlen":
        return G.factgrass_compress_grouped_varlen(G.GroupedLayers(st["dicts"]), st["out"], st["workspace"], st["B"],
                                                   st["T"], st["tok_begin"], st["tok_count"])
    if op == "score":
        return (G.grass_score if st["dtype"] == "f32" else G.grass_score_bf16)(st["train"], st["test"])
    # The factor takes the matrix's place and its upper triangle is scratch, so what comes back is what the program
    # goes on with: the solved test rows and the scores.
    F = G.grass_fim(st["train"])
    G.grass_fim_factor(F, st["lam"])
    solved = G.grass_fim_apply(F, st["test"].clone())
    return {"solved": solved, "scores": G.grass_score(st["train"], solved)}


# ------------------------------------------------------------------------------------------------ what it takes

def _sectors(p, kprime, size):
    """Expected 32-byte sectors of a row of p elements that a uniform mask of kprime of them touches, in bytes."""
    per = 32 // size
    if kprime == 0 or kprime >= p:
        return p * size
    return 32 * math.ceil(p / per) * (1.0 - (1.0 - kprime / p) ** per)


def work(case):
    op, size = case["op"], SIZE[case.get("dtype", "f32")]
    if op == "grass":
        n, kprime = case["n"], case["kprime"]
        bytes_ = n * _sectors(case["p"], kprime, size) + 4 * kprime + n * case["k"] * SIZE[case["out"]]
        return {"bytes": bytes_, "flops": n * (kprime or case["p"]) * (1.0 - case["zero_prob"])}
    if op in ("layer", "grouped", "varlen"):
        layers = [W.LinearLayer("layer", case["d_in"], case["d_out"])] if op == "layer" else \
            LAYERS[case["layers"]](case["blocks"])
        tokens = case["B"] * case["T"] * (0.625 if op == "varlen" else 1.0)     # mean length of the packed samples
        row = sum(_sectors(l.d_in, case["kin"], size) + _sectors(l.d_out, case["kout"], size) for l in layers)
        bytes_ = tokens * row + len(layers) * (4 * (case["kin"] + case["kout"]) + case["B"] * case["k"] * 4)
        return {"bytes": bytes_, "flops": 2.0 * tokens * case["kin"] * case["kout"] * len(layers)}
    if op == "score":
        N, M, D = case["N"], case["M"], case["D"]
        return {"bytes": (N + M) * D * size + 4 * N * M, "flops": 2.0 * N * M * D}
    n, k, M = case["n"], case["k"], case["M"]
    return {"bytes": 4.0 * (n * k + k * k + 2 * M * k + n * M),
            "flops": float(n) * k * (k + 1) + k ** 3 / 3.0 + 2.0 * M * k * k + 2.0 * n * M * k}


def tolerance(case):
    """fp32 sums throughout (bf16 products are exact in fp32).  A bf16 output is the same sum rounded once: values
    near a rounding boundary may fall on the other side, one unit in the last place (2^-8) apart.  The solve carries
    the condition number of F + 0.1 I (below 100 at these shapes)."""
    if case["op"] == "grass" and case["out"] == "bf16":
        return {"rel": 2e-3, "max": 0.01}
    if case["op"] == "fim":
        return {"rel": 1e-4, "max": 4e-3}
    return {"rel": 1e-5, "max": 4e-4}
