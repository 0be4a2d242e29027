"""What the framework is timed on: the calls a program makes that keeps its linear weights entropy-coded.

Such a program codes a checkpoint tensor by tensor (``encode_device``, the bytes into GPU memory of its own), keeps
the streams there and decodes a weight before every use of it (``decode``; ``decode_many`` for all weights of a block;
``decode_tile_range`` for a rank's shard), brings a stream in from page-locked host memory first where the model does
not fit (``upload``, then ``decode``), or multiplies a few tokens straight from the stream (``decode_matmul``).

The weights are the random matrices of ``paper_2609_34185_b200.synth`` (rows of one scale each; Gaussian, Laplace,
Student-t, Gaussian with outliers), drawn on the GPU.  Sizes are those of the benchmark's configurations, the
paper's reference layer, and generic ones.

A case: ``kind`` decode | many | shard | stream | matmul | encode; ``R``, ``C`` of the matrix (``many``: ``H`` and ``F``,
four H x H and three H x F matrices); ``bpp`` target bits per weight; ``dist`` of the rows; ``out`` type of the
decoded weights; ``tile`` 8-weight blocks per tile (0: the encoder's default, -1: the size the library suggests for the
GPU); ``ranks`` and ``rank`` of a shard; ``T`` tokens of a product.
"""
import math

import torch

import paper_2609_34185_b200 as ep

OUT = {"bf16": ep.BF16, "fp16": ep.FP16, "fp8": ep.FP8_E4M3, "int8": ep.INT8, "fp32": ep.FP32}
SCALES = {"gauss": (0.005, 0.05), "outlier": (0.005, 0.05), "laplace": (0.005, 0.03), "student": (0.01, 0.04)}


def listed():
    return [
        # the smallest weight anyone compresses: latency of one call.  One tile per 64 rows, eight in all
        {"name": "small layer, 8 tiles", "kind": "decode", "R": 512, "C": 512, "bpp": 4.0, "dist": "gauss", "out": "bf16", "tile": 4096},
        # an ordinary square projection as a plain encode() call leaves it (the paper's tile size)
        {"name": "square layer 3 bpp", "kind": "decode", "R": 4096, "C": 4096, "bpp": 3.0, "dist": "student", "out": "bf16", "tile": 0},
        # a large weight at the paper's two headline rates; tiles sized for the GPU, and the paper's
        {"name": "large layer 4 bpp", "kind": "decode", "R": 8192, "C": 8192, "bpp": 4.0, "dist": "laplace", "out": "fp16", "tile": -1},
        {"name": "large layer 8 bpp", "kind": "decode", "R": 8192, "C": 8192, "bpp": 8.0, "dist": "laplace", "out": "fp16", "tile": 0},
        # a ragged middle-sized weight for an integer matrix product
        {"name": "ragged layer int8", "kind": "decode", "R": 3000, "C": 1736, "bpp": 3.5, "dist": "laplace", "out": "int8", "tile": 0},
        # all weights of a transformer block before its matrix products: 8-bit container, and one layer of a deep stack
        {"name": "block of 7, fp8", "kind": "many", "H": 5120, "F": 17408, "bpp": 2.5, "dist": "outlier", "out": "fp8", "tile": -1},
        {"name": "block of 7, bf16", "kind": "many", "H": 5120, "F": 17408, "bpp": 3.5, "dist": "gauss", "out": "bf16", "tile": -1},
        # one rank of eight decodes its tiles of a shared weight
        {"name": "shard 3 of 8", "kind": "shard", "R": 8192, "C": 8192, "bpp": 4.0, "dist": "laplace", "out": "bf16", "tile": 0, "ranks": 8, "rank": 3},
        # a weight that lives in host memory, brought in and decoded for its use
        {"name": "streamed layer", "kind": "stream", "R": 4096, "C": 4096, "bpp": 3.5, "dist": "gauss", "out": "bf16", "tile": 0},
        # token generation on the paper's reference layer, the dense weight never written
        {"name": "16 tokens times layer", "kind": "matmul", "R": 10240, "C": 3840, "bpp": 4.0, "dist": "gauss", "T": 16},
        # compression: the reference layer, and a small tensor of the same checkpoint
        {"name": "encode reference layer", "kind": "encode", "R": 10240, "C": 3840, "bpp": 4.0, "dist": "gauss", "tile": 0},
        {"name": "encode small layer", "kind": "encode", "R": 512, "C": 1024, "bpp": 4.0, "dist": "gauss", "tile": 0},
    ]


def _log_size(rng, lo, hi, step):
    """A multiple of `step` in [lo, hi], spread evenly over the logarithm."""
    return max(lo, min(hi, step * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)))


def draw(rng):
    """One more case: mostly single decodes, which is what a served model spends its calls on."""
    kind = rng.choice(["decode"] * 5 + ["many", "shard", "stream", "matmul", "encode", "encode"])
    bpp = rng.choice([2.0, 2.5, 3.0, 3.5, 4.0, 4.5, 5.0, 5.5, 6.0, 7.0, 8.0])
    dist = rng.choice(["gauss", "outlier", "laplace", "laplace"] + (["student"] if bpp <= 5.0 else []))
    c = {"kind": kind, "bpp": bpp, "dist": dist}
    if kind == "many":
        c.update(H=_log_size(rng, 512, 5120, 128), F=_log_size(rng, 1024, 17408, 256), bpp=min(bpp, 6.0))
    else:
        # rows to any count, columns a multiple of 8 (of 256 for the fused product)
        c.update(R=_log_size(rng, 256, 8192, 1), C=_log_size(rng, 512, 8192, 256 if kind == "matmul" else 8))
    if kind == "matmul":
        c.update(bpp=min(max(bpp, 3.0), 6.0), T=_log_size(rng, 1, 64, 1))
        return c
    c["tile"] = rng.choice([0, 0, -1])
    if kind != "encode":
        c["out"] = rng.choice(["bf16", "bf16", "fp16", "fp8", "int8", "fp32"])
        if c["out"] in ("fp8", "int8"):                      # values on an 8-bit grid hold little more than these rates
            c["bpp"] = min(c["bpp"], 4.0)
    if kind == "shard":
        c["ranks"] = rng.choice([2, 4, 8])
        c["rank"] = rng.randrange(c["ranks"])
    return c


def _weights(R, C, dist, out, seed):
    """float32 [R, C] on the GPU; for the 8-bit containers scaled per row to their range and rounded to their grid,
    as the FP8 and INT8 routes do before they compress."""
    g = torch.Generator("cuda").manual_seed(seed)
    lo, hi = SCALES[dist]
    row = torch.rand(R, 1, generator=g, device="cuda").mul_(math.log(hi / lo)).exp_().mul_(lo)
    if dist == "laplace":
        u = torch.rand(R, C, generator=g, device="cuda").sub_(0.5)
        W = u.sign() * torch.log1p(u.abs().mul_(-2.0).clamp_(min=-0.99999994)).neg_()
    else:
        W = torch.randn(R, C, generator=g, device="cuda")
        if dist == "student":
            chi2 = torch.zeros(R, C, device="cuda")
            for _ in range(5):
                chi2 += torch.randn(R, C, generator=g, device="cuda").square_()
            W *= chi2.div_(5.0).rsqrt_()
        elif dist == "outlier":
            u = torch.rand(R, C, generator=g, device="cuda")
            W = torch.where(u < 0.001, torch.where(u < 0.0005, -8.0, 8.0), W)
    W *= row
    if out in ("fp8", "int8"):
        W /= W.abs().amax(1, keepdim=True).clamp_(min=1e-30) / (448.0 if out == "fp8" else 127.0)
        W = W.to(torch.float8_e4m3fn).float() if out == "fp8" else W.round_()
    return W.contiguous()


def _coded(W, bpp, tile, **opts):
    R, C = W.shape
    if tile < 0:
        tile = ep.suggest_tile_vectors(R, C, bpp, 148 * ep.decode_tiles_per_sm())
    return ep.encode_device(W, bpp, tile_vectors=tile, **opts)


def _empty_out(n, out):
    types = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp8": torch.float8_e4m3fn, "int8": torch.int8, "fp32": torch.float32}
    return torch.empty(n, dtype=types[out], device="cuda")


def prepare(case, seed):
    kind, bpp, dist = case["kind"], case["bpp"], case["dist"]
    s = {"kind": kind}
    if kind == "many":
        shapes = [(case["H"], case["H"])] * 4 + [(case["H"], case["F"])] * 3
        tile = ep.suggest_tile_vectors_batch(shapes, bpp, 148) if case["tile"] < 0 else case["tile"]
        s["blobs"] = []
        for i, (R, C) in enumerate(shapes):
            W = _weights(R, C, dist, case["out"], 7 * seed + i)
            s["blobs"].append(ep.upload(_coded(W, bpp, tile)))
        s["dtype"] = OUT[case["out"]]
        s["outs"] = [_empty_out(sh, case["out"]) for sh in shapes]      # one set of buffers, used for every layer
        return s
    R, C = case["R"], case["C"]
    W = _weights(R, C, dist, case.get("out"), 7 * seed)
    if kind == "encode":
        s["W"], s["bpp"] = W, bpp
        tile = case["tile"]
        s["tile"] = ep.suggest_tile_vectors(R, C, bpp, 148 * ep.decode_tiles_per_sm()) if tile < 0 else tile
        opts = ep.binding.encode_opts(tile_vectors=s["tile"])
        need = ep.load().ep_encode_device_workspace_bytes(R, C, bpp, opts)
        s["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")     # kept from tensor to tensor
        # where the finished stream goes on the GPU: the serving program's own memory, with room to spare
        s["arena"] = torch.zeros(int(R * C * (bpp + 1) / 8) + (1 << 17), dtype=torch.uint8, device="cuda")
        return s
    if kind == "matmul":
        # the fused product reads one tile per row, 11-bit frequencies
        s["blob"] = ep.upload(_coded(W, bpp, C // 8, b_start=11, b_max=11))
        g = torch.Generator("cuda").manual_seed(7 * seed + 1)
        s["x"] = torch.randn(case["T"], C, generator=g, device="cuda").to(torch.bfloat16)
        s["y"] = torch.empty(case["T"], R, device="cuda")
        return s
    blob = _coded(W, bpp, case["tile"])
    s["dtype"] = OUT[case["out"]]
    if kind == "stream":
        s["blob"] = blob
        s["pinned"] = torch.from_numpy(blob.data).pin_memory()
        s["out"] = _empty_out((R, C), case["out"])
        return s
    s["blob"] = ep.upload(blob)
    if kind == "shard":
        I = blob.info
        s["tiles"] = range(I.n_tiles * case["rank"] // case["ranks"], I.n_tiles * (case["rank"] + 1) // case["ranks"])
        if not len(s["tiles"]):                                          # fewer tiles than ranks: the first rank's share
            s["tiles"] = range(0, 1)
        blocks = min(s["tiles"].stop * I.V, R * C // 8) - s["tiles"].start * I.V
        s["out"] = _empty_out(8 * blocks, case["out"])
    else:
        s["out"] = _empty_out((R, C), case["out"])
    return s


def run(state):
    kind = state["kind"]
    if kind == "decode":
        return ep.decode(state["blob"], state["dtype"], out=state["out"])
    if kind == "many":
        ep.decode_many(state["blobs"], state["dtype"], state["outs"])
        return state["outs"]
    if kind == "shard":
        return ep.decode_tile_range(state["blob"], state["tiles"], state["dtype"], out=state["out"])
    if kind == "stream":
        dev = ep.upload(state["blob"], pinned=state["pinned"], non_blocking=True)
        return ep.decode(dev, state["dtype"], out=state["out"])
    if kind == "matmul":
        return ep.decode_matmul(state["blob"], state["x"], out=state["y"])
    blob = ep.encode_device(state["W"], state["bpp"], workspace=state["workspace"], tile_vectors=state["tile"])
    state["arena"][:len(blob)].copy_(torch.from_numpy(blob.data), non_blocking=True)
    state["blob"] = blob                                                 # alive while its bytes are under way
    return state["arena"]


def work(case):
    """Bytes: the stream at its target rate and the dense side, each once.  Entropy decoding has no floating-point count;
    the product has 2 T R C."""
    if case["kind"] == "many":
        n = 4 * case["H"] * case["H"] + 3 * case["H"] * case["F"]
    else:
        n = case["R"] * case["C"]
    if case["kind"] == "shard":
        n /= case["ranks"]
    stored = n * case["bpp"] / 8
    if case["kind"] == "encode":
        return {"bytes": 4 * n + stored, "flops": 0}
    if case["kind"] == "matmul":
        T = case["T"]
        return {"bytes": stored + 2 * T * case["C"] + 4 * T * case["R"], "flops": 2.0 * T * n}
    width = {"bf16": 2, "fp16": 2, "fp8": 1, "int8": 1, "fp32": 4}[case["out"]]
    return {"bytes": stored + width * n, "flops": 0}


def tolerance(case):
    """Streams are the same bytes and weights the same bits whoever makes them; the product sums exact bf16 products
    in float32 in any order."""
    return {"rel": 1e-5} if case["kind"] == "matmul" else "exact"
