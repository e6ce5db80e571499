"""Workloads of Bi-Level Routing Attention, as programs that use this library run them.

A case is one attention layer of one stage of a network, called through the package's public entry
points: an inference step is `bra_forward` into the program's own output tensor; a training step is
`bra_forward` with the index and the log-sum-exp kept, then `bra_backward` with every gradient, the
results allocated by the calls as an autograd function would.  Problem, LCE weights and scratch buffer
are kept between passes, as a network keeps them with its layer.

Four kinds of network, with the sizes of this repository's configurations and their neighbours:
  classify  four stages with maps of 1/4 ... 1/32 of the image, widths 64 or 96 times 2^stage, heads of
            32 channels, 7 x 7 regions, topk 1, 4, 16, 49; 49 regions of the last stage are single tokens
  segment   512 x 512 and other square images, 8 x 8 regions, topk 4 and others
  detect    rectangular images up to 800 x 1333, 16 x 16 regions; the map is seldom a multiple of 16
  vit       one plain map, heads of 64 channels, 8 x 8 regions, topk 12
"""
import math

import torch

import paper_2303_08810_b200 as bra


def _case(name, B, H, W, heads, head_dim, S, topk, dtype="bf16", train=False, routing="scattered"):
    c = {"B": B, "H": H, "W": W, "heads": heads, "head_dim": head_dim, "S": S, "topk": topk,
         "dtype": dtype, "train": train, "routing": routing}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem, single precision: a gradient check or a unit test of a training program
        _case("tiny-fp32-train", 1, 16, 16, 1, 32, 4, 2, "f32", train=True),
        # first stage at 224 x 224: one image (an interactive request), a batch, a training batch
        _case("stage1-one-image", 1, 56, 56, 2, 32, 7, 1),
        _case("stage1-batch", 64, 56, 56, 2, 32, 7, 1),
        _case("stage1-train", 64, 56, 56, 2, 32, 7, 1, train=True),
        # second stage, the layer most of whose time is the backward pass; and the same layer in single
        # precision, the precision the paper's throughput table was taken in
        _case("stage2-train", 64, 28, 28, 4, 32, 7, 4, train=True),
        _case("stage2-batch-fp32", 64, 28, 28, 4, 32, 7, 4, "f32"),
        # third stage (the deepest: 8 of 14 or 18 of 30 layers), inference and training
        _case("stage3-batch", 64, 14, 14, 8, 32, 7, 16),
        _case("stage3-train", 64, 14, 14, 8, 32, 7, 16, train=True),
        # last stage: every region is one token and all of them are routed to, plain attention over 49 tokens
        _case("stage4-batch", 64, 7, 7, 16, 32, 7, 49),
        # 512 x 512 segmentation map at stride 4
        _case("segment-512", 2, 128, 128, 2, 32, 8, 4),
        # 800 x 1333 detection image at stride 8, the wide network: a ragged map, fine-tuned with two images a GPU
        _case("detect-ragged-train", 2, 100, 167, 6, 32, 16, 4, train=True, routing="clustered"),
        # plain vision transformer whose attention layers are replaced and fine-tuned
        _case("vit-train", 16, 32, 32, 12, 64, 8, 12, train=True),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["classify", "classify", "classify", "segment", "detect", "vit"])
    dtype, routing = "bf16", rng.choice(["scattered", "clustered"])
    train = rng.random() < 0.5
    head_dim = 32
    if kind == "classify":
        stage = rng.randrange(4)
        side = 32 * rng.randint(5, 12) >> (2 + stage)
        H = W = side
        heads, S, topk = rng.choice([2, 3]) << stage, 7, (1, 4, 16, 49)[stage]
        if rng.random() < 0.2:
            dtype = "f32"
        # at most the tokens x channels of the largest listed batch (single precision: a quarter of it)
        room = 64 * 56 * 56 * 64 // (4 if dtype == "f32" else 1) // (2 if dtype == "f32" and train else 1)
        B = _log_int(rng, 1, max(1, min(64, room // (H * W * heads * 32))))
    elif kind == "segment":
        stage = rng.randrange(3)
        H = W = 32 * rng.randint(8, 16) >> (2 + stage)
        heads, S, topk, B = rng.choice([2, 3]) << stage, 8, rng.choice([1, 2, 4, 8]), rng.randint(1, 2)
    elif kind == "detect":
        stride = rng.choice([8, 16])
        short, ratio = rng.randint(480, 800), rng.uniform(1.0, 1.66)
        H, W = -(-short // stride), -(-int(short * ratio) // stride)
        if rng.random() < 0.5:
            H, W = W, H
        heads, S, topk, B = rng.choice([4, 6]) * (stride // 8), 16, rng.choice([2, 4]) * (stride // 8), rng.randint(1, 2)
        if stride == 8:
            topk = min(topk, 4)
    else:
        H = W = rng.randint(14, 32)
        heads, head_dim, S, topk, B = rng.choice([3, 6, 12]), 64, 8, 12, _log_int(rng, 1, 16)
    return _case(None, B, H, W, heads, head_dim, S, topk, dtype, train, routing)


def _tensor(case, gen, offset=None):
    B, H, W, C = case["B"], case["H"], case["W"], case["heads"] * case["head_dim"]
    x = torch.randn(B, H, W, C, device="cuda", generator=gen)
    if offset is not None:
        x += offset
    return x.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)


def _region_offsets(case, gen, centres):
    """[B,H,W,C]: every region belongs to one of four semantic groups, so that regions of a group route
    to one another and a few key regions receive most of the routes."""
    B, H, W, S = case["B"], case["H"], case["W"], case["S"]
    hs, ws = -(-H // S), -(-W // S)
    group = torch.randint(0, centres.shape[0], (B, S, S), device="cuda", generator=gen)
    group = group.repeat_interleave(hs, dim=1).repeat_interleave(ws, dim=2)
    return centres[group[:, :H, :W]]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    C = case["heads"] * case["head_dim"]
    off_q = off_k = None
    if case["routing"] == "clustered":
        centres = torch.randn(4, C, device="cuda", generator=gen)
        off_q, off_k = _region_offsets(case, gen, centres), _region_offsets(case, gen, centres)
    st = {"train": case["train"]}
    st["Q"], st["K"], st["V"] = _tensor(case, gen, off_q), _tensor(case, gen, off_k), _tensor(case, gen)
    st["w"] = 0.02 * torch.randn(C, 5, 5, device="cuda", generator=gen)
    st["b"] = 0.02 * torch.randn(C, device="cuda", generator=gen)
    if case["train"]:
        st["dO"] = _tensor(case, gen)
    else:
        st["O"] = torch.empty_like(st["Q"])
    st["p"] = bra.make_problem(case["B"], case["H"], case["W"], C, case["heads"], case["S"], case["topk"],
                               case["dtype"])
    st["ws"] = bra.workspace(st["p"])
    return st


def run(st):
    p, Q, K, V, w, b, ws = (st[n] for n in ("p", "Q", "K", "V", "w", "b", "ws"))
    if not st["train"]:
        O, _, _ = bra.bra_forward(p, Q, K, V, w, b, O=st["O"], ws=ws, want_index=False, want_lse=False)
        return O
    O, index, lse = bra.bra_forward(p, Q, K, V, w, b, ws=ws)
    dQ, dK, dV, dw, db = bra.bra_backward(p, Q, K, V, index, w, lse, st["dO"], ws=ws, want_bias_grad=True)
    return {"O": O, "index": index, "lse": lse, "dQ": dQ, "dK": dK, "dV": dV, "d_lce_w": dw, "d_lce_b": db}


def work(case):
    """Forward: Q, K, V in, O out (and index, lse of a training step).  Backward: Q, K, V, dO, index, lse in,
    dQ, dK, dV out.  Products: two contractions forward, five backward, over the routed tokens; affinity;
    the 25-tap depthwise filter forward, its transpose and its weight gradient backward."""
    B, H, W, S, k = (case[n] for n in ("B", "H", "W", "S", "topk"))
    heads, C = case["heads"], case["heads"] * case["head_dim"]
    R, region = S * S, -(-H // S) * -(-W // S)
    tensor = B * H * W * C * (2 if case["dtype"] == "bf16" else 4)
    weights = C * 26 * 4
    nbytes = 4 * tensor + weights
    attention = 2 * B * H * W * k * region * C
    flops = 2 * attention + 2 * B * R * R * C + 50 * B * H * W * C
    if case["train"]:
        saved = 4 * (B * heads * R * k + B * heads * H * W)
        nbytes += 7 * tensor + 2 * saved + 2 * weights
        flops += 5 * attention + 100 * B * H * W * C
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Against the same path in 64 bits (same index), over the listed and a few dozen drawn cases: bf16 at most
    3.3e-3 (2-norm; 1.7e-3 is the rounding of the results alone) and 0.11 (one element, over the root mean
    square), single precision at most 1.5e-6 and 5e-5.  Four times that.  Routing scores are fp32 sums:
    neighbours in a row may tie to the last bits, so a few index entries may differ."""
    if case["dtype"] == "f32":
        return {"rel": 6e-6, "max": 2e-4, "differ": 1e-4}
    return {"rel": 1.3e-2, "max": 0.45, "differ": 1e-4}
