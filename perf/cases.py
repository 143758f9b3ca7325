"""The work that users of this library have it do, as cases that can be timed: one layer call each, through the public
entry points (``layer.VmobaLayer``, ``layer.SteppedAttention``, ``binding.vmoba_full_attn``).

A case is one attention layer on one GPU: the latent grid (T, H, W), the block shape (bT, bH, bW), batch, heads,
head_dim, storage type, block-choice rule and whether the backward follows.  Three kinds of work:

* ``sparse``  the VMoBA layer: partition, block scores, selection, attention over the selected blocks (and, with
  ``backward``, its gradients);
* ``dense``   full attention: the sampler's first denoising steps (forward, raster tensors, through the step switch)
  or, with ``backward``, the training step the sparse layer is compared with.

Inputs follow the package's own recipes (``inputs.py``), drawn on the GPU: ``smooth`` = N(0,1) plus a field that is
smooth over the grid and shared by q, k and v (what gives video tokens their locality), ``white`` = N(0,1) alone (no
locality: early in training), ``sine`` = N(0,1) plus a plane wave.
"""
import math

import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import SteppedAttention, VmobaLayer, default_capacity

HEAD_DIM = 128


def _case(name, kind, grid, block, B=1, heads=12, head_dim=HEAD_DIM, dtype="bf16", inputs="smooth", tau=0.25, topk=0,
          backward=False):
    return {"name": name, "kind": kind, "T": grid[0], "H": grid[1], "W": grid[2], "bT": block[0], "bH": block[1],
            "bW": block[2], "B": B, "heads": heads, "head_dim": head_dim, "dtype": dtype, "inputs": inputs, "tau": tau,
            "topk": topk, "backward": backward}


def listed():
    return [
        # the smallest call: a layer of a toy model or of a unit test of a training loop, fp32, head_dim 64
        _case("tiny_f32_train", "sparse", (4, 8, 8), (1, 8, 8), heads=2, head_dim=64, dtype="f32", inputs="sine",
              backward=True),
        # a layer of a short, small clip (1,872 tokens): latency and launches count
        _case("small_train_1p9k", "sparse", (6, 12, 26), (3, 6, 13), heads=12, backward=True),
        # fine-tuning at low resolution (320 x 512 video, 13,440 tokens), spatial blocks of 840 keys
        _case("lowres_train_13k_2d", "sparse", (21, 20, 32), (21, 5, 8), backward=True),
        # inference at 480p (32,760 tokens), 3D layer with short blocks of 234 keys
        _case("infer_33k_3d", "sparse", (21, 30, 52), (3, 6, 13)),
        # the training-free setting at 480p: every query keeps its 6 best of 20 spatial blocks (1,638 keys)
        _case("infer_33k_2d_topk6", "sparse", (21, 30, 52), (21, 6, 13), topk=6),
        # the training-free setting at 720p (75,600 tokens): 9 of 280 short blocks per query
        _case("infer_76k_3d_topk9", "sparse", (21, 45, 80), (3, 9, 10), topk=9),
        # training at 480p, two samples per GPU, 3D layer
        _case("train_33k_3d_b2", "sparse", (21, 30, 52), (3, 6, 13), B=2, backward=True),
        # the same grid where the selection finds no locality (density 0.23, every query has many blocks)
        _case("train_33k_3d_white", "sparse", (21, 30, 52), (3, 6, 13), inputs="white", backward=True),
        # fine-tuning on a longer clip (576 x 1024 video, 55,296 tokens), 3D layer of 768-key blocks
        _case("train_55k_3d", "sparse", (24, 36, 64), (8, 12, 8), backward=True),
        # the largest: training at 720p with 40 heads, 1D layer of 3,600-key blocks
        _case("train_76k_1d_h40", "sparse", (21, 45, 80), (1, 45, 80), heads=40, backward=True),
        # a dense denoising step of the sampler at 480p
        _case("dense_infer_33k", "dense", (21, 30, 52), (3, 6, 13)),
        # a dense training step at low resolution
        _case("dense_train_13k", "dense", (21, 20, 32), (21, 5, 8), backward=True),
    ]


def _flops_bound(case):
    """Attention FLOPs that a case can reach: what keeps drawn cases below the largest listed one."""
    S, share = case["T"] * case["H"] * case["W"], _density(case)
    return (14 if case["backward"] else 4) * case["head_dim"] * share * float(S) ** 2 * case["B"] * case["heads"]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case between the smallest and the largest listed one: grids of 256 to 76,000 tokens with any divisor structure,
    1D / 2D / 3D blocks of 48 to 4,700 keys, 1 to 40 heads, both directions, both storage types, all input recipes."""
    while True:
        kind = "dense" if rng.random() < 0.2 else "sparse"
        f32 = rng.random() < 0.12
        part = rng.choice(["1d", "2d", "3d"])
        target = _spread(rng, 256, 6000 if f32 else 76000)
        if part == "1d":
            block = (rng.choice([1, 1, 2, 3]), _spread(rng, 6, 48), _spread(rng, 8, 80))
            count = (max(2, round(target / (block[0] * block[1] * block[2]))), 1, 1)
        elif part == "2d":
            block = (_spread(rng, 4, 36), rng.randint(3, 9), rng.randint(4, 13))
            n = max(4, target / (block[0] * block[1] * block[2]))
            nh = max(2, round(math.sqrt(n) * rng.uniform(0.7, 1.2)))
            count = (1, nh, max(2, round(n / nh)))
        else:
            block = (rng.choice([2, 3, 4, 8]), rng.randint(3, 12), rng.randint(5, 13))
            n = max(8, target / (block[0] * block[1] * block[2]))
            side = n ** (1 / 3)
            nt, nh = max(2, round(side * rng.uniform(0.6, 1.1))), max(2, round(side * rng.uniform(0.7, 1.3)))
            count = (nt, nh, max(2, round(n / (nt * nh))))
        grid = tuple(b * c for b, c in zip(block, count))
        S, sb, nb = grid[0] * grid[1] * grid[2], block[0] * block[1] * block[2], count[0] * count[1] * count[2]
        topk = 0
        if kind == "sparse" and not f32 and rng.random() < 0.25:
            topk = max(1, round(nb * rng.uniform(0.04, 0.35)))
        case = _case("", kind, grid, block, B=rng.choice([1, 1, 2]), heads=_spread(rng, 2, 40),
                     head_dim=64 if f32 and rng.random() < 0.5 else HEAD_DIM, dtype="f32" if f32 else "bf16",
                     inputs=rng.choice(["smooth"] * 6 + ["white", "sine"]),
                     tau=rng.choice([0.15, 0.25, 0.25, 0.35, 0.5]), topk=topk, backward=rng.random() < 0.5)
        del case["name"]
        if not 256 <= S <= 76000 or not 48 <= sb <= 4700 or not 4 <= nb <= 1024:
            continue
        rows = S * case["B"] * case["heads"]
        pairs = rows * (topk or nb * min(1.0, 1.05 * case["tau"]))
        # no drawn case costs more than the largest listed one, in arithmetic or in memory
        if _flops_bound(case) > 8e13 * (0.005 if f32 else 1.0):
            continue
        if rows > 3.03e6 or pairs > 3e7:
            continue
        return case


def _density(case):
    """Share of (query, key-block) pairs that are kept: exact for top-k and dense; for the threshold rule what the
    recipes give, roughly (measured at tau = 0.25: white inputs 0.230; smooth ones 0.006 with 234-key blocks, 0.049
    with 768, 0.20 with 3,600: the smaller a block, the better its centroid tells near queries from far ones)."""
    if case["kind"] == "dense":
        return 1.0
    if case["topk"]:
        nb = (case["T"] // case["bT"]) * (case["H"] // case["bH"]) * (case["W"] // case["bW"])
        return min(1.0, case["topk"] / nb)
    if case["inputs"] != "smooth":
        return 0.92 * case["tau"]
    return case["tau"] * min(0.8, 0.19 * (case["bT"] * case["bH"] * case["bW"] / 768) ** 1.5)


def _field(shape, gen):
    """White noise of [T, H, W, d] blurred along the grid axes (Gaussian, sigma 2, periodic), unit deviation."""
    f = torch.randn(shape, generator=gen, device="cuda")
    taps = [math.exp(-0.5 * (i / 2.0) ** 2) for i in range(-8, 9)]
    total = sum(taps)
    for axis in range(3):
        out = torch.zeros_like(f)
        for i, t in zip(range(-8, 9), taps):
            out.add_(torch.roll(f, i, dims=axis), alpha=t / total)
        f = out
    return f / f.std()


def _inputs(case, seed):
    """q, k, v (and dO) in raster order [B, S, heads, head_dim]."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    T, H, W, d = case["T"], case["H"], case["W"], case["head_dim"]
    S, B, heads = T * H * W, case["B"], case["heads"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    names = ["q", "k", "v"] + (["do"] if case["backward"] else [])
    x = {n: torch.empty((B, S, heads, d), dtype=dt, device="cuda") for n in names}
    wave = None
    if case["inputs"] == "sine":
        t, h, w = (torch.arange(n, device="cuda", dtype=torch.float32) / n for n in (T, H, W))
        wave = 2 * math.pi * (t[:, None, None] + h[None, :, None] + w[None, None, :])
    for b in range(B):
        for head in range(heads):
            base = 0.0
            if case["inputs"] == "smooth":
                base = _field((T, H, W, d), gen).reshape(S, d)
            elif case["inputs"] == "sine":
                base = (0.5 * torch.sin(wave + 2 * math.pi * head / heads)).reshape(S, 1)
            for n in names:
                noise = torch.randn((S, d), generator=gen, device="cuda")
                x[n][b, :, head] = (noise if n == "do" else noise + base).to(dt)
    return x


def prepare(case, seed):
    shape = vb.make_shape(case["B"], case["heads"], case["head_dim"], (case["T"], case["H"], case["W"]),
                          (case["bT"], case["bH"], case["bW"]), case["dtype"])
    st = {"case": case, "shape": shape, **_inputs(case, seed)}
    outs = ["o"] + (["dq", "dk", "dv"] if case["backward"] else [])
    if case["kind"] == "sparse":
        # a top-k rule keeps exactly S * k pairs per head, the threshold rule at most about tau of them
        capacity = (shape.B * shape.heads * shape.S * min(case["topk"], shape.n_blocks) if case["topk"]
                    else default_capacity(shape, case["tau"]))
        st["layer"] = VmobaLayer(shape, capacity, with_backward=case["backward"])
        like = st["q"]
    elif case["backward"]:
        # the dense kernels take [B, heads, S, d]: a training program keeps its tensors that way
        for n in ("q", "k", "v", "do"):
            st[n] = st[n].permute(0, 2, 1, 3).contiguous()
        like = st["q"]
        st["lse"] = torch.empty(shape.B * shape.heads * shape.S, dtype=torch.float32, device="cuda")
        st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        st["ws"] = torch.empty(vb.workspace_bytes(shape, vb.STAGE_FULL_BWD), dtype=torch.uint8, device="cuda")
    else:
        # the sampler's switch: its first steps are dense, the layer behind it is the sparse one of the later steps
        st["stepped"] = SteppedAttention(VmobaLayer(shape, default_capacity(shape, case["tau"])), case["tau"], n_steps=50)
        like = st["q"]
    st["out"] = {n: torch.empty_like(like) for n in outs}
    return st


def run(st):
    case, out = st["case"], st["out"]
    if case["kind"] == "dense":
        if not case["backward"]:
            st["stepped"].forward(0, st["q"], st["k"], st["v"], out["o"])
            return out
        vb.vmoba_full_attn(st["shape"], st["q"], st["k"], st["v"], out["o"], st["lse"], st["do"], out["dq"], out["dk"],
                           out["dv"], st["status"], st["ws"])
        return {**out, "lse": st["lse"]}
    L = st["layer"]
    if case["topk"]:
        L.partition(st["q"], L.q_bm, perm=L.perm)
        L.partition(st["k"], L.k_bm)
        L.partition(st["v"], L.v_bm)
        L.block_scores()
        L.select_rule(vb.SELECT_TOPK_LOCAL, topk=case["topk"])
        L.attn_fwd()
        L.partition(out["o"], L.o_bm, inverse=True)
    else:
        L.forward(st["q"], st["k"], st["v"], case["tau"], out["o"])
    if case["backward"]:
        L.backward(st["do"], out["dq"], out["dk"], out["dv"])
    return {**out, "mask_bits": L.mask_bits}


def work(case):
    """Each input read once, each output written once; attention arithmetic on the kept pairs (4 d flops per query and
    key forward, 10 d more backward) plus, for the sparse layer, the query x centroid products."""
    S, d = case["T"] * case["H"] * case["W"], case["head_dim"]
    rows = case["B"] * case["heads"] * S
    es = 2 if case["dtype"] == "bf16" else 4
    tensors = 8 if case["backward"] else 4
    flops = _flops_bound(case)
    if case["kind"] == "sparse":
        nb = (case["T"] // case["bT"]) * (case["H"] // case["bH"]) * (case["W"] // case["bW"])
        flops += 2.0 * rows * nb * d
    return {"bytes": tensors * rows * d * es, "flops": flops}


def tolerance(case):
    """bf16, against the same inputs through the fp32 kernels: off by 3e-3 in the 2-norm and by up to 0.15 rms in a
    single value (P and dS enter the second product rounded to bf16, and so are the results).  fp32, against 64 bits:
    3e-7 and 3e-6 on the tiny case, more where the sums are longer.  A score within rounding of the cutoff may fall
    on either side of it: that is one mask bit and the rows of one query."""
    if case["dtype"] == "bf16":
        return {"rel": 1.2e-2, "max": 0.6, "differ": 1e-3}
    return {"rel": 5e-6, "max": 5e-5, "differ": 1e-3}
