"""The workloads this library is timed on: ToMA-wrapped transformer blocks over the sizes that diffusion models
run them at, called the way a denoising loop calls them (one `toma_block*` call per step, state kept between the
steps of a reuse interval).

A case is one pass = `steps` consecutive steps of the schedule, beginning at step `first`:
  first 0, steps 1   a refresh step: destinations, merge weights, merge, module, unmerge
  first 1, steps 1   a reuse step: merge, module, unmerge with the kept destinations and weights
  first 0, steps 5   a whole reuse interval of five steps, the tokens drifting from step to step
  first 5, steps 5   the second half of the 10/5 schedule: weights from new tokens at kept destinations, four reuses
Step t of a pass has its own tokens and its own output, as the layers and steps of a model do.
"""
import math

import torch

import paper_2509_10918_b200 as toma

DRIFT = 0.05     # change of the tokens from one denoising step to the next
LATTICE = 8      # tokens between the nodes of the smooth component of an image's features
NOISE = 0.3      # per-token noise on top of it: neighbouring tokens have a cosine of about 0.8


def _case(name, **kw):
    case = dict(name=name, module="attention", dtype="bf16", batch=2, grid_h=64, grid_w=64, dim=640, heads=10, tile_h=16, tile_w=16,
                ratio=0.5, extra=0, hidden=0, global_merge=False, unmerge="transpose", first=0, steps=1, reuse=5, weight_reuse=0)
    case.update(kw)
    return case


def listed():
    return [
        # fp32 mode on 1024 tokens: what a user checks a bf16 run against; the least work of all
        _case("f32_1024_refresh", dtype="f32", batch=1, grid_h=32, grid_w=32, tile_h=8, tile_w=8),
        # mid-resolution U-Net block, conditional and unconditional half in one batch: the smallest calls of a sampler,
        # where launches and latencies count; most steps are reuse steps
        _case("mid_reuse", grid_h=32, grid_w=32, dim=1280, heads=20, tile_h=8, tile_w=8, first=1),
        # ... and the step that chooses destinations and weights anew
        _case("mid_refresh", grid_h=32, grid_w=32, dim=1280, heads=20, tile_h=8, tile_w=8),
        # high-resolution U-Net block, one reuse interval: the ordinary case
        _case("high_interval", steps=5),
        # the same size with the whole attention module (projections included) inside the wrap, and few tokens removed
        _case("high_module_r25_interval", module="proj", ratio=0.25, steps=5),
        # the MLP of that block as the wrapped module, unmerged through the softmax shares
        _case("high_mlp_reuse", module="mlp", hidden=2560, unmerge="shares", first=1),
        # a portrait image: a grid that is no power of two, cut into 4 x 4 regions of 18 x 14 = 252 tokens
        _case("portrait_interval", grid_h=72, grid_w=56, tile_h=18, tile_w=14, steps=5),
        # image-wide merge under the 10/5 schedule: the paper's default variant
        _case("global_10_5", global_merge=True, first=5, steps=5, reuse=10, weight_reuse=5),
        # joint attention of a DiT: 4096 image tokens, 512 text tokens that are never merged, head_dim 128
        _case("joint_reuse", batch=1, dim=3072, heads=24, extra=512, first=1),
        _case("joint_refresh", batch=1, dim=3072, heads=24, extra=512),
        # 16384 tokens, batch 4, one reuse interval: the largest
        _case("large_interval", batch=4, grid_h=128, grid_w=128, steps=5),
        # the same tokens in regions of 32 x 32, the largest region there is: long greedy selections
        _case("large_tiles_refresh", batch=4, grid_h=128, grid_w=128, tile_h=32, tile_w=32),
    ]


def draw(rng):
    """One more block of the same ranges: 256 to 16384 tokens, regions of 16 to 1024 tokens of any shape."""
    while True:
        pick = rng.random()
        dtype = "f32" if rng.random() < 0.12 else "bf16"
        if rng.random() < 0.45:  # regions whose sides are powers of two, squares and stripes
            tile_h, tile_w = rng.choice([(8, 8), (16, 16), (8, 16), (32, 32), (4, 32), (16, 32), (4, 64), (32, 8)])
        else:                    # any other region: what divides an image of another aspect ratio
            tile_h, tile_w = rng.randint(4, 28), rng.randint(4, 28)
        tokens = 2.0 ** rng.uniform(8, 14)
        aspect = 2.0 ** rng.uniform(-0.8, 0.8)
        tiles_y = max(1, round(math.sqrt(tokens * aspect) / tile_h))
        tiles_x = max(1, round(math.sqrt(tokens / aspect) / tile_w))
        wide = rng.random() < 0.3
        head_dim = 128 if wide else 64
        heads = rng.randint(6, 24) if wide else rng.randint(4, 24)
        module = "attention" if pick < 0.7 else "proj" if pick < 0.85 else "mlp"
        first, steps, reuse, weight_reuse = rng.choice([(0, 1, 5, 0), (1, 1, 5, 0), (0, 5, 5, 0), (0, 5, 5, 0), (5, 5, 10, 5)])
        case = _case("", module=module, dtype=dtype, batch=rng.randint(1, 4), grid_h=tiles_y * tile_h, grid_w=tiles_x * tile_w,
                     dim=heads * head_dim, heads=heads, tile_h=tile_h, tile_w=tile_w,
                     ratio=rng.choice([0.25, 0.5, 0.5, 0.75, round(rng.uniform(0.2, 0.8), 2)]),
                     extra=rng.choice([77, 256, 512]) if wide else 0, hidden=4 * heads * head_dim if module == "mlp" else 0,
                     global_merge=rng.random() < 0.12, unmerge="shares" if rng.random() < 0.15 else "transpose",
                     first=first, steps=steps, reuse=reuse, weight_reuse=weight_reuse)
        del case["name"]
        n_loc, n = tile_h * tile_w, case["grid_h"] * case["grid_w"]
        if not 16 <= n_loc <= 1024 or not 256 <= n <= 16384:
            continue
        if case["global_merge"] and n > 4608:  # image-wide weights of larger images do not pay in anybody's loop
            continue
        # no more work than the largest listed case, counting an fp32 operation as the many bf16 ones it takes the time of
        if work(case)["flops"] * (60 if dtype == "f32" else 3 if case["global_merge"] else 1) > work(_LARGEST)["flops"]:
            continue
        return case


_LARGEST = next(c for c in listed() if c["name"] == "large_interval")


def _dest_per_tile(case):
    n_loc = case["tile_h"] * case["tile_w"]
    return n_loc - int(math.floor(torch.tensor(case["ratio"], dtype=torch.float32).item() * n_loc + 0.5))


def _tokens(case, gen):
    """[batch][image tokens + text tokens][dim] fp32: a smooth field plus noise per image token, N(0,1) text tokens."""
    b, h, w, d = case["batch"], case["grid_h"], case["grid_w"], case["dim"]
    nodes = torch.randn(b, d, h // LATTICE + 2, w // LATTICE + 2, generator=gen, device="cuda")
    ys = torch.arange(h, device="cuda") / LATTICE
    xs = torch.arange(w, device="cuda") / LATTICE
    y0, x0 = ys.floor().long(), xs.floor().long()
    fy, fx = (ys - y0)[:, None], (xs - x0)[None, :]
    rows0, rows1 = nodes[:, :, y0], nodes[:, :, y0 + 1]
    field = (1 - fy) * ((1 - fx) * rows0[..., x0] + fx * rows0[..., x0 + 1]) + fy * ((1 - fx) * rows1[..., x0] + fx * rows1[..., x0 + 1])
    image = field.permute(0, 2, 3, 1).reshape(b, h * w, d).contiguous()
    image = image + NOISE * torch.randn(image.shape, generator=gen, device="cuda")
    if not case["extra"]:
        return image
    return torch.cat([image, torch.randn(b, case["extra"], d, generator=gen, device="cuda")], dim=1)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    desc = toma.make_desc(batch=case["batch"], grid_h=case["grid_h"], grid_w=case["grid_w"], dim=case["dim"], tile_h=case["tile_h"],
                          tile_w=case["tile_w"], merge_ratio=case["ratio"], tau=0.1, n_heads=case["heads"],
                          head_dim=case["dim"] // case["heads"], dtype=case["dtype"], reuse_interval=case["reuse"],
                          weight_reuse_interval=case["weight_reuse"], n_extra=case["extra"], global_merge=case["global_merge"],
                          unmerge_mode=case["unmerge"])
    dtype = toma.torch_dtype(desc)
    state = dict(desc=desc, module=case["module"], first=case["first"], idx=toma.alloc_idx(desc), w=toma.alloc_weights(desc).zero_(),
                 ws=toma.alloc_workspace(desc), status=torch.zeros(1, dtype=torch.int32, device="cuda"), dtype=dtype, x=[], out=[])
    d, f = case["dim"], case["hidden"]

    def weight(rows, cols):
        return (torch.randn(rows, cols, generator=gen, device="cuda") / math.sqrt(rows)).to(dtype)

    state["params"] = [weight(d, d) for _ in range(4)] if case["module"] == "proj" else [weight(d, f), weight(f, d)] if f else []
    tokens = _tokens(case, gen)
    if case["first"] > 0:  # the steps before this pass have left their destinations and weights
        x = tokens.to(dtype)
        _step(state, 0, x, torch.empty_like(x))
        tokens = tokens + DRIFT * torch.randn(tokens.shape, generator=gen, device="cuda")
    for t in range(case["steps"]):
        if t > 0:
            tokens += DRIFT * torch.randn(tokens.shape, generator=gen, device="cuda")
        state["x"].append(tokens.to(dtype))
        state["out"].append(torch.empty_like(state["x"][-1]))
    return state


def _step(state, step, x, out):
    args = (state["idx"], state["w"], state["ws"], state["status"])
    if state["module"] == "proj":
        toma.toma_block_proj(state["desc"], step, x, *state["params"], out, *args)
    elif state["module"] == "mlp":
        toma.toma_block_mlp(state["desc"], step, x, *state["params"], out, *args)
    else:
        toma.toma_block(state["desc"], step, x, out, *args)


def run(state):
    for t, (x, out) in enumerate(zip(state["x"], state["out"])):
        _step(state, state["first"] + t, x, out)
    # every step's output, and what the block keeps: destinations, merge weights (as stored), the device's status word
    return {"out": state["out"], "idx": state["idx"], "w": state["w"].view(state["dtype"]), "status": state["status"]}


def work(case):
    b, d, n_loc, d_loc = case["batch"], case["dim"], case["tile_h"] * case["tile_w"], _dest_per_tile(case)
    n = case["grid_h"] * case["grid_w"]
    dests = n // n_loc * d_loc
    merged = b * (dests + case["extra"])              # rows the wrapped module sees
    pairs = b * n * (dests if case["global_merge"] else d_loc)  # (source, destination) pairs with a weight
    esz = 4 if case["dtype"] == "f32" else 2
    planes = 1 if case["unmerge"] == "transpose" else 2
    period = case["weight_reuse"] or case["reuse"]
    flops = nbytes = 0
    for step in range(case["first"], case["first"] + case["steps"]):
        if step % case["reuse"] == 0:
            flops += 2 * b * n * n_loc * d + 2 * b * n * n_loc  # similarities and the gains of the first pick
        if step % period == 0:
            flops += 2 * pairs * d
        flops += 4 * pairs * d                                  # merge and unmerge
        if case["module"] == "mlp":
            flops += 4 * merged * d * case["hidden"]
        else:
            flops += 4 * merged * (dests + case["extra"]) * d
            flops += 8 * merged * d * d if case["module"] == "proj" else 0
        nbytes += 2 * b * (n + case["extra"]) * d * esz         # tokens in, tokens out
    # the weights that the steps share are read or written once, and so are the module's parameters
    nbytes += 4 * pairs * planes + 4 * b * dests
    nbytes += esz * (2 * d * case["hidden"] if case["module"] == "mlp" else 4 * d * d if case["module"] == "proj" else 0)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Destinations are exact: the selection is defined in integers.  bf16 tokens carry 8 significant bits through merge,
    # module and unmerge.  fp32: a logit of some hundreds rounds by 3e-5, which is the relative error of a weight.
    return {"rel": 5e-5, "max": 2e-3, "differ": 0.0} if case["dtype"] == "f32" else {"rel": 1e-2, "max": 0.1, "differ": 0.0}
