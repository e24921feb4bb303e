"""The framework's work as its users have it done, as cases that can be timed and checked.

Three kinds of work, all through the public entry points of `paper_2305_02299_b200.binding`:

  linear   one condensed layer forward (cfi_forward).  Layer shapes are the ViT-B/16 MLP linears (768 <-> 3072) and the
           4096 x 4096 layers of the repository's workloads, at the sparsities of its sweep (80 .. 99 %); the batch runs
           from one request to a training-size batch of tokens; fp32 or bf16 storage, with or without the exact GELU, with
           ablated neurons, and with odd widths.
  stack    a chain of layers (cfi_stack_forward): the MLP blocks of a transformer, up with GELU and down without.  With
           "compact" the hidden layer is in the paper's compact output form (cfi_compact_producer / cfi_compact_consumer:
           ablated neurons are removed altogether), so that its width is whatever number of neurons is left.
  update   one SRigL mask update of a layer in training (cfi_srigl_update).
  pack     the packing of a trained layer into the condensed arrays that a layer is created from (cfi_pack_device).

Weights ~ N(0, 1/k) on k distinct uniform columns per row, bias ~ N(0, 0.01), x ~ N(0, 1): the distributions of the
repository's own inputs.  Layers are created with every device layout unless "layouts" says otherwise.
"""
import math

import torch

from paper_2305_02299_b200 import binding as cfi

ALL, ONLINE, NO_DENSE = 7, 1, 3  # every layout; the small-batch one alone; the condensed ones without the dense copy


def _linear(name, inn, out, k, batch, dtype="f32", act="none", ablated=0, layouts=ALL):
    return {"name": name, "kind": "linear", "in": inn, "out": out, "k": k, "ablated": ablated, "batch": batch, "dtype": dtype,
            "act": act, "layouts": layouts}


def _stack(name, blocks, d_model, d_hidden, k_up, k_down, abl_up, abl_down, batch, dtype, compact=False, layouts=ALL):
    return {"name": name, "kind": "stack", "blocks": blocks, "d_model": d_model, "d_hidden": d_hidden, "k_up": k_up, "k_down": k_down,
            "abl_up": abl_up, "abl_down": abl_down, "batch": batch, "dtype": dtype, "compact": compact, "layouts": layouts}


def _update(name, out, inn, k, ablated, swap, gamma):
    return {"name": name, "kind": "update", "out": out, "in": inn, "k": k, "ablated": ablated, "swap": swap, "gamma": gamma}


def _pack(name, out, inn, k, ablated):
    return {"name": name, "kind": "pack", "out": out, "in": inn, "k": k, "ablated": ablated}


def listed():
    return [
        # Online inference, one request: a single layer call, and all MLP layers of a ViT-B/16 in one call.
        _linear("vit_up_f32_b1", 768, 3072, 77, 1),
        _linear("sq4096_s80_f32_b1", 4096, 4096, 819, 1, layouts=ONLINE),
        _stack("vit_mlp24_f32_b1", 12, 768, 3072, 77, 307, 0, 0, 1, "f32"),
        # A few requests served together on a very sparse wide layer.
        _linear("sq4096_s95_f32_b16", 4096, 4096, 205, 16),
        # The batch the paper's GPU figure uses: ViT-B/16's first MLP layer, and a wide layer.
        _linear("vit_up_f32_b256", 768, 3072, 77, 256),
        _linear("sq4096_s90_f32_b256", 4096, 4096, 410, 256),
        # The tokens of eight images through a layer with ablated neurons.
        _linear("vit_down_f32_b1576", 3072, 768, 307, 1576, ablated=77),
        # The tokens of one image through one block in the compact form: its hidden layer keeps 2918 of 3072 neurons.
        _stack("vit_block_compact_bf16_b197", 1, 768, 3072, 77, 307, 154, 38, 197, "bf16", compact=True),
        # A training-size batch (256 images x 197 tokens) through the 24 MLP layers in bf16: the largest.
        _stack("vit_mlp24_bf16_b50432", 12, 768, 3072, 77, 307, 154, 38, 50432, "bf16"),
        # Mask updates in training, early in the schedule (30 % of the weights swapped), and the packing of a layer.
        _update("srigl_3072x768", 3072, 768, 77, 154, 0.3, 0.3),
        _update("srigl_4096x4096", 4096, 4096, 819, 0, 0.3, 0.3),
        _pack("pack_3072x768", 3072, 768, 77, 154),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """Mostly widths as networks have them, one in four whatever number comes up."""
    w = _log(rng, lo, hi)
    return w if rng.random() < 0.25 else max(lo, w // 64 * 64)


def _fan_in(rng, inn):
    return max(1, int(round((1.0 - rng.uniform(0.80, 0.99)) * inn)))


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "linear", "stack", "stack", "update", "pack"])
    if kind == "linear":
        inn, out = _width(rng, 256, 4096), _width(rng, 256, 4096)
        batch = _log(rng, 1, 4096)
        layouts = rng.choice([ALL, ALL, ALL, ONLINE if batch <= 8 else NO_DENSE if batch <= 256 else ALL])
        c = _linear("", inn, out, _fan_in(rng, inn), batch, rng.choice(["f32", "f32", "bf16"]), rng.choice(["none", "gelu"]),
                    int(out * rng.choice([0.0, 0.05, 0.10])), layouts)
    elif kind == "stack":
        d, h = _width(rng, 256, 1024), _width(rng, 512, 4096)
        compact, dtype = rng.random() < 0.4, rng.choice(["f32", "bf16"])
        c = _stack("", rng.randint(1, 2 if compact else 4), d, h, _fan_in(rng, d), 0, int(h * rng.uniform(0.0, 0.1)),
                   int(d * rng.uniform(0.0, 0.1)), _log(rng, 1, 4096 if compact or dtype == "f32" else 16384), dtype, compact)
        c["k_down"] = _fan_in(rng, h - c["abl_up"] if compact else h)
    else:
        out, inn = _width(rng, 256, 4096), _width(rng, 256, 4096)
        k, ablated = _fan_in(rng, inn), int(out * rng.choice([0.0, 0.05, 0.10]))
        c = _pack("", out, inn, k, ablated) if kind == "pack" else _update("", out, inn, k, ablated, rng.uniform(0.02, 0.3), rng.choice([0.3, 0.3, 0.95]))
    del c["name"]
    return c


def _specs(case):
    """(in, out, k, ablated, act) of each layer as it is trained, full width."""
    if case["kind"] == "stack":
        up = (case["d_model"], case["d_hidden"], case["k_up"], case["abl_up"], "gelu")
        down = (case["d_hidden"], case["d_model"], case["k_down"], case["abl_down"], "none")
        return [up, down] * case["blocks"]
    return [(case["in"], case["out"], case["k"], case["ablated"], case["act"])]


def _rand(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17)


def _structure(gen, inn, out, k, ablated):
    """Rows that are left (ascending) and k distinct columns for each of them, uniform, ascending."""
    rows = torch.randperm(out, generator=gen, device="cuda")[ablated:].sort().values
    cols = torch.rand((rows.numel(), inn), generator=gen, device="cuda").topk(k, dim=1, sorted=False).indices
    return rows.to(torch.int32), cols.sort(dim=1).values.to(torch.int32)


def _layer_arrays(gen, inn, out, k, ablated):
    rows, cols = _structure(gen, inn, out, k, ablated)
    values = torch.randn(cols.shape, generator=gen, device="cuda") / math.sqrt(k)
    bias = 0.1 * torch.randn(out, generator=gen, device="cuda")
    return [t.cpu().numpy() for t in (values, cols, rows, bias)]


def _x(gen, case, width):
    x = torch.randn((case["batch"], width), generator=gen, device="cuda")
    return x.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)


def _condensed(case, gen):
    """(values, indices, rows, bias, in, out, act) of each layer that is created."""
    layers = [list(_layer_arrays(gen, *s[:4])) + [s[0], s[1], s[4]] for s in _specs(case)]
    if case.get("compact"):
        # Each block's hidden layer drops its ablated neurons; what they emitted goes into the next layer's bias.
        for up, down in zip(layers[0::2], layers[1::2]):
            const = torch.nn.functional.gelu(torch.from_numpy(up[3]).double()).to(torch.float32)
            if case["dtype"] == "bf16":
                const = const.to(torch.bfloat16).to(torch.float32)
            down[0], down[1], down[3] = cfi.cfi_compact_consumer(up[2], up[5], const.numpy(), down[0], down[1], down[2], down[3])
            down[4] = up[2].shape[0]
            up[3], up[2] = cfi.cfi_compact_producer(up[3], up[2], up[5])
            up[5] = up[2].shape[0]
    return layers


def prepare(case, seed):
    gen = _rand(seed)
    if case["kind"] in ("update", "pack"):
        rows, cols = _structure(gen, case["in"], case["out"], case["k"], case["ablated"])
        mask = torch.zeros((case["out"], case["in"]), dtype=torch.uint8, device="cuda")
        mask[rows.long().unsqueeze(1), cols.long()] = 1
        w = torch.randn(mask.shape, generator=gen, device="cuda") / math.sqrt(case["k"]) * mask
        if case["kind"] == "pack":
            return {"case": case, "w": w, "mask": mask}
        grad = 1e-3 * torch.randn(mask.shape, generator=gen, device="cuda")
        return {"case": case, "w0": w, "mask0": mask, "grad": grad, "w": w.clone(), "mask": mask.clone(),
                "K": int(case["swap"] * rows.numel() * case["k"])}
    layers = [cfi.cfi_create(v, ix, rows, b, inn, out, dtype=case["dtype"], act=act, layouts=case["layouts"])
              for v, ix, rows, b, inn, out, act in _condensed(case, gen)]
    x = _x(gen, case, layers[0].in_features)
    y = torch.empty((case["batch"], layers[-1].out_features), dtype=x.dtype, device="cuda")
    state = {"case": case, "layers": layers, "x": x, "y": y}
    if case["kind"] == "stack":
        state["stack"] = cfi.cfi_stack_create(layers, case["batch"])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "linear":
        cfi.cfi_forward(state["layers"][0], state["x"], state["y"], case["batch"])
        return state["y"]
    if case["kind"] == "stack":
        cfi.cfi_stack_forward(state["stack"], state["x"], state["y"], case["batch"])
        return state["y"]
    if case["kind"] == "pack":
        return cfi.cfi_pack_device(state["w"], state["mask"])
    # The update works in place.  A training loop's optimiser writes new weights before each update; here the same
    # weights are put back, so that every pass is an update of a trained layer and not of the last update's result.
    w, mask = state["w"], state["mask"]
    w.copy_(state["w0"])
    mask.copy_(state["mask0"])
    k_new, n_active = cfi.cfi_srigl_update(w, mask, state["grad"], state["K"], case["gamma"])
    return w, mask, k_new, n_active


def work(case):
    if case["kind"] == "update":  # w, mask and gradient read, w and mask written
        return {"bytes": 14 * case["out"] * case["in"], "flops": 0}
    if case["kind"] == "pack":  # the mask and the kept weights read, the condensed arrays written
        return {"bytes": case["out"] * case["in"] + 12 * (case["out"] - case["ablated"]) * case["k"], "flops": 0}
    es = 2 if case["dtype"] == "bf16" else 4
    specs = _specs(case)
    total, flops = case["batch"] * (specs[0][0] + specs[-1][1]) * es, 0
    for _, out, k, ablated, _ in specs:
        nnz = (out - ablated) * k
        total += nnz * (es + 4) + 4 * out
        flops += 2 * case["batch"] * nnz
    return {"bytes": total, "flops": flops}


def tolerance(case):
    if case["kind"] in ("update", "pack"):
        return "exact"  # selections and copies
    if case["dtype"] == "bf16":
        # bf16 results: an element whose sum falls on the other side of a rounding boundary moves by one unit in the last
        # place, and a chain carries that on.
        return {"rel": 0.008, "max": 0.1} if case["kind"] == "stack" else {"rel": 0.002, "max": 0.016}
    return {"rel": 1e-5, "max": 1e-4}  # sums of fp32 products in another order (up to 4e-6 from 64 bits over 4096 columns)


def exact(case, seed):
    if case["kind"] in ("update", "pack"):
        return None  # whole numbers and copies: compared bit for bit
    gen = _rand(seed)
    specs = _specs(case)
    layers = [_layer_arrays(gen, *s[:4]) for s in specs]  # full width: the compact form computes the same
    bf16 = case["dtype"] == "bf16"
    h = _x(gen, case, specs[0][0]).double()
    for i, ((v, ix, rows, b), (inn, out, _, _, act)) in enumerate(zip(layers, specs)):
        values = torch.from_numpy(v).cuda()
        if bf16:  # stored in bf16, as the layer's type says
            values = values.to(torch.bfloat16)
        w = torch.zeros((out, inn), dtype=torch.float64, device="cuda")
        w[torch.from_numpy(rows).cuda().long().unsqueeze(1), torch.from_numpy(ix).cuda().long()] = values.double()
        h = h @ w.t() + torch.from_numpy(b).cuda().double()
        if act == "gelu":
            h = torch.nn.functional.gelu(h)
        if bf16 and i + 1 < len(layers):  # what one layer hands to the next is stored in bf16 too
            h = h.to(torch.bfloat16).double()
    return h
