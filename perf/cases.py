"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one of the four ways into the path, on one of the five configurations of ``synth.CONFIGS``:

* ``step``: one fine-tuning step on device buffers (``Engine.train_step``);
* ``host``: the same step fed from pinned host memory (``Engine.train_step_host``), as an input pipeline feeds it;
* ``loop``: a run of steps with the cosine schedule evaluated on the device (``Engine.train_steps``);
* ``eval``: inference with the same token dropping (``Engine.eval_forward``).

The options are those of the method: which blocks train (the last ones, or the paper's 4th, 8th and 12th), how many
tokens every drop location keeps, how dropped tokens are fused, AdamW or SGD, the 8-bit gradient-free prefix.  Batch
sizes run from one image (on-device use: latency) to the largest batch of the configuration's own benchmark (twice that
for the small model), odd ones included.

Weights and images are drawn on the GPU by the recipe of ``synth``, with what training puts into a ViT on top of it:
images have salient patches and kinds of content, the classification token attends to the salient ones, routers know
the kinds of content.  (With plain random weights the scores around the K-th are equal to within their rounding, and
which tokens a step keeps is a matter of the order of its sums.)  A program keeps an engine with its weights, its input
buffers and its loss buffer, and runs on a stream of its own, as ``bench.py`` does.
"""
import math

import torch

from paper_2405_10951_b200 import binding, synth

PAPER_BLOCKS = "3,7,11"          # the paper's choice: 4th, 8th and 12th block
LOOP_STEPS = 4
LR = 1e-5                        # a fine-tuning rate


def listed():
    return [
        # headline workload of the benchmark: last four blocks of ViT-B, batch 128
        dict(name="vit_b_step_128", way="step", model="vit_b", batch=128, trainable="8,9,10,11", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
        # the paper's ViT-B recipe (SGD, batch 32, its trainable blocks and drop rate) fed from host memory
        dict(name="vit_b_host_sgd_32", way="host", model="vit_b", batch=32, trainable=PAPER_BLOCKS, keep=0.5, fuse=1, optimizer="sgd", fp8=False),
        # the small model at its benchmark batch
        dict(name="deit_s_step_64", way="step", model="deit_s", batch=64, trainable="8,9,10,11", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
        # the paper's DeiT-S recipe: AdamW, batch 128, blocks 4, 8 and 12, half the tokens dropped
        dict(name="deit_s_paper_128", way="step", model="deit_s", batch=128, trainable=PAPER_BLOCKS, keep=0.5, fuse=1, optimizer="adamw", fp8=False),
        # on-device fine-tuning one image at a time: latency and launches
        dict(name="deit_s_step_1", way="step", model="deit_s", batch=1, trainable="8,9,10,11", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
        # long sequences (384 px, 577 tokens) at the benchmark batch
        dict(name="vit_b_384_step_32", way="step", model="vit_b_384", batch=32, trainable="10,11", keep=0.5, fuse=1, optimizer="adamw", fp8=False),
        # long sequences with the paper's trainable blocks, an odd batch, weighted-mean fusion
        dict(name="vit_b_384_paper_7", way="step", model="vit_b_384", batch=7, trainable=PAPER_BLOCKS, keep=0.5, fuse=2, optimizer="adamw", fp8=False),
        # mixture of experts, two tasks
        dict(name="moe_vit_s_step_64", way="step", model="moe_vit_s", batch=64, trainable="8,9,10,11", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
        # 8-bit gradient-free prefix, an odd batch, dropped tokens not fused
        dict(name="vit_b_fp8_step_45", way="step", model="vit_b", batch=45, trainable="8,9,10,11", keep=0.7, fuse=0, optimizer="adamw", fp8=True),
        # inference over a large batch, and of a single image
        dict(name="vit_b_eval_128", way="eval", model="vit_b", batch=128, trainable="8,9,10,11", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
        dict(name="deit_s_eval_1", way="eval", model="deit_s", batch=1, trainable="8,9,10,11", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
        # the float32 configuration, a run of steps in one call
        dict(name="tiny_fp32_loop_8", way="loop", model="tiny_fp32", batch=8, trainable="4,5", keep=0.7, fuse=1, optimizer="adamw", fp8=False),
    ]


# Largest batch of a configuration.
MAX_BATCH = {"tiny_fp32": 32, "deit_s": 128, "vit_b": 128, "vit_b_384": 32, "moe_vit_s": 64}


def draw(rng):
    model = rng.choice(["deit_s", "deit_s", "vit_b", "vit_b", "vit_b_384", "moe_vit_s", "tiny_fp32"])
    way = rng.choice(["step", "step", "step", "host", "loop", "eval", "eval"])
    if model == "tiny_fp32":
        trainable = rng.choice(["4,5", "2,3,4,5", "1,3,5"])
    else:
        trainable = rng.choice(["8,9,10,11", "10,11", PAPER_BLOCKS])
    case = dict(way=way, model=model, batch=1, trainable=trainable, keep=rng.choice([0.3, 0.5, 0.7]), fuse=rng.choice([0, 1, 1, 2]),
                optimizer=rng.choice(["adamw", "adamw", "sgd"]), fp8=model == "vit_b" and rng.random() < 0.25)
    batch = int(round(math.exp(rng.uniform(0.0, math.log(MAX_BATCH[model])))))
    most = max(_cost(c) for c in listed())
    while True:
        case["batch"] = batch
        if batch == 1 or _cost(case) <= most:
            return case
        batch -= 1 + batch // 8


def _cost(case):
    """Seconds at round figures for the card's bf16 and memory rates."""
    w = work(case)
    return max(w["flops"] / 1.6e15, w["bytes"] / 6.5e12)


def _config(case):
    keep = {0.3: (3, 10), 0.5: (1, 2), 0.7: (7, 10)}[case["keep"]]
    return synth.CONFIGS[case["model"]].with_(
        batch=case["batch"], trainable=tuple(int(t) for t in case["trainable"].split(",")), keep_num=keep[0], keep_den=keep[1],
        fuse_mode=case["fuse"], optimizer=case["optimizer"], frozen_fp8=int(case["fp8"]), lr=LR)


_stream = None


def _run_stream():
    """The one stream the program runs on (the library replays a step as a CUDA graph on any stream but the default)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _keeps(cfg):
    """Tokens kept at every drop location (K of the method, counted without the classification token)."""
    m, out = cfg.num_patches, []
    for _ in cfg.drop_blocks:
        k = min(m, max(1, -(-cfg.keep_num * m // cfg.keep_den)))
        out.append(k)
        m = k + (1 if cfg.fuse_mode and k < m else 0)
    return out


CONTENTS = 16                    # kinds of patch content
SALIENCE_GAIN, CONTENT_GAIN = 2.0, 6.0


def _directions(cfg, gen):
    """What a trained model has learnt, as directions.  In pixels: the pattern of a salient patch and one pattern per
    kind of content.  In the embedding: the same, and the classification token's own."""
    pin = cfg.in_chans * cfg.patch_size ** 2
    pixels = torch.linalg.qr(torch.randn(pin, 1 + CONTENTS, generator=gen, device="cuda"))[0].T
    features = torch.linalg.qr(torch.randn(cfg.dim, 2 + CONTENTS, generator=gen, device="cuda"))[0].T
    return pixels, features


def _params(cfg, gen, pixels, features):
    """synth's recipe N(0, 0.02^2) within two sigma, plus what training puts on top of it: salient patches and the kinds
    of content have directions in the embedding, the classification token attends to salient patches in every head
    (Eq. 6 ranks by that attention), and a router sends a kind of content to its experts and each task's
    classification token to others."""
    D, H, hd = cfg.dim, cfg.heads, cfg.dim // cfg.heads
    std = 0.02 * math.sqrt(cfg.in_chans * cfg.patch_size ** 2)            # of a patch's embedding, element by element
    salient, cls, content = features[0], features[1], features[2:]
    for name, shape in synth.param_shapes(cfg).items():
        if name.endswith("bias"):
            p = torch.zeros(shape, device="cuda")
        elif "norm" in name and name.endswith("weight"):
            p = torch.ones(shape, device="cuda")
        else:
            u = torch.rand(shape, generator=gen, device="cuda").mul_(0.9545).add_(0.02275)      # uniform between Phi(-2) and Phi(2)
            p = torch.special.ndtri(u).mul_(0.02)
        if name == "patch_embed.weight":
            p += std * (SALIENCE_GAIN * torch.outer(salient, pixels[0]) + CONTENT_GAIN * content.T @ pixels[1:])
        elif name == "cls_token":
            p += math.sqrt(D) * cls
        elif name.endswith("attn.qkv.weight"):
            r = torch.nn.functional.normalize(torch.randn(H, hd, generator=gen, device="cuda"), dim=1).reshape(D)
            p[:D] += math.sqrt(8.0 / D) * torch.outer(r, cls)
            p[D: 2 * D] += math.sqrt(8.0 / D) * torch.outer(r, salient)
        elif name.endswith("moe.gate.weight"):
            E = cfg.moe_experts
            e = torch.arange(E, device="cuda")
            p += 0.5 * (content[e % CONTENTS] + 0.6 * content[(e + 1) % CONTENTS])
            p += (4.0 / math.sqrt(D)) * torch.rand(cfg.num_tasks, E, 1, generator=gen, device="cuda").argsort(1) * cls / 2
        yield name, (p if cfg.dtype == "fp32" else p.bfloat16())


def _images(cfg, gen, lead, pixels):
    """N(0, 1) pixels; every patch shows one kind of content, and patches come in levels of salience, as many to a level
    as the drop locations sort out one after the other."""
    n, P = cfg.num_patches, cfg.patch_size
    g = cfg.image_size // P
    level = torch.zeros(n, device="cuda")
    for k in _keeps(cfg):
        level[:k] += 1.0
    place = torch.rand(lead + (n,), generator=gen, device="cuda").argsort(-1)
    kind = torch.randint(CONTENTS, lead + (n,), generator=gen, device="cuda")
    patches = torch.randn(lead + (n, pixels.shape[1]), generator=gen, device="cuda")
    patches += math.sqrt(cfg.dim) * (level[place].unsqueeze(-1) * pixels[0] / 2 + pixels[1 + kind] / 6)
    x = patches.reshape(lead + (g, g, cfg.in_chans, P, P)).movedim(-3, -5)
    return x.transpose(-2, -3).reshape(lead + (cfg.in_chans, cfg.image_size, cfg.image_size))


def _gradients(cfg, flat):
    """The gradient buffer as one view per trainable tensor (in parameter order, each padded to a multiple of 64), an MoE
    layer's gate and experts in one."""
    views, off = {}, 0
    for name, shape in synth.param_shapes(cfg).items():
        block = int(name.split(".")[1]) if name.startswith("blocks.") else None
        if block in cfg.trainable if block is not None else name.startswith(("norm.", "head.")):
            n = math.prod(shape)
            if ".moe." in name:
                layer = name[: name.index(".moe.") + 4]
                start = views[layer].storage_offset() - flat.storage_offset() if layer in views else off
                views[layer] = flat[start: off + n]
            else:
                views[name] = flat[off: off + n].view(shape)
            off += (n + 63) // 64 * 64
    return views


def prepare(case, seed):
    cfg = _config(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B, way = cfg.batch, case["way"]
    lead = (LOOP_STEPS, B) if way == "loop" else (B,)
    with torch.cuda.stream(_run_stream()):
        eng = binding.Engine(cfg)
        pixels, features = _directions(cfg, gen)
        for name, value in _params(cfg, gen, pixels, features):
            eng.set_param(name, value)
        images = _images(cfg, gen, lead, pixels).to(eng.storage_dtype)
        tasks = None
        classes = torch.full((B,), cfg.num_classes[0], device="cuda")
        if cfg.num_tasks > 1:                            # first half of the batch task 0, second half task 1
            tasks = (torch.arange(B, device="cuda") >= -(-B // 2)).int()
            classes = torch.tensor(cfg.num_classes, device="cuda")[tasks.long()]
        labels = (torch.rand(lead, generator=gen, device="cuda") * classes).int()
        if tasks is not None:
            tasks = tasks.expand(lead).contiguous()
        loss = torch.zeros(LOOP_STEPS if way == "loop" else 1, device="cuda")
        if way == "host":
            images, labels, loss = images.cpu().pin_memory(), labels.cpu().pin_memory(), loss.cpu().pin_memory()
            tasks = tasks.cpu().pin_memory() if tasks is not None else None
        torch.cuda.current_stream().synchronize()
    return {"way": way, "engine": eng, "images": images, "labels": labels, "tasks": tasks, "loss": loss, "grads": _gradients(cfg, eng.grad_buffer())}


def run(state):
    eng = state["engine"]
    with torch.cuda.stream(_run_stream()):
        if state["way"] == "eval":
            return eng.eval_forward(state["images"], state["tasks"], want_kept=False)[0]
        if state["way"] == "host":
            eng.train_step_host(state["images"], state["labels"], state["tasks"], loss=state["loss"])
        elif state["way"] == "loop":
            eng.train_steps(state["images"], state["labels"], state["tasks"], lr_max=LR, lr_min=0.0, total_steps=1000, want_kept=False,
                            out=(state["loss"], None))
        else:
            eng.train_step(state["images"], state["labels"], state["tasks"], want_kept=False, out=(state["loss"], None))
    return {"loss": state["loss"], "grads": state["grads"]}


def work(case):
    """Products of the forward pass at each block's token count; of the trainable blocks twice that again backward, of a frozen
    block in the gradient path once (no weight gradient).  In the last block only the classification row goes on past the
    attention product.  Bytes: images and weights once, and per trainable parameter its gradient, master copy, moments
    and stored copy."""
    cfg = _config(case)
    B, D, F = cfg.batch, cfg.dim, cfg.mlp_hidden
    tokens = cfg.num_patches + 1
    train = case["way"] != "eval"
    patch = cfg.in_chans * cfg.patch_size ** 2
    flops = 2.0 * cfg.num_patches * patch * D
    params = trained = 0
    for l in range(cfg.depth):
        ta = tokens
        if l in cfg.drop_blocks:
            m = tokens - 1
            k = min(m, max(1, -(-cfg.keep_num * m // cfg.keep_den)))
            if k < m:
                tokens = 1 + k + (1 if cfg.fuse_mode else 0)
        tf = tokens
        last = l == cfg.depth - 1 and l not in cfg.drop_blocks
        tp, tf, tq = (1, 1, 1) if last else (ta, tf, ta)
        moe = l in cfg.moe_blocks
        linear = 2.0 * (tq * D * D + ta * 2 * D * D + tp * D * D + tf * 2 * D * F * (cfg.moe_top_k if moe else 1))
        attn = 4.0 * tq * ta * D
        flops += linear + attn
        n = 4 * D * D + 2 * D * F * (cfg.moe_experts if moe else 1)
        params += n
        if train and l >= min(cfg.trainable):
            on = l in cfg.trainable
            flops += (2 if on else 1) * linear + 2 * attn
            trained += n if on else 0
    head = max(cfg.num_classes) * D
    flops += 2.0 * head * (3 if train else 1)
    params += patch * D + head
    trained += head
    es = 4 if cfg.dtype == "fp32" else 2
    image = cfg.in_chans * cfg.image_size ** 2 * es
    steps = LOOP_STEPS if case["way"] == "loop" else 1
    nbytes = B * image + es * params
    if train:                       # gradient written, master copy and moments read and written, stored copy written
        nbytes += trained * (4 + 8 + (16 if cfg.optimizer == "adamw" else 8) + (es if es == 2 else 0))
    return {"bytes": float(steps * nbytes), "flops": float(steps * B * flops)}


def tolerance(case):
    """About four times the largest difference seen, tensor by tensor, against the same step without tensor cores (sums in
    another order, exact erf and exponentials) and after a change of the patch embedding far below its rounding: bf16 and
    the 8-bit prefix 0.3 to 1.1 %, most where a kept token changes places with its equal (single values 14 % of a tensor's
    spread; 29 % where a token's routing tips over), float32 1e-6 and 1.6e-5."""
    if case["model"] == "tiny_fp32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 0.03, "max": 0.9 if case["model"] == "moe_vit_s" else 0.6}
