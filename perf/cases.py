"""Workloads of the AlexNet library for timing, as a training or evaluation program calls it.

A case is one pass through the public entry points of `paper_1412_2302_b200.alexnet`:

  train      load_batch_async + train_step + loss_async: one SGD step on a fresh minibatch (the load of a pass overlaps the
             step of the pass before it, through the handle's two batch slots)
  gradients  load_batch_async + forward_backward + apply_update + loss_async: the step in its data-parallel form, where the
             gradient is complete in memory before it is applied
  replicas   two replicas in one GPU memory, each with a minibatch of its own, and their exchange-and-average:
             `literal` = two train_steps, then replica_average; `one_pass` = two forward_backwards, then
             update_and_average; `shared` = the same with one copy of the parameters
  evaluate   eval_batch: forward pass on the centre crops, top-1 / top-5 counts and loss, synchronous
  bias_grad  bias_grad_noalloc: the bias gradient of one layer for a caller that cannot allocate

Ranges: minibatches of 4 to 512 images for training, 8 to 192 per replica for two replicas, 1 to 512 for evaluation; images
in pinned host memory (a loader's ring) or already on the GPU; training with and without the update fused into the FC weight
gradients, plain or inverted dropout, with and without the intensity augmentation.
"""
import math

import torch

from paper_1412_2302_b200 import synth
from paper_1412_2302_b200.alexnet import (FLAG_FUSED_FC_UPDATE, FLAG_INVERTED_DROPOUT, FLAG_SHARED_REPLICA_WEIGHTS, AlexNet,
                                          bias_grad_noalloc)

PARAMS = 60_965_224
CROP_BYTES = 227 * 227 * 3                  # what a pass needs of each 256 x 256 x 3 image
MEAN_BYTES = 4 * 256 * 256 * 3
TRAIN_FLOPS = 4.1356e9                      # per image: forward, backward-data without conv1, backward-weight
FORWARD_FLOPS = 1.4488e9                    # per image
FORMS = ("literal", "one_pass", "shared")


def _train(kind, batch, source, fused, inverted, augment):
    return {"kind": kind, "batch": batch, "source": source, "fused": fused, "inverted": inverted, "augment": augment}


def listed():
    return [
        # the smallest call: a layer's bias gradient (13 x 13 layers of 384 channels at batch 128, on their 14 x 14 grid)
        {"name": "bias_grad_25088x384", "kind": "bias_grad", "rows": 25088, "channels": 384},
        # one picture at a time, where the answer is waited for
        {"name": "evaluate_1", "kind": "evaluate", "batch": 1, "source": "host"},
        # a validation set in batches of an ordinary and of a large size
        {"name": "evaluate_100", "kind": "evaluate", "batch": 100, "source": "host"},
        {"name": "evaluate_256", "kind": "evaluate", "batch": 256, "source": "host"},
        # fine tuning with a small minibatch: the parameters' traffic and the launches count
        dict(_train("train", 8, "host", True, False, False), name="train_8"),
        # one step of the small configuration of the tests
        dict(_train("train", 32, "host", True, False, False), name="train_32"),
        # a batch size that fills no tile, with the options of later practice
        dict(_train("train", 100, "host", True, True, True), name="train_100_inverted_augmented"),
        # the paper's minibatch: the benchmark's workload
        dict(_train("train", 128, "host", True, False, False), name="train_128"),
        # a handle with default flags (every gradient stays readable)
        dict(_train("train", 256, "host", False, False, False), name="train_256_default"),
        # a large minibatch, the data set resident in GPU memory
        dict(_train("train", 512, "device", True, False, False), name="train_512_resident"),
        # the step of a rank of a data-parallel job
        dict(_train("gradients", 128, "host", False, False, False), name="gradients_128"),
        # the paper's two replicas
        {"name": "replicas_128", "kind": "replicas", "batch": 128, "source": "host", "form": "literal"},
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("train", "train", "train", "train", "evaluate", "evaluate", "gradients", "replicas", "bias_grad"))
    source = rng.choice(("host", "host", "device"))
    if kind == "evaluate":
        return {"kind": kind, "batch": _log_uniform(rng, 1, 512), "source": source}
    if kind == "replicas":
        return {"kind": kind, "batch": _log_uniform(rng, 8, 192), "source": source, "form": rng.choice(FORMS)}
    if kind == "bias_grad":
        return {"kind": kind, "rows": _log_uniform(rng, 128, 200000), "channels": 8 * _log_uniform(rng, 12, 512 if rng.random() < 0.3 else 48)}
    batch = _log_uniform(rng, 4, 512)
    if kind == "gradients":
        return _train(kind, batch, source, False, rng.random() < 0.3, False)
    return _train(kind, batch, source, rng.random() < 0.7, rng.random() < 0.3, rng.random() < 0.3)


def _minibatch(gen, batch, source):
    """uint8 images and int32 labels, where a program has them before the load."""
    img = torch.randint(0, 256, (batch, 256, 256, 3), dtype=torch.uint8, device="cuda", generator=gen)
    lab = torch.randint(0, 1000, (batch,), dtype=torch.int32, device="cuda", generator=gen)
    if source == "device":
        return img, lab
    himg, hlab = torch.empty(img.shape, dtype=torch.uint8, pin_memory=True), torch.empty(lab.shape, dtype=torch.int32, pin_memory=True)
    himg.copy_(img)
    hlab.copy_(lab)
    return himg, hlab


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    if kind == "bias_grad":
        dy = torch.randn((case["rows"], case["channels"]), device="cuda", generator=gen).to(torch.bfloat16)
        return {"kind": kind, "dy": dy, "db": torch.empty(case["channels"], device="cuda")}
    flags, replicas = 0, 1
    if kind == "replicas":
        replicas = 2
        flags = {"literal": FLAG_FUSED_FC_UPDATE, "one_pass": 0, "shared": FLAG_SHARED_REPLICA_WEIGHTS}[case["form"]]
    elif kind != "evaluate":
        flags = (FLAG_FUSED_FC_UPDATE if case["fused"] else 0) | (FLAG_INVERTED_DROPOUT if case["inverted"] else 0)
    net = AlexNet(batch=case["batch"], replicas=replicas, seed=int(seed), init_std=0.01, flags=flags, mean_image=synth.mean_image(int(seed)))
    if case.get("augment"):
        # principal components of the colours of natural images: grey first, then the two differences
        net.set_color_augmentation([[0.58, 0.72, 0.40], [0.58, 0.00, -0.82], [0.58, -0.69, 0.42]], [55.0, 4.8, 1.2], 0.1)
    state = {"kind": kind, "form": case.get("form"), "net": net, "step": 0,
             "batches": [_minibatch(gen, case["batch"], case["source"]) for _ in range(replicas)]}
    if kind != "evaluate":
        state["views"] = [net.param_views(r) for r in range(replicas)]
        # gradients are an output of every pass that leaves them readable
        state["with_g"] = kind == "gradients" or (kind == "train" and not case["fused"]) or case.get("form") in ("one_pass", "shared")
        state["loss"] = torch.zeros(replicas, dtype=torch.float32, pin_memory=True)
    torch.cuda.synchronize()
    return state


def run(state):
    kind = state["kind"]
    if kind == "bias_grad":
        bias_grad_noalloc(state["dy"], state["db"])
        return state["db"]
    net, step = state["net"], state["step"]
    if kind == "evaluate":
        return net.eval_batch(0, *state["batches"][0])
    state["step"] = step + 1
    for r, (images, labels) in enumerate(state["batches"]):
        net.load_batch_async(r, images, labels, step)
    loss = state["loss"]
    for r in range(len(state["batches"])):
        if kind == "train" or state["form"] == "literal":
            net.train_step(r)
        else:
            net.forward_backward(r)
        net.loss_async(r, loss[r:r + 1])
    if kind == "gradients":
        net.apply_update(0, 1.0)
    elif state["form"] == "literal":
        net.replica_average()
    elif state["form"] is not None:
        net.update_and_average()
    out = {"loss": loss}
    for r, (w, v, g) in enumerate(state["views"]):
        out["w%d" % r], out["v%d" % r] = w, v
        if state["with_g"]:
            out["g%d" % r] = g
    return out


def work(case):
    if case["kind"] == "bias_grad":
        n = case["rows"] * case["channels"]
        return {"bytes": 2 * n + 4 * case["channels"], "flops": n}
    images = case["batch"] * CROP_BYTES + MEAN_BYTES
    if case["kind"] == "evaluate":
        return {"bytes": 4 * PARAMS + images, "flops": FORWARD_FLOPS * case["batch"]}
    if case["kind"] == "replicas":
        # both replicas' parameters and momentum in and out, and the gradients where they stay readable; one copy when shared
        per = {"literal": 32, "one_pass": 40, "shared": 24}[case["form"]]
        return {"bytes": per * PARAMS + 2 * images, "flops": 2 * TRAIN_FLOPS * case["batch"]}
    # parameters and momentum in and out; the gradient where it stays readable
    per = 20 if case["kind"] == "gradients" or not case["fused"] else 16
    return {"bytes": per * PARAMS + images, "flops": TRAIN_FLOPS * case["batch"]}


def tolerance(case):
    if case["kind"] == "bias_grad":
        return {"rel": 1e-5}                # bf16 inputs, 32-bit sums
    # bf16 operands and activations between 32-bit sums; the counts of an evaluation are whole numbers
    return {"rel": 1e-2}
