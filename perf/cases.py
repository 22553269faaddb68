"""The work a user of this library has it do, as cases that can be timed: training a segment over a
resident data set, training it on label rows, training a left segment through the frozen right one,
and computing stored responses.

A case is a dict of plain values:
  task       "epoch"        seg_train_epochs, one pass over the data set (the last batch may be partial)
             "loop"         the caller's own loop over seg_train_step, batch by batch
             "label_input"  a loop over seg_train_step_label_input (the fully separate variant)
             "recover"      a loop over seg_recovery_step, left segment through the frozen right one
             "infer"        seg_forward_dataset through all segments of the network
  net        layer widths, segments separated by "|"
  final      whether the (single) trained segment is the network's last one
  precision, optimizer, batch, samples
  labels     distribution of the intermediate labels
  own_stream a stream of the segment's own instead of the current one
"""
import math

import torch

from paper_2403_11204_b200 import binding
from paper_2403_11204_b200.binding import Segment

L2_BYTES = 126e6
# Adam's step is a sign-like function of the gradient: where a gradient element is no larger than its own rounding
# error, two correct implementations move the weight by up to 2 lr apart, and the trajectories separate from there.
# With this rate and at most 16 steps a pass they stay comparable.
ADAM_LR = 1e-4


def _case(name, task, net, final, precision, optimizer, batch, samples, labels="normal", own_stream=False):
    return {"name": name, "task": task, "net": net, "final": final, "precision": precision, "optimizer": optimizer,
            "batch": batch, "samples": samples, "labels": labels, "own_stream": own_stream}


def listed():
    return [
        # Answering one batch of requests with a trained, joined network: the smallest call there is.
        _case("infer_tiny_fp32", "infer", "784-128-128-64|64-64-64-47", True, "fp32", "sgd", 64, 64),
        # A user's own training loop on a small network with small batches: launches and host work per step.
        _case("tiny_loop_fp32", "loop", "784-128-128-64", False, "fp32", "sgd", 64, 2048),
        # The paper's own experiment (Section 3): an epoch of the left partition, 80 steps of 1410 ...
        _case("paper_left_fp32", "epoch", "784-80-60", False, "fp32", "momentum", 1410, 112800, "uniform_kappa"),
        # ... and of the right partition on the class labels.
        _case("paper_right_fp32", "epoch", "60-60-60-47", True, "fp32", "momentum", 1410, 112800),
        # The default precision on layers wider than the paper's, the last batch partial.
        _case("wider_left_fp32", "epoch", "784-1024-1024-512", False, "fp32", "adam", 256, 4000),
        # EMNIST-sized layers in TF32: the left partition, full batches and a partial one.
        _case("shaped_left_tf32", "epoch", "784-1024-1024-512", False, "tf32", "adam", 256, 4000),
        # The final partition of the same network.
        _case("shaped_right_tf32", "epoch", "512-512-256-47", True, "tf32", "adam", 256, 4000),
        # Recovery epochs (Section 5) of that network: the left partition through the frozen right one.
        _case("recover_tf32", "recover", "784-1024-1024-512|512-512-256-47", True, "tf32", "adam", 256, 2048),
        # Wide layers in bf16, the last batch partial.
        _case("wide_left_bf16", "epoch", "784-4096-4096-2048", False, "bf16", "adam", 1024, 8692),
        # A middle partition of the fully separate variant: label rows in, label rows as targets.
        _case("middle_cut_bf16", "label_input", "4096-4096-4096-4096", False, "bf16", "adam", 2048, 8192, own_stream=True),
        # The stored response handed to the next partition: the wide left partition over a large set.
        _case("response_bf16", "infer", "784-4096-4096-2048", False, "bf16", "adam", 1024, 33000),
        # The largest segment: bound by the matrix products and the update's memory traffic.
        _case("large_right_bf16", "epoch", "8192-8192-8192-1000", True, "bf16", "momentum", 4096, 12288, own_stream=True),
    ]


def _log_int(rng, lo, hi, odd_share=0.3):
    """A size spread evenly over its logarithm: a multiple of 8 where it is large enough, or any integer."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < odd_share or v < 32:
        return max(lo, min(hi, int(round(v))))
    return max(lo, min(hi, int(round(v / 8)) * 8))


# What a drawn case may cost: product FLOPs of a pass (the FFMA path's rate is a fraction of the tensor cores').
_FLOP_LIMIT = {"fp32": 6e10, "tf32": 1.5e12, "bf16": 6e12}


def draw(rng):
    """A case of the same ranges: small fp32 networks like the paper's, mid-sized ones in every precision, wide ones in bf16."""
    while True:
        kind = rng.choice(["small", "mid", "mid", "mid", "wide"])
        if kind == "small":
            precision = "fp32"
            widths = [_log_int(rng, 16, 1024)] + [_log_int(rng, 16, 128) for _ in range(rng.randint(2, 4))]
            batch = _log_int(rng, 32, 2048)
        elif kind == "mid":
            precision = rng.choice(["fp32", "tf32", "tf32", "bf16", "bf16"])
            widths = [_log_int(rng, 64, 1024)] + [_log_int(rng, 128, 2048) for _ in range(rng.randint(2, 3))]
            batch = _log_int(rng, 64, 1024)
        else:
            precision = "bf16"
            widths = [_log_int(rng, 784, 8192)] + [_log_int(rng, 1024, 8192) for _ in range(rng.randint(2, 3))]
            batch = _log_int(rng, 512, 4096)
        task = rng.choice(["epoch", "epoch", "epoch", "loop", "label_input", "recover", "infer"])
        final = task == "recover" or (task != "label_input" and rng.random() < 0.4)
        classes = rng.choice([10, 47, 62, 1000 if kind == "wide" else 100])
        if task == "recover":
            hidden = _log_int(rng, 16, 128) if kind == "small" else _log_int(rng, 128, 512)
            net = "-".join(map(str, widths)) + "|" + "-".join(map(str, [widths[-1], hidden, classes]))
        else:
            if final:
                widths[-1] = classes
            net = "-".join(map(str, widths))
        optimizer = rng.choice(["sgd", "momentum", "adam", "adam"])
        steps = rng.randint(4, 16 if optimizer == "adam" else 40)
        samples = max(1, steps * batch - (rng.randint(1, batch - 1) if rng.random() < 0.5 else 0))
        case = {"task": task, "net": net, "final": final, "precision": precision,
                "optimizer": optimizer, "batch": batch, "samples": samples,
                "labels": rng.choice(["normal", "uniform_kappa"]) if kind == "small" else "normal",
                "own_stream": rng.random() < 0.3}
        if work(case)["flops"] <= _FLOP_LIMIT[precision]:
            return case


def _segments(case):
    return [[int(w) for w in part.split("-")] for part in case["net"].split("|")]


def prepare(case, seed):
    segs = _segments(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, batch, precision = case["samples"], case["batch"], case["precision"]
    dtype = torch.bfloat16 if precision == "bf16" else torch.float32
    n_classes = segs[-1][-1] if case["final"] else 47
    stream = torch.cuda.Stream() if case["own_stream"] else None
    handles = []
    for k, widths in enumerate(segs):
        last = case["final"] and k == len(segs) - 1
        seg = Segment(widths, n_classes, last, precision=precision, optimizer=case["optimizer"],
                      lr=ADAM_LR if case["optimizer"] == "adam" else 0.01, max_batch=batch, segment_id=k,
                      init_seed=seed % (1 << 31), stream=stream)
        if not last:
            seg.gen_labels(seed % (1 << 31) + 1, case["labels"], 10.0)
        handles.append(seg)
    state = {"case": case, "segs": handles,
             "cls": torch.randint(0, n_classes, (n,), generator=g, device="cuda", dtype=torch.int32),
             "losses": torch.zeros(-(-n // batch), device="cuda")}
    if case["task"] == "label_input":
        state["sil_in"] = torch.randn(n_classes, segs[0][0], generator=g, device="cuda")
    else:
        x = torch.rand(n, segs[0][0], generator=g, device="cuda")      # image-like features, or a stored ReLU response
        state["x"] = x.to(dtype)
    torch.cuda.synchronize()
    return state


def run(state):
    case, segs, cls, losses = state["case"], state["segs"], state["cls"], state["losses"]
    task, n, batch, seg = case["task"], case["samples"], case["batch"], segs[0]
    if task == "infer":
        cur, out = state["x"], []
        for s in segs:
            cur = s.forward_dataset(cur, batch)
            out.append(cur)
        return {"responses": out}
    if task == "epoch":
        seg.train_epochs(state["x"], cls, batch, 1, losses)
    else:
        for i, lo in enumerate(range(0, n, batch)):
            hi = min(n, lo + batch)
            if task == "loop":
                seg.train_step(state["x"][lo:hi], cls[lo:hi], losses[i:i + 1])
            elif task == "label_input":
                seg.train_step_label_input(state["sil_in"], cls[lo:hi], losses[i:i + 1])
            else:
                binding.recovery_step(seg, segs[1], state["x"][lo:hi], cls[lo:hi], losses[i:i + 1])
    return {"losses": losses, "params": [seg.params(l) for l in range(seg.n_layers)]}


def work(case):
    """Products of every sample; the data set once, the results once, and per step the parameters with their
    optimizer state read and written (once in all where they fit the L2 cache)."""
    segs, n = _segments(case), case["samples"]
    es = 2 if case["precision"] == "bf16" else 4
    macs = [[a * b for a, b in zip(w, w[1:])] for w in segs]
    params = sum(macs[0]) + sum(segs[0][1:])
    if case["task"] == "infer":
        flops = 2 * n * sum(sum(m) for m in macs)
        weights = sum(sum(m) for m in macs) * es
        return {"bytes": n * es * segs[0][0] + weights + sum(n * w[-1] * es for w in segs), "flops": flops}
    flops = 2 * n * (3 * sum(macs[0]) - macs[0][0])
    if case["task"] == "recover":
        flops += 2 * n * 2 * sum(macs[1])
    steps = -(-n // case["batch"])
    state = params * {"sgd": 8, "momentum": 16, "adam": 24}[case["optimizer"]]
    x_bytes = 0 if case["task"] == "label_input" else n * es * segs[0][0]
    return {"bytes": x_bytes + 4 * n + 4 * steps + state * (steps if state > L2_BYTES else 1) + 4 * params, "flops": flops}


# About four times the difference measured between two correct orders of summation (the FFMA products against the tensor
# cores', input features permuted, the step launch by launch), over two passes: responses 4.4e-7 / 6e-5 / 8.4e-4 in fp32 /
# TF32 / bf16; trained weights 8.2e-4 / 4.5e-4 / 6.0e-4 under SGD and momentum, 6e-3 / 8e-3 / 9e-3 under Adam (see ADAM_LR).
_TOLERANCE = {
    ("infer", "fp32"): {"rel": 2e-6, "max": 2e-5},
    ("infer", "tf32"): {"rel": 3e-4, "max": 4e-3},
    ("infer", "bf16"): {"rel": 4e-3, "max": 5e-2},
    ("train", "fp32"): {"rel": 3e-3, "max": 2e-2},
    ("train", "tf32"): {"rel": 2e-3, "max": 1e-2},
    ("train", "bf16"): {"rel": 2.5e-3, "max": 2e-2},
    ("adam", "fp32"): {"rel": 2.5e-2, "max": 0.4},
    ("adam", "tf32"): {"rel": 3e-2, "max": 0.5},
    ("adam", "bf16"): {"rel": 3e-2, "max": 0.9},
}


def tolerance(case):
    kind = "infer" if case["task"] == "infer" else "adam" if case["optimizer"] == "adam" else "train"
    return dict(_TOLERANCE[kind, case["precision"]])
