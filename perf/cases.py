"""What a user of the library has it do, as cases that can be timed and compared.

The path is: quantize a dense fp32 sample matrix twice into packed code planes (on uniform levels or on
variance-optimal ones), run minibatch SGD epochs over the planes, look at the loss on the way; or hand the whole
job over from host memory; or take the steps one by one, as a rank of a row-sharded run does.  Every case goes
through `paper_1611_05402_b200.binding` (or `sharded`) and returns everything the call computed.

A case is a dict: `kind` is the call, `values` the distribution of the samples, the rest sizes and options.
"""
import math

import torch

from paper_1611_05402_b200 import binding, sharded

HIST_BINS = 1024
NOISE = 0.05                                  # of the labels, as in the synthetic workloads


def _epoch(name, m, n, bits, batch, values, **more):
    return {"name": name, "kind": "epoch", "m": m, "n": n, "bits": bits, "batch": batch, "values": values, "levels": "uniform",
            "model_bits": 0, "grad_bits": 0, "reg": 0, **more}


def listed():
    return [
        # A small regression table (the size of the usual LIBSVM sets), small batches: 256 dependent steps of 1 KB.
        _epoch("epoch_small", 4096, 64, 4, 16, "uniform"),
        # The ordinary dense problem: a thousand features at 8 bits, 391 steps of half a megabyte.
        _epoch("epoch_medium", 100_000, 1000, 8, 256, "normal"),
        # End-to-end low precision: 2-bit samples, model and gradient quantized to 8 bits in every step.
        _epoch("epoch_end_to_end", 1_000_000, 2048, 2, 1024, "uniform", model_bits=8, grad_bits=8),
        # Skewed features on variance-optimal 3-bit levels.
        _epoch("epoch_levels", 500_000, 512, 3, 512, "skewed", levels="optimal"),
        # Tomography: rows much wider than they are many, mostly zeros, large batches.
        _epoch("epoch_wide", 65_536, 32_768, 4, 2048, "sparse"),
        # Large batches over rows of ordinary width and an odd number of features, 6 bits (the paper's operating
        # point), l2 regularised, the last batch ragged: what one does to fill a large device.
        _epoch("epoch_large_batch", 300_007, 1999, 6, 8192, "normal", reg=1),
        # Single steps, each its own calls, as a rank of a row-sharded run takes them: sixteen launch-bound steps.
        {"name": "steps_sharded", "kind": "steps", "m": 4096, "n": 1000, "bits": 8, "batch": 256, "values": "normal",
         "levels": "uniform", "model_bits": 0, "grad_bits": 8, "reg": 0},
        # Quantization of the ordinary dense problem, odd sizes (rows that are not 16-byte aligned).
        {"name": "quantize_medium", "kind": "quantize", "m": 100_003, "n": 1001, "bits": 8, "values": "normal", "levels": "uniform"},
        # Quantization of the large sparse matrix: 8.6 GB of samples.
        {"name": "quantize_wide", "kind": "quantize", "m": 65_536, "n": 32_768, "bits": 4, "values": "sparse", "levels": "uniform"},
        # Placing variance-optimal levels and quantizing onto them: two calls that belong together.
        {"name": "quantize_levels", "kind": "quantize", "m": 500_000, "n": 512, "bits": 3, "values": "skewed", "levels": "optimal"},
        # Loss from the stored codes, what a training loop monitors once the fp32 samples are gone.
        {"name": "loss_codes", "kind": "loss", "m": 1_000_000, "n": 2048, "bits": 2, "values": "uniform", "levels": "uniform"},
        # The whole job from host memory: copy, quantize, five epochs with decaying steps, loss, model back.
        {"name": "fit_from_host", "kind": "fit", "m": 100_000, "n": 1000, "bits": 8, "batch": 256, "values": "normal",
         "levels": "uniform", "model_bits": 0, "grad_bits": 0, "reg": 0, "epochs": 5},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["epoch"] * 6 + ["steps", "quantize", "quantize", "loss", "fit"])
    values = rng.choice(["uniform", "normal", "skewed", "sparse"])
    levels = "optimal" if values == "skewed" and rng.random() < 0.7 else "uniform"
    bits = rng.choice([2, 3, 4]) if levels == "optimal" else rng.choice([2, 3, 4, 4, 5, 6, 8, 8])
    n = _log_int(rng, 16, 2048 if levels == "optimal" else 32_768)
    if rng.random() < 0.5:                                        # half of the sizes round, as tables often are
        n = max(16, n // 16 * 16)
    case = {"kind": kind, "n": n, "bits": bits, "values": values, "levels": levels}
    if kind in ("quantize", "loss"):
        case["m"] = _log_int(rng, 1 << 18, 1 << 30) // n + 1
        return case
    model_bits, grad_bits = rng.choice([(0, 0), (0, 0), (0, 8), (8, 8), (4, 6)])
    case.update(batch=_log_int(rng, 16, 16_384), model_bits=model_bits, grad_bits=grad_bits, reg=rng.choice([0, 0, 0, 1, 2, 3]))
    if rng.random() < 0.7:
        case["batch"] = max(16, case["batch"] // 16 * 16)
    most = (1 << (26 if kind == "fit" else 30)) // n              # rows that keep a case below the largest listed one
    if kind == "steps":
        case["batch"] = min(case["batch"], 1024)
        case["m"] = case["batch"] * rng.randint(4, 24)
    else:
        case["m"] = max(16, min(most, case["batch"] * _log_int(rng, 8, 1024) - rng.randrange(case["batch"])))
    if kind == "fit":
        case["epochs"] = rng.randint(1, 5)
    return case


def _samples(case, g):
    """The sample matrix, in pieces that keep the temporary memory small."""
    m, n, values = case["m"], case["n"], case["values"]
    A = torch.empty((m, n), dtype=torch.float32, device="cuda")
    scale = None
    rows = max(1, (1 << 26) // n)
    for r in range(0, m, rows):
        part = A[r:r + rows]
        if values == "uniform":
            part.uniform_(-1, 1, generator=g)
        elif values == "normal":
            part.normal_(generator=g).clamp_(-3, 3)
        elif values == "skewed":                                  # a sign and a log-normal size, scaled per feature into [-1, 1]
            sign = torch.empty_like(part).uniform_(-1, 1, generator=g).sign_()
            part.normal_(std=1.5, generator=g).exp_().mul_(sign)
            top = part.abs().amax(dim=0)
            scale = top if scale is None else torch.maximum(scale, top)
        else:                                                     # 5 % of the entries, uniform in [0, 1]
            keep = torch.empty_like(part).uniform_(generator=g) < 0.05
            part.uniform_(generator=g).mul_(keep)
    if scale is not None:
        A /= scale
    return A


def _problem(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = _samples(case, g)
    n = case["n"]
    if case["values"] == "sparse":
        true = torch.rand(n, generator=g, device="cuda")          # densities of an image: not negative
    else:
        true = torch.randn(n, generator=g, device="cuda") / math.sqrt(n)
    b = A @ true
    b += NOISE * torch.randn(case["m"], generator=g, device="cuda")
    return A, b, true


_contexts = {}


def _context():
    """One context for the process, on its current device, as a program keeps it."""
    at = torch.cuda.current_device()
    if at not in _contexts:
        _contexts[at] = binding.Context(torch.device("cuda", at))
    return _contexts[at]


def _quantize(ctx, case, A, seed):
    if case["levels"] == "optimal":
        levels = ctx.zipml_optimal_levels(A, case["bits"], HIST_BINS)
        return ctx.zipml_quantize(A, case["bits"], seed, binding.LEVELS_TABLE, levels)
    return ctx.zipml_quantize(A, case["bits"], seed)


def _step_length(ctx, case, A):
    """A step length that the quantized samples bear: a fifth of the inverse of a row's mean square norm, the
    variance of its rounding included."""
    power = A.square().mean()
    if case["levels"] == "optimal":                               # the objective: 4 bins^2 times the variance, on a unit range
        levels, objective = ctx.zipml_optimal_levels(A, case["bits"], HIST_BINS, want_objective=True)
        power += ((levels[:, -1] - levels[:, 0]) ** 2 * objective).mean() / (4 * HIST_BINS ** 2 * case["m"])
    else:                                                         # p (1 - p) of the cell's square, 1/6 on average
        power += ((A.amax() - A.amin()) / ((1 << case["bits"]) - 1)) ** 2 / 6
    return float(0.2 / (case["n"] * power))


def _options(case):
    return {"model_bits": case["model_bits"], "grad_bits": case["grad_bits"], "reg": case["reg"], "reg_param": 1e-3 if case["reg"] else 0.0,
            "seed": 7}


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    A, b, true = _problem(case, seed)
    state = {"case": case, "ctx": ctx, "seed": seed % (1 << 31)}
    if kind == "quantize":
        state["A"] = A
        return state
    state["lr"] = _step_length(ctx, case, A)
    if kind == "fit":
        for key, v in (("A", A), ("b", b)):                       # the user's own buffers: pinned host memory
            state[key] = torch.empty(v.shape, dtype=v.dtype, pin_memory=True).copy_(v)
        return state
    state["data"] = _quantize(ctx, case, A, state["seed"])
    ctx.zipml_sync()
    state["b"] = b
    state["x0"] = 0.5 * true                                      # a model on its way
    if kind == "steps":
        plan = sharded.ShardPlan(case["m"], case["batch"], 0, 1)
        state["rank"] = sharded.ShardedEpoch(ctx, plan, state["data"], b, state["x0"].clone(), state["lr"], **_options(case))
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "quantize":
        data = _quantize(ctx, case, state["A"], state["seed"])
        return {"plane1": data.plane1, "plane2": data.plane2, "lo": data.feat_lo,
                "scale": data.levels if data.levels is not None else data.feat_step}
    if kind == "loss":
        return ctx.zipml_loss(binding.LOSS_CODES, state["b"], state["x0"], data=state["data"])
    if kind == "fit":
        x = torch.zeros(case["n"])
        loss = ctx.zipml_train_host(state["A"], state["b"], x, case["bits"], case["batch"], state["lr"], case["epochs"],
                                    optimal_levels=case["levels"] == "optimal", hist_bins=HIST_BINS, quantize_seed=state["seed"],
                                    lr_decay=True, **_options(case))
        return {"x": x, "loss": loss}
    if kind == "steps":
        rank = state["rank"]
        rank.x.copy_(state["x0"])
        rank.run()
        return {"x": rank.x, "gradient": rank.g2}
    x = state["x0"].clone()
    ctx.zipml_sgd_epoch(state["data"], state["b"], x, case["batch"], state["lr"], **_options(case))
    return x


def work(case):
    """Each input once, each output once; four multiply-adds per sample, feature and epoch (two dots, two gradients)."""
    m, n, bits = case["m"], case["n"], case["bits"]
    container = 2 if bits <= 2 else 4 if bits <= 4 else 8
    planes = 2 * m * (((n * container + 7) // 8 + 15) // 16 * 16)      # rows start on 16 bytes
    scale = 4 * n * ((1 << bits) if case["levels"] == "optimal" else 2)
    if case["kind"] == "quantize":
        return {"bytes": 4 * m * n + planes + scale, "flops": 0}
    if case["kind"] == "loss":
        return {"bytes": planes + scale + 4 * m + 4 * n, "flops": 4 * m * n}
    if case["kind"] == "fit":
        return {"bytes": 4 * m * n + 4 * m + 4 * n, "flops": (8 * case["epochs"] + 2) * m * n}
    return {"bytes": planes + scale + 4 * m + 8 * n, "flops": 8 * m * n}


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        return "exact"                                            # codes, levels and ranges are pinned bit for bit
    if kind == "loss":
        return {"rel": 1e-5}
    # The library's engines differ from each other, and from its double-precision one, by 1e-7 in the model after an
    # epoch and by 2e-6 in a gradient; where the model or the gradient is rounded stochastically, a last bit can turn
    # a draw over: 2e-5 in the model was the most seen, at 4 bits of model and 6 of gradient.
    if case["model_bits"] or case["grad_bits"]:
        return {"rel": 2e-4}
    return {"rel": 1e-5}
