"""What a user of this framework has it do, as cases that can be timed: inference and minibatch SGD of sparse networks of
L square layers, through the public calls of ``paper_2104_11805_b200``.

The sizes are those of the repository's configurations (1024 x 120, 4096 x 120, 16384 and 65536 neurons, 32 links per
neuron, minibatches of 1, 16 and 64) or of no particular origin (odd widths, ragged rows, odd batches).  The wide nets are
cut to a few layers: a layer costs the same whatever the depth, and even the cut nets are larger than the L2 cache.

A case is a dict:
  do        "infer", "infer_host" (buffers in pinned host memory), "infer_noalloc", "train", "train_host", "train_averaged"
  n, layers neurons per layer, layers
  inputs    inference: inputs per call; training: inputs per minibatch
  steps     training: minibatch steps before the weights are taken out (0 for inference)
  links     "uniform" (32 per neuron, anywhere), "ragged" (8 to 56 per neuron, as after pruning), "blocks" (32 per neuron
            within hidden blocks of 1024 neurons)
  act       "relu" (clamped at 32; weights N(0, 2/32), bias 0: half of the neurons stay active at every depth),
            "sigmoid" (weights uniform in [-1, 1), bias 0: the training set-up of the paper's experiments),
            "dying" (inference; all weights 1/16, bias -0.35: an input either dies out within a few layers or saturates)
  counts    inference: also the number of nonzero outputs per input
  bias      training: the biases are trained too
"""
import math

import numpy as np
import torch

import paper_2104_11805_b200 as sdnn

K = 32                  # links per neuron (mean of the ragged nets)
BLOCK = 1024            # neurons per block of the "blocks" nets
MINIBATCHES = 8         # distinct minibatches a training case goes through
TILE = 1024             # inputs a handle for inference is created for, where the call brings at least so many


def _case(name, do, n, layers, inputs, steps=0, links="uniform", act="relu", counts=False, bias=False):
    c = dict(do=do, n=n, layers=layers, inputs=inputs, steps=steps, links=links, act=act, counts=counts, bias=bias)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one request to the smallest network: 120 dependent layers with next to nothing in them
        _case("infer 1024x120, one input", "infer", 1024, 120, 1),
        # a full tile of it, with the category scores the Graph Challenge asks for
        _case("infer 1024x120, 256 inputs", "infer", 1024, 120, 256, counts=True),
        # a test set through a network of ordinary width
        _case("infer 4096x120, 10000 inputs", "infer", 4096, 120, 10000, counts=True),
        # a pruned network of odd width with a smooth activation: rows of any length, a batch that is no multiple of anything
        _case("infer 20011x12 ragged sigmoid", "infer", 20011, 12, 1501, links="ragged", act="sigmoid"),
        # the widest network, its links in hidden blocks (set-up reordering and shared-memory windows asked for)
        _case("infer 65536x6 blocks", "infer", 65536, 6, 4096, links="blocks"),
        # most inputs die on the way and may be dropped; the surviving neurons are asked for by number
        _case("infer 4096x120 dying", "infer", 4096, 120, 5000, act="dying", counts=True),
        # a service: requests of a few hundred inputs that come from and go back to host memory
        _case("infer 3000x40 ragged host", "infer_host", 3000, 40, 700, links="ragged", counts=True),
        # a caller that keeps the network in its own arrays and may not allocate
        _case("infer 4096x24 noalloc", "infer_noalloc", 4096, 24, 100, links="ragged"),
        # per-input SGD as the paper prints it, a checkpoint after 64 inputs
        _case("train 1024x48, B=1 sigmoid", "train", 1024, 48, 1, steps=64, act="sigmoid"),
        # minibatch SGD on the middle network
        _case("train 16384x24, B=64", "train", 16384, 24, 64, steps=64),
        # and on the widest one
        _case("train 65536x12, B=16 sigmoid", "train", 65536, 12, 16, steps=128, act="sigmoid"),
        # a training loop over host data that logs every loss: odd width, odd minibatch, ragged rows, trained biases
        _case("train 6007x24, B=37 ragged host", "train_host", 6007, 24, 37, steps=32, links="ragged", act="sigmoid", bias=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: widths from 600 to 65536, depths from 4 to 120 as far as the set-up stays short, batches from one
    input to thousands, every kind of call, link pattern and activation."""
    do = rng.choice(["infer", "infer", "infer", "infer_host", "infer_noalloc", "train", "train", "train", "train_host", "train_averaged"])
    n = _log_uniform(rng, 600, 65536)
    bias = do == "train_host" or (do.startswith("train") and rng.random() < 0.3)
    deepest = 24 if bias else 56 if do.startswith("train") else 120      # the weights of every layer come back, one output each
    layers = max(4, min(deepest, int(rng.uniform(0.4, 1.0) * 600000 / n)))
    links = rng.choice(["uniform", "uniform", "ragged"])
    if do == "infer_noalloc":
        # activation tiles of at most 2^20 numbers; the width of a tile is the batch rounded up to 4, 8, .. 128, multiples of 128
        top = (1 << 20) // n
        top = top // 128 * 128 if top >= 128 else 1 << (top.bit_length() - 1)
        return _case(None, do, n, layers, _log_uniform(rng, 1, min(top, 1000)), links=links)
    if do.startswith("infer"):
        act = rng.choice(["relu", "relu", "sigmoid", "dying" if do == "infer" and links == "uniform" else "relu"])
        if do == "infer" and n >= 4096 and act == "relu" and rng.random() < 0.3:
            n, links = n // BLOCK * BLOCK, "blocks"
            layers = min(layers, 600000 // n)
        most = min(10000, int(1.0e11 / (n * K * layers)))
        least = 100 if act == "dying" else 1      # of a few inputs all would die, or none
        return _case(None, do, n, layers, _log_uniform(rng, least, most), links=links, act=act,
                     counts=rng.random() < 0.5 and (act != "relu" or n <= 8192))
    inputs = _log_uniform(rng, 1, 128)
    steps = max(8, min(128, int(6.0e10 / (n * K * layers * inputs))))
    # trained biases and the averaged step with the smooth activation only: on the clamped ReLU's kinks they are chaotic
    act = rng.choice(["relu", "sigmoid"]) if do == "train" and not bias else "sigmoid"
    return _case(None, do, n, layers, inputs, steps=steps, links=links, act=act, bias=bias)


def _layers(case, gen):
    """Row pointers, columns and values of all layers, made on the GPU: column numbers ascend within a row."""
    n, depth, links = case["n"], case["layers"], case["links"]
    row_ptr, cols, vals = [], [], []
    wide = 56 if links == "ragged" else K
    for _ in range(depth):
        span = BLOCK if links == "blocks" else n
        # `wide` distinct columns: sorted draws with repetition from a range shorter by wide - 1, spread out by their rank
        c = torch.randint(0, span - wide + 1, (n, wide), device="cuda", generator=gen).sort(dim=1).values
        c += torch.arange(wide, device="cuda")
        if links == "blocks":
            place = torch.randperm(n, device="cuda", generator=gen)
            c = place[c + torch.arange(n, device="cuda").div(BLOCK, rounding_mode="floor")[:, None] * BLOCK].sort(dim=1).values
        if links == "ragged":
            # every length from 8 to 56 equally often, in any order
            length = 8 + torch.randperm(n, device="cuda", generator=gen).mul(wide - 7).div(n, rounding_mode="floor")
            keep = torch.rand(n, wide, device="cuda", generator=gen).argsort(dim=1) < length[:, None]
            c, count = c[keep], keep.sum(dim=1)
        else:
            c, count = c.reshape(-1), torch.full((n,), wide, device="cuda")
        rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
        rp[1:] = count.cumsum(0)
        if case["act"] == "dying":
            v = torch.full((c.numel(),), 1.0 / 16.0, device="cuda")
        elif case["act"] == "sigmoid":
            v = torch.rand(c.numel(), device="cuda", generator=gen) * 2.0 - 1.0
        else:
            v = torch.randn(c.numel(), device="cuda", generator=gen) * math.sqrt(2.0 / K)
        row_ptr.append(rp)
        cols.append(c.int())
        vals.append(v)
    return row_ptr, cols, vals


def _inputs(case, count, gen):
    """0/1 vectors with a tenth of the pixels set; between 5 % and 50 % where the network sorts its inputs by that."""
    p = 0.1
    if case["act"] == "dying":
        p = torch.rand(count, 1, device="cuda", generator=gen) * 0.45 + 0.05
    return (torch.rand(count, case["n"], device="cuda", generator=gen) < p).float()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, depth, do, inputs = case["n"], case["layers"], case["do"], case["inputs"]
    row_ptr, cols, vals = _layers(case, gen)
    bias = np.full(n, -0.35 if case["act"] == "dying" else 0.0, dtype=np.float32)
    s = {"case": case}
    if do == "infer_noalloc":
        at = np.zeros(depth, dtype=np.int64)      # every layer's entries begin at a multiple of four
        for k in range(1, depth):
            at[k] = (at[k - 1] + cols[k - 1].numel() + 3) // 4 * 4
        s["at"] = at
        s["col"] = torch.zeros(int(at[-1]) + cols[-1].numel(), dtype=torch.int32, device="cuda")
        s["val"] = torch.zeros(s["col"].numel(), device="cuda")
        for k in range(depth):
            s["col"][at[k]:at[k] + cols[k].numel()] = cols[k]
            s["val"][at[k]:at[k] + cols[k].numel()] = vals[k]
        s["row_ptr"] = torch.stack(row_ptr)
        s["bias"] = torch.zeros(depth, n, device="cuda")
    else:
        train = do.startswith("train")
        flags = sdnn.FLAG_REORDER | sdnn.FLAG_SMEM_WINDOWS if case["links"] == "blocks" else sdnn.FLAG_SKIP_DEAD if case["act"] == "dying" else 0
        s["net"] = sdnn.Sdnn.create([r.cpu().numpy() for r in row_ptr], [c.cpu().numpy() for c in cols], [v.cpu().numpy() for v in vals], [bias] * depth,
                                    max_batch=inputs if train else min(inputs, TILE), train=train, update_bias=case["bias"], flags=flags,
                                    activation=sdnn.ACT_SIGMOID if case["act"] == "sigmoid" else sdnn.ACT_CLAMPED_RELU)
    if do.startswith("train"):
        s["x"] = [_inputs(case, inputs, gen) for _ in range(MINIBATCHES)]
        s["y"] = [torch.rand(inputs, n, device="cuda", generator=gen) for _ in range(MINIBATCHES)]
        if do == "train_host":
            s["x"] = [x.cpu().pin_memory() for x in s["x"]]
            s["y"] = [y.cpu().pin_memory() for y in s["y"]]
        return s
    s["x"] = _inputs(case, inputs, gen)
    s["y"] = torch.zeros(inputs, n, device="cuda")
    s["count"] = torch.zeros(inputs, dtype=torch.int32, device="cuda") if case["counts"] else None
    if do == "infer_host":
        s["x"], s["y"] = s["x"].cpu().pin_memory(), s["y"].cpu().pin_memory()
        s["count"] = s["count"].cpu().pin_memory() if case["counts"] else None
    if case["act"] == "dying":
        s["ids"] = torch.zeros(inputs * n, dtype=torch.int32, device="cuda")
    return s


def run(s):
    case = s["case"]
    inputs = case["inputs"]
    if case["do"] == "infer_noalloc":
        sdnn.infer_noalloc(case["layers"], case["n"], s["row_ptr"], s["col"], s["val"], s["at"], s["bias"], s["x"], inputs, s["y"])
        return s["y"]
    net = s["net"]
    if case["do"].startswith("infer"):
        if "ids" in s:
            total = net.infer_batch(s["x"], inputs, s["y"], s["count"], s["ids"], inputs * case["n"], want_total=True)
            return {"y": s["y"], "count": s["count"], "ids": s["ids"], "total": total}      # ids: zeros from `total` on
        net.infer_batch(s["x"], inputs, s["y"], s["count"], host=case["do"] == "infer_host")
        return {"y": s["y"], "count": s["count"]}
    # with the clamped ReLU small enough that rounding does not grow from step to step
    eta = 0.01 if case["act"] == "sigmoid" else 1e-5
    losses = []
    for t in range(case["steps"]):
        x, y = s["x"][t % MINIBATCHES], s["y"][t % MINIBATCHES]
        log = case["do"] == "train_host" or t == case["steps"] - 1
        losses.append(net.train_step(x, y, inputs, eta, want_loss=log, host=case["do"] == "train_host", averaged=case["do"] == "train_averaged"))
    state = [net.get_weights(k, want_bias=case["bias"]) for k in range(case["layers"])]
    return {"loss": np.array([v for v in losses if v is not None]), "state": state}


def work(case):
    """Inference: the network once (4-byte column and 4-byte weight per link), inputs and outputs once, a multiply-add per
    link and input.  A training step: the network forwards (8 bytes per link) and, after all layers, backwards with the
    updated weight written (12 bytes), every activation written and read, three multiply-adds per link and input; then the
    weights once out to the caller."""
    n, depth, inputs = case["n"], case["layers"], case["inputs"]
    links = n * depth * K
    if not case["do"].startswith("train"):
        ids = inputs * n if case["act"] == "dying" else 0      # about a third of the inputs survive with every neuron
        return {"bytes": 8 * links + 4 * n * depth + 8 * n * inputs + 4 * ids / 3, "flops": 2 * links * inputs}
    step = 20 * links + 8 * n * depth * inputs + 8 * n * inputs
    return {"bytes": case["steps"] * step + 4 * links, "flops": 6 * links * inputs * case["steps"]}


def tolerance(case):
    """Sums of 32-bit products in another order, carried through the layers (and, in training, through the steps).  With the
    ReLU a neuron in a million is so close to 0 that the order decides whether it counts as active: of thousands of
    neurons, in up to one input of a hundred."""
    return {"rel": 1e-5, "max": 4e-4, "differ": 0.01 if case["act"] == "relu" else 0.0}
