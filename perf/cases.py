"""Measured cases: the calls that a program makes which trains or evaluates a
binary multi-layer perceptron with this library, over the range of its use.

A case is a dict of plain values; ``kind`` names the call:

  train     BMLP.train on one window of n patterns (mini-batches of bs)
  predict   BMLP.predict of n patterns
  layers    BMLP.predict_layers (early exit: the labels of every layer)
  forward   bmlp_layer_forward of n packed rows through one layer
  binarize  bmlp_binarize_median of n real-valued patterns
  expand    bmlp_expand_sign of n byte patterns through a fixed +-1 layer

``prepare`` makes the inputs on the GPU from the seed: i.i.d. fair bits, bits
with a probability of their own per feature, thresholded smooth 32 x 32 x 3
fields, or noisy class prototypes, labelled by a random +-1 teacher network
(the prototypes by their class).  A training state holds several windows, and
each pass trains on the next one, as a program does that streams its data set.

Every output is a bit or a whole number, and the rule reproduces each of them
exactly (random draws are keyed by seed, layer, neuron and step), so the
tolerance is "exact" throughout.
"""
import math

import torch

from paper_2412_00119_gb300 import bmlp as B

DEV = "cuda"
INPUTS = ("iid", "bias", "fields", "prototypes")


def _train(name, widths, classes, n, inputs="bias", bs=100, h_max=255, group_mode=0, epoch=False,
           windows=8):
    return dict(name=name, kind="train", widths=widths, classes=classes, n=n, inputs=inputs, bs=bs,
                h_max=h_max, group_mode=group_mode, epoch=epoch, windows=windows)


def listed():
    return [
        # one mini-batch per call on the smallest network of the workload
        # table: online training, where the call's latency is what counts
        _train("train one batch 784-256", "784,256", 10, 100, windows=200),
        # the Random Prototypes experiment: a whole epoch of 10,000 patterns
        # with its error count and p_r rescale, widths that fill no tile
        _train("train epoch 1000-255-255", "1000,255,255", 10, 10000, "prototypes", epoch=True,
               windows=1),
        # an image-sized network, a tenth of its training set per call
        _train("train 784-1024x3", "784,1024,1024,1024", 10, 6000),
        # the same for inputs of 32 x 32 x 3 with mini-batches above 128, a
        # last one that is short, and groups redrawn at every mini-batch
        _train("train 3072-2048x3 bs 512", "3072,2048,2048,2048", 10, 5000, "fields", bs=512,
               group_mode=2),
        # four wide hidden layers and 100 classes, a tenth of the training set
        _train("train 3072-4096x4 c 100", "3072,4096,4096,4096,4096", 100, 5000, "fields"),
        # the throughput benchmark's network, a piece of its stream
        _train("train 8192-8192x4", "8192,8192,8192,8192,8192", 10, 1600, "iid", windows=24),
        # one small batch of requests against a trained network
        dict(name="predict 100 784-1024x3", kind="predict", widths="784,1024,1024,1024", classes=10,
             n=100, inputs="bias"),
        # early-exit evaluation of a test set: labels of all layers, 100 classes
        dict(name="layers 10000 3072-4096x4", kind="layers", widths="3072,4096,4096,4096,4096",
             classes=100, n=10000, inputs="fields"),
        # the forward-only sweep of the benchmark
        dict(name="predict 65536 8192-8192x4", kind="predict", widths="8192,8192,8192,8192,8192",
             classes=10, n=65536, inputs="iid"),
        # one layer of a program that runs the network layer by layer, at an odd
        # batch and with rows of 1000 and 525 bits
        dict(name="forward 2000 1000-525", kind="forward", widths="1000,525", classes=10, n=2000,
             inputs="prototypes"),
        # front ends for a whole image data set: grey levels to bits by each
        # pattern's median, and bytes through a fixed random +-1 layer
        dict(name="binarize 60000x784", kind="binarize", n=60000, K=784, values="pixels"),
        dict(name="expand 60000x784-1024", kind="expand", n=60000, D=784, K=1024, values="pixels"),
    ]


# The most that a drawn case may cost, as bit pairs of its forward passes (the
# listed sweep costs 1.8e13).
_MOST_PAIRS = {"train": 4e11, "predict": 1e13, "layers": 1e13, "forward": 1e13}


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "predict", "layers", "forward", "binarize", "expand"])
    if kind == "binarize":
        return dict(kind=kind, n=_log(rng, 1, 60000), K=_log(rng, 16, 3072),
                    values=rng.choice(["pixels", "gauss"]))
    if kind == "expand":
        return dict(kind=kind, n=_log(rng, 1, 60000), D=_log(rng, 16, 3072), K=_log(rng, 64, 2048),
                    values=rng.choice(["pixels", "full"]))
    layers = 1 if kind == "forward" else rng.randint(1, 4)
    inputs = rng.choice(INPUTS)
    first = 3072 if inputs == "fields" else _log(rng, 100, 8192)
    widths = [first] + [_log(rng, 64, 8192) for _ in range(layers)]
    if rng.random() < 0.5:   # most programs choose round hidden widths
        widths[1:] = [max(64, w // 64 * 64) for w in widths[1:]]
    pairs = sum(a * b for a, b in zip(widths, widths[1:]))
    most = int(_MOST_PAIRS[kind] // pairs)
    case = dict(kind=kind, widths=",".join(map(str, widths)), inputs=inputs,
                classes=rng.choice([10, 10, 10, 100, rng.randint(2, 200)]))
    if kind == "train":
        case.update(n=min(_log(rng, 50, 10000), max(100, most)), windows=8,
                    bs=rng.choice([100, 100, 100, 64, 128, rng.randint(20, 128), rng.randint(129, 600)]),
                    h_max=rng.choice([255, 255, 255, 127, 15, 2 * rng.randint(0, 511) + 1]),
                    group_mode=rng.choice([0, 0, 0, 1, 2]), epoch=rng.random() < 0.25)
    else:
        case.update(n=min(_log(rng, 1, 65536), max(1, most)))
    return case


# -- inputs ---------------------------------------------------------------------

def _widths(case):
    return [int(w) for w in case["widths"].split(",")]


def _words(K):
    return (K + 63) // 64


def _pack(bits):
    """n x K truth values -> n x ceil(K/64) int64 words (bit j of word w = feature 64 w + j)."""
    n, K = bits.shape
    out = torch.empty(n, _words(K), dtype=torch.int64, device=DEV)
    place = torch.ones(64, dtype=torch.int64, device=DEV) << torch.arange(64, device=DEV)
    for s in range(0, n, 4096):
        b = torch.nn.functional.pad(bits[s:s + 4096], (0, _words(K) * 64 - K))
        out[s:s + 4096] = (b.view(b.shape[0], -1, 64) * place).sum(-1)
    return out


def _inputs(kind, n, K, classes, gen):
    """(packed patterns, labels): the bits of one of INPUTS, made in chunks."""
    rand = lambda *shape: torch.rand(*shape, device=DEV, generator=gen)  # noqa: E731
    x = torch.empty(n, _words(K), dtype=torch.int64, device=DEV)
    y = torch.empty(n, dtype=torch.int32, device=DEV)
    hidden = 512
    w1 = torch.where(rand(K, hidden) < 0.5, 1.0, -1.0).to(torch.bfloat16)
    w2 = torch.where(rand(hidden, classes) < 0.5, 1.0, -1.0).to(torch.bfloat16)
    prob = 0.3 + 0.4 * rand(K)
    proto = rand(classes, K) < 0.5
    f = torch.fft.fftfreq(32, device=DEV)
    smooth = torch.exp(-2.0 * math.pi ** 2 * 9.0 * (f[:, None] ** 2 + f[None, :] ** 2))
    for s in range(0, n, 8192):
        m = min(8192, n - s)
        if kind == "prototypes":
            label = torch.arange(s, s + m, device=DEV) % classes
            bits = proto[label] ^ (rand(m, K) < 0.44)
            y[s:s + m] = label.to(torch.int32)
        else:
            if kind == "fields":
                g = torch.randn(m, 3, 32, 32, device=DEV, generator=gen)
                bits = (torch.fft.ifft2(torch.fft.fft2(g) * smooth).real > 0).reshape(m, K)
            else:
                bits = rand(m, K) < (prob if kind == "bias" else 0.5)
            h = torch.where(torch.where(bits, 1.0, -1.0).to(torch.bfloat16) @ w1 >= 0, 1.0, -1.0)
            y[s:s + m] = (h.to(torch.bfloat16) @ w2).float().argmax(1).to(torch.int32)
        x[s:s + m] = _pack(bits)
    return x, y


def _pixels(n, K, full, gen):
    """n x K bytes: grey levels with about 60 % zeros, or all 256 values alike."""
    v = torch.randint(0 if full else 1, 256, (n, K), device=DEV, generator=gen, dtype=torch.uint8)
    if not full:
        v[torch.rand(n, K, device=DEV, generator=gen) < 0.6] = 0
    return v


# -- states -----------------------------------------------------------------------

class _Layer(dict):
    """A layer's state as the model holds it, copied out when it is read: the
    hidden weights (the visible weights are their signs, returned as well) and
    the local classifier stay on the device between training calls."""

    def __init__(self, model, layer):
        super().__init__(H=None, W=None, P=None, p_r=None, step=None)
        self.model, self.layer, self.got = model, layer, None

    def __getitem__(self, key):
        if self.got is None:
            H, W, P, p_r, step = self.model.state(self.layer)
            self.got = dict(H=H, W=W.view("int64"), P=P, p_r=p_r, step=step)
        return self.got[key]


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    kind, n = case["kind"], case["n"]
    if kind == "binarize":
        K = case["K"]
        if case["values"] == "gauss":
            x = torch.randn(n, K, device=DEV, generator=gen)
        else:
            x = _pixels(n, K, False, gen).float()
        return dict(kind=kind, x=x, out=torch.empty(n, _words(K), dtype=torch.int64, device=DEV))
    if kind == "expand":
        D, K = case["D"], case["K"]
        x = _pixels(n, D, case["values"] == "full", gen)
        E = torch.empty(K, _words(D), dtype=torch.int64, device=DEV)
        B.bmlp_expand_weights(seed, K, D, E)
        return dict(kind=kind, x=x, E=E, K=K,
                    out=torch.empty(n, _words(K), dtype=torch.int64, device=DEV))
    widths = _widths(case)
    if kind == "train":
        model = B.BMLP(widths, case["classes"], h_max=case["h_max"], seed=seed, bs=case["bs"],
                       group_mode=case["group_mode"])
        x, y = _inputs(case["inputs"], n * case["windows"], widths[0], case["classes"], gen)
        # a state's windows are trained in turn, whatever window comes next
        return dict(kind=kind, model=model, epoch=case["epoch"], turn=0,
                    windows=[(x[s:s + n], y[s:s + n]) for s in range(0, x.shape[0], n)])
    model = B.BMLP(widths, case["classes"], seed=seed)
    x, _ = _inputs(case["inputs"], n, widths[0], case["classes"], gen)
    if kind == "forward":
        out = torch.empty(n, _words(widths[1]), dtype=torch.int64, device=DEV)
    elif kind == "layers":
        out = torch.empty(len(widths) - 1, n, dtype=torch.int32, device=DEV)
    else:
        out = torch.empty(n, dtype=torch.int32, device=DEV)
    return dict(kind=kind, model=model, x=x, out=out)


def run(state):
    kind = state["kind"]
    if kind == "train":
        model, windows = state["model"], state["windows"]
        x, y = windows[state["turn"] % len(windows)]
        state["turn"] += 1
        # a program asks for the error count where it closes an epoch
        epoch = state["epoch"]
        errors = model.train(x, y, epoch_end=epoch, count_errors=epoch)
        out = [_Layer(model, l + 1) for l in range(model.info["L"])]
        return dict(errors=errors, layers=out) if epoch else dict(layers=out)
    if kind == "predict":
        state["model"].predict(state["x"], state["out"])
    elif kind == "layers":
        state["model"].predict_layers(state["x"], state["out"])
    elif kind == "forward":
        B.bmlp_layer_forward(state["model"].h, 1, state["x"], state["out"])
    elif kind == "binarize":
        B.bmlp_binarize_median(state["x"], state["out"])
    else:
        B.bmlp_expand_sign(state["x"], state["E"], state["K"], state["out"])
    return state["out"]


# -- what a pass cannot do without ---------------------------------------------------

# A GPU's second-level cache, in bytes: hidden weights that fit in it need be
# read and written once per pass, larger ones once per mini-batch.
_ON_CHIP = 126e6


def work(case):
    """Bytes: inputs and outputs once; for training also the hidden weights
    (the bits of h_max each) read and written once per pass, or, where they
    are larger than the on-chip cache, those of the neurons that get an update
    once per mini-batch, and the visible weights read.  Flops: 2 per bit pair
    of the forward passes and classifiers, and 1 per input value to binarise."""
    kind, n = case["kind"], case["n"]
    if kind == "binarize":
        K = case["K"]
        return dict(bytes=4.0 * n * K + 8.0 * n * _words(K), flops=1.0 * n * K)
    if kind == "expand":
        D, K = case["D"], case["K"]
        return dict(bytes=1.0 * n * D + 8.0 * K * _words(D) + 8.0 * n * _words(K), flops=2.0 * n * D * K)
    w, c = _widths(case), case["classes"]
    pairs = sum(a * b + b * c for a, b in zip(w, w[1:]))
    visible = sum(8.0 * b * _words(a) for a, b in zip(w, w[1:]))
    inputs = 8.0 * n * _words(w[0])
    if kind == "train":
        bs = case["bs"]
        steps = -(-n // bs)
        bits = max(1, int(case["h_max"]).bit_length())
        hidden = sum(a * b * bits / 8.0 for a, b in zip(w, w[1:]))
        if hidden <= _ON_CHIP:
            state = 2.0 * hidden + 2.0 * visible
        else:
            state = 0.0
            for a, b in zip(w, w[1:]):
                # a neuron gets an update when one of the patterns chooses it in its group
                some = 1.0 - (1.0 - 1.0 / B.bmlp_gamma_rule(b)) ** bs
                state += steps * (some * 2.0 * a * b * bits / 8.0 + (1.0 + some) * 8.0 * b * _words(a))
        return dict(bytes=inputs + 4.0 * n + state, flops=2.0 * n * pairs)
    outputs = 8.0 * n * _words(w[1]) if kind == "forward" else 4.0 * n * (len(w) - 1 if kind == "layers" else 1)
    if kind == "forward":
        pairs = w[0] * w[1]
    return dict(bytes=inputs + visible + outputs, flops=2.0 * n * pairs)


def tolerance(case):
    return "exact"


def exact(case, seed):
    """The two front ends in 64 bits; None for the network (its weights come
    from the library's own random streams)."""
    kind, n = case["kind"], case["n"]
    if kind not in ("binarize", "expand"):
        return None
    state = prepare(case, seed)
    out = []
    for s in range(0, n, 4096):
        x = state["x"][s:s + 4096].double()
        if kind == "binarize":
            rank = (case["K"] + 1) // 2 - 1
            bits = x > x.sort(1).values[:, rank:rank + 1]
        else:
            word = state["E"].unsqueeze(-1) >> torch.arange(64, device=DEV) & 1
            e = (word.reshape(case["K"], -1)[:, :case["D"]] * 2 - 1).double()
            bits = x @ e.t() >= 0
        out.append(_pack(bits))
    return torch.cat(out)
