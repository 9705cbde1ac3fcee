"""Cases of the Monte-Carlo PREDICT / CERTIFY path, through the library's public entry points.

A case is one call of a user's program on a loaded network: the network (a generator of `workloads` and its sizes),
the entry point, the number of noisy samples, the noise level and law, and the launch batch.  The networks have random
int8 weights; their last layer is balanced on the case's image and noise level so that the votes of the noisy copies
spread over the classes with a favourite, as a trained network's do on an image it is unsure of.  A unanimous vote,
which a network of random weights gives otherwise, would leave the confidence bound its closed form.

A program loads a network once and sends image after image through the handle, so the handle of a (network, noise,
launch batch) is kept; what a seed changes is the images and the random stream.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2108_09413_b200 as isc
import workloads as wl

ALPHA = 0.001


def _case(name=None, net="cifar", blocks="3", width=16, hw=32, classes=10, entry="certify", n0=100, n=1000, images=1,
          sigma=0.25, noise=0, launch=0):
    """net: "tiny" (two convolutions), "cifar" (basic blocks per stage, widths w, 2w, 4w) or "bottleneck" (blocks of
    the four stages as digits).  n0 / n: selection and estimation samples; launch: samples per launch, 0 = automatic."""
    c = dict(net=net, blocks=blocks, width=width, hw=hw, classes=classes, entry=entry, n0=n0, n=n, images=images,
             sigma=sigma, noise=noise, launch=launch)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest CERTIFY in use: configuration 0, one image through the tiny CNN; launches and host work count
        _case("tiny_certify_1k", net="tiny", n=1000),
        # an interactive PREDICT at the smallest n of the paper's appendix C
        _case("resnet20_predict_100", entry="predict", n=100),
        # configuration 1: one CIFAR-10 image at full N and its lowest noise level
        _case("resnet20_certify_100k", n=100_000, sigma=0.12),
        # configuration 1 as a data set is certified: images resident on the GPU, 1,024 samples per launch
        _case("resnet20_batch_8x10k", entry="batch", n=10_000, images=8, sigma=0.5, launch=1024),
        # configuration 2, the headline: ResNet-110 at full N
        _case("resnet110_certify_100k", blocks="18", n=100_000),
        # configuration 4: the sweep's cell of the smallest launches and the most noise
        _case("resnet110_launch_256", blocks="18", n=10_000, sigma=1.0, launch=256),
        # configuration 3: ResNet-50 on a 224 x 224 image, N = 10,000
        _case("resnet50_certify_10k", net="bottleneck", blocks="3463", width=64, hw=224, classes=101, n=10_000, sigma=0.5),
        # the same network asked for one quick answer
        _case("resnet50_predict_100", net="bottleneck", blocks="3463", width=64, hw=224, classes=101, entry="predict",
              n=100, sigma=0.5),
        # an image size no tile divides, per-sample logits returned for analysis
        _case("bottleneck_75_logits_1k", net="bottleneck", blocks="1221", width=64, hw=75, classes=37, entry="counts",
              n=1001),
        # a wider residual network (32 / 64 / 128 channels) with the integer form of the radius
        _case("wide_resnet_integer_5k", blocks="3", width=32, entry="integer", n=5000),
        # widths that no tensor tile divides on 40 x 40 images, with the comparison method's rounded Gaussian noise
        _case("resnet_w24_40px_rounded_3k", blocks="2", width=24, hw=40, classes=43, n=3000, sigma=0.5, noise=1),
        # the allocation-free entry point of a service that owns its device memory
        _case("resnet20_static_2k", entry="static", n=2000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    sigma = round(math.exp(rng.uniform(math.log(0.12), math.log(1.0))), 3)
    noise = 1 if rng.random() < 0.2 else 0
    kind = rng.choice(["resident"] * 4 + ["bottleneck"] * 2 + ["wide"] * 2 + ["static"])
    entry, images, launch = rng.choice(["certify", "certify", "predict", "integer", "counts", "batch"]), 1, 0
    n = _log_int(rng, 100, 100_000)
    if kind == "resident":
        net = rng.choice(["tiny", "cifar", "cifar", "cifar"])
        c = dict(net=net, blocks="1" if net == "tiny" else str(_log_int(rng, 1, 18)), width=16, hw=32,
                 classes=10 if net == "tiny" else rng.randint(2, 100))
        launch = rng.choice([0, 0, 256, 1024, 4096, 16384])
        cap = 2e13
    elif kind == "bottleneck":
        c = dict(net="bottleneck", blocks="".join(str(rng.randint(1, m)) for m in (3, 4, 6, 3)), width=64,
                 hw=_log_int(rng, 40, 224), classes=rng.randint(2, 300))
        cap = 1e13
    else:
        c = dict(net="cifar", blocks=str(rng.randint(1, 4)), width=rng.choice([16, 20, 24, 32, 40, 48, 64, 80, 96]),
                 hw=rng.randint(24, 72), classes=rng.randint(2, 200))
        cap = 1e12
        if kind == "static":
            entry, cap = "static", 3e11
            c.update(width=rng.choice([8, 16, 24, 32]), hw=rng.randint(20, 40))
    if entry == "batch":
        images = rng.randint(2, 12)
    elif entry == "counts":
        n = min(n, 20_000)
    per = 2.0 * wl.macs_per_sample(_network(**_key(c)))
    n = max(50, min(n, int(cap / per / images)))
    return _case(entry=entry, n=n, images=images, sigma=sigma, noise=noise, launch=launch, **c)


# ------------------------------------------------------------------------------------------- networks and handles

def _key(case):
    return {k: case[k] for k in ("net", "blocks", "width", "hw", "classes")}


@functools.lru_cache(maxsize=4)
def _network(net, blocks, width, hw, classes):
    if net == "tiny":
        return wl.tiny_cnn()
    if net == "cifar":
        model = wl.cifar_resnet(int(blocks), 0x15170001, n_classes=classes, hw=hw, widths=(width, 2 * width, 4 * width))
        side = hw
        for _ in range(2):
            side = (side + 1) // 2
    else:
        model = wl.resnet50(0x15170003, n_classes=classes, hw=hw, blocks=tuple(int(b) for b in blocks), base=width)
        side = hw
        for _ in range(5):
            side = (side + 1) // 2
    # the pool's multiplier for the true size of its map: 1 / side^2 = mult / 2^(31 + shift)
    area = side * side
    shift = area.bit_length() - 1
    if area == 1 << shift:
        shift, mult = shift - 1, 1 << 30
    else:
        mult = round((1 << (31 + shift)) / area)
    pool = dict(model["layers"][-2], mult=np.array([mult], np.int32), shift=np.array([shift], np.int8))
    return dict(model, layers=model["layers"][:-2] + [pool, model["layers"][-1]])


@functools.lru_cache(maxsize=4)
def _base_image(hw):
    return wl.images(1, shape=(3, hw, hw), seed=0x15174000)[0]


def _balanced(model, image, sigma, noise):
    """The network with a last layer whose class means are equal on `image`, but for class 0's, three deviations up."""
    fc = model["layers"][-1]
    features = []
    base = isc.Model(model)
    base.set_option("noise", noise)
    for j in range(24):
        features.append(base.debug_tensor(image, 7, 0, 0, j, sigma, len(model["layers"]) - 1, fc["cin"]))
    base.close()
    rng = np.random.default_rng(5)
    w = rng.integers(-16, 17, (fc["cout"], fc["cin"])).astype(np.int8)
    acc = (np.stack(features).astype(np.int64) - fc["zp_in"]) @ w.T.astype(np.int64)
    spread = max(1.0, float(acc.std(axis=0).mean()))
    bias = -np.round(acc.mean(axis=0)).astype(np.int32)
    bias[0] += int(3.0 * spread)
    shift = min(15, max(1, int(round(math.log2(spread / 4.0)))))
    head = dict(fc, w=w.reshape(fc["cout"], fc["cin"], 1, 1), bias=bias, mult=np.full(fc["cout"], 3 << 29, np.int32),
                shift=np.full(fc["cout"], shift, np.int8))
    return dict(model, layers=model["layers"][:-1] + [head])


@functools.lru_cache(maxsize=16)
def _handle(net, blocks, width, hw, classes, sigma, noise, launch):
    model = _network(net, blocks, width, hw, classes)
    handle = isc.Model(_balanced(model, _base_image(hw), sigma, noise))
    handle.set_option("noise", noise)
    handle.set_option("batch", launch)
    return handle


# ------------------------------------------------------------------------------------------- what is measured

def prepare(case, seed):
    handle = _handle(**_key(case), sigma=case["sigma"], noise=case["noise"], launch=case["launch"])
    rng = np.random.default_rng(seed)
    # photographs of one scene: the balanced image with a few levels of difference per pixel
    shape = (case["images"], 3, case["hw"], case["hw"])
    x = np.clip(_base_image(case["hw"]).astype(np.int16) + rng.integers(-3, 4, shape), 0, 255).astype(np.uint8)
    on_gpu = torch.from_numpy(x).cuda() if case["entry"] == "batch" else None
    return dict(handle=handle, x=x if on_gpu is not None else x[0], on_gpu=on_gpu, seed=int(rng.integers(1 << 40)), case=case)


def run(state):
    h, x, seed, c = state["handle"], state["x"], state["seed"], state["case"]
    n0, n, sigma = c["n0"], c["n"], c["sigma"]
    if c["entry"] == "certify":
        return h.certify(x, seed, 0, n0, n, sigma, ALPHA)
    if c["entry"] == "predict":
        return h.predict(x, seed, 0, n, sigma, ALPHA)
    if c["entry"] == "integer":
        return h.certify_integer(x, seed, 0, n0, n, sigma, ALPHA, two_sided=True)
    if c["entry"] == "counts":
        return h.sample_counts(x, seed, 0, 1, 0, n, sigma, want_logits=True)
    if c["entry"] == "static":
        return h.sample_counts_static(x, seed, 0, 1, 0, n, sigma)
    return h.certify_batch(None, c["images"], seed, 0, n0, n, sigma, ALPHA, stream=torch.cuda.current_stream(),
                           device_ptr=state["on_gpu"].data_ptr())


def work(case):
    """Multiply-accumulates of every noisy forward pass, two operations each; the parameters and images once, and the
    counts (or logits) that come back.  Noise is generated and activations can stay on the chip: no other bytes."""
    model = _network(**_key(case))
    phases = case["n"] + (case["n0"] if case["entry"] in ("certify", "integer", "batch") else 0)
    samples = phases * case["images"]
    weights = sum(layer["w"].size for layer in model["layers"] if layer["w"] is not None)
    out = 8 * case["classes"] * case["images"] + (case["n"] * case["classes"] if case["entry"] == "counts" else 0)
    return {"bytes": weights + 3 * case["hw"] ** 2 * case["images"] + out, "flops": 2.0 * wl.macs_per_sample(model) * samples}


def tolerance(case):
    # the whole path is integer arithmetic, and the bound's doubles are evaluated in one fixed order
    return "exact"
