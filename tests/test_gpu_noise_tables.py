"""The noise search of the layer-by-layer engine's first convolution, shown by a layer that passes its pixels through, and
of the resident engine's input phase.  Standard deviations with tables of bins of every size, too wide for one, and of so
few levels that most bins are open; both noise laws; widths of whole Philox blocks and not."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [0.001, 0.01, 0.25, 0.5, 1.0, 1.5])
@pytest.mark.parametrize("noise", [0, 1])
@pytest.mark.parametrize("h,w", [(64, 64), (61, 67)])
def test_every_level_that_is_drawn(sigma, noise, h, w):
    rng = np.random.default_rng(7)
    first = _conv(rng, 0, 3, 16, 1, 1, 0, 128, 0)
    first.update(w=np.zeros((16, 3, 1, 1), np.int8), bias=np.zeros(16, np.int32), mult=np.full(16, 1 << 30, np.int32), shift=np.zeros(16, np.int8))
    for c in range(16):
        first["w"][c, c % 3] = 2                       # 2 (pixel - 128) / 2
    layers = [first, wl._gavgpool(1, 16, h * w, 0), dict(_conv(rng, 2, 16, 9, 1, 1, 0, 0, 0), op=wl.OP_FC, pad=0)]
    gm = isc.Model(dict(in_shape=(3, h, w), n_classes=9, layers=layers))
    gm.set_option("engine", 2)
    gm.set_option("noise", noise)
    x = rng.integers(0, 256, (3, h, w)).astype(np.uint8)
    oracle.set_noise_kind(noise)
    try:
        for sample in range(6):
            want = oracle.noisy_input(x, 9, 1, 1, sample, sigma).astype(np.int32) - 128
            got = np.asarray(gm.debug_tensor(x, 9, 1, 1, sample, sigma, 1, 16 * h * w)).reshape(16, h, w)
            np.testing.assert_array_equal(got[:3], want)
    finally:
        oracle.set_noise_kind(0)


@pytest.mark.parametrize("sigma", [0.001, 0.01, 0.25, 0.5, 1.0, 1.5])
@pytest.mark.parametrize("noise", [0, 1])
def test_every_level_of_the_resident_engine(sigma, noise):
    gm = isc.Model(wl.spread_model("resnet20"))
    gm.set_option("engine", 3)
    gm.set_option("noise", noise)
    x = np.random.default_rng(8).integers(0, 256, (3, 32, 32)).astype(np.uint8)
    oracle.set_noise_kind(noise)
    try:
        for sample in range(12):
            want = oracle.noisy_input(x, 9, 1, 1, sample, sigma).ravel()
            np.testing.assert_array_equal(gm.debug_tensor(x, 9, 1, 1, sample, sigma, 0, x.size), want)
    finally:
        oracle.set_noise_kind(0)
