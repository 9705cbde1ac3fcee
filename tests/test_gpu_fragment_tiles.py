"""Accumulators read as fragments, in the layer-by-layer engine's two kernels: every width of a block of output channels,
tiles that end inside the batch and inside a row, with and without a residual operand, and each of the ways in which the
input tile of a stride-1 filter is copied.  Every tensor equals the CPU oracle's, a batch's logits the plain kernels'."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv

pytestmark = pytest.mark.gpu


def _check(rng, shape, layers, samples, stride=1):
    """layers, then global pool -> FC; the last layer's output zero-point is -128"""
    c, side = layers[-1]["cout"], [(n - 1) // stride + 1 for n in shape[1:]]
    layers = layers + [wl._gavgpool(len(layers), c, max(2, side[0] * side[1]), -128)]
    layers = layers + [dict(_conv(rng, len(layers), c, 9, 1, 1, 0, -128, 0), op=wl.OP_FC, pad=0)]
    model = dict(in_shape=shape, n_classes=9, layers=layers)
    gm, om = isc.Model(model), oracle.Model(model)
    gm.set_option("engine", 2)
    x = rng.integers(0, 256, shape).astype(np.uint8)
    a0 = oracle.noisy_input(x, 5, 1, 1, 2, 0.25)
    for t in range(1, om.n_layers + 1):
        got = gm.debug_tensor(x, 5, 1, 1, 2, 0.25, t, oracle.tensor_size(om, t))
        np.testing.assert_array_equal(got, oracle.forward(om, a0, dump_tensor=t)[1], err_msg=f"tensor {t}")
    many = gm.sample_counts(x, 5, 1, 1, 0, samples, 0.25, want_logits=True)
    assert gm.get_info("engine") == 2
    gm.set_option("engine", 1)
    plain = gm.sample_counts(x, 5, 1, 1, 0, samples, 0.25, want_logits=True)
    np.testing.assert_array_equal(many[1], plain[1])
    np.testing.assert_array_equal(many[0], plain[0])


# (h, w): rows against the steps of 32, 16 and 8 positions in which they are copied: one short step, one whole one, just
# more than one, with little and with much of the last one idle, more positions than a lane keeps
@pytest.mark.parametrize("h,w", [(7, 7), (5, 8), (15, 14), (9, 16), (6, 28), (4, 32), (3, 76)])
@pytest.mark.parametrize("c0,c1", [(16, 32), (32, 48), (48, 16), (64, 64), (32, 80), (64, 112), (80, 144)])
def test_filters_with_a_resident_tile(h, w, c0, c1):
    rng = np.random.default_rng(c0 * c1 + w)
    _check(rng, (3, h, w), [_conv(rng, 0, 3, c0, 3, 1, 1, 3, -128), _conv(rng, 1, c0, c1, 3, 1, 1, -128, -20),
                            _conv(rng, 2, c1, c1, 3, 1, 1, -20, -128, res=2, zp_res=-20)], 1 + 60_000 // (h * w))


# output widths of one to four groups of 64 channels and of two tiles; batches that leave 0, 1 and 127 pixels of the
# last 128 or 256
@pytest.mark.parametrize("c0,c1,stride", [(64, 64, 1), (128, 128, 1), (64, 192, 1), (64, 256, 1), (128, 512, 1), (64, 128, 2), (64, 320, 1), (64, 80, 1)])
@pytest.mark.parametrize("h,w,samples", [(16, 16, 160), (5, 5, 2053), (1, 1, 4095), (3, 3, 2049)])
def test_whole_tiles_of_one_by_one_layers(c0, c1, stride, h, w, samples):
    rng = np.random.default_rng(c0 + c1 + w)
    _check(rng, (3, h, w), [_conv(rng, 0, 3, c0, 3, 1, 1, 3, -128), _conv(rng, 1, c0, c1, 1, stride, 1, -128, -20),
                            _conv(rng, 2, c1, c1, 1, 1, 1, -20, -128, res=2, zp_res=-20)], samples, stride)
