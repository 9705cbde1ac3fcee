"""The first convolution on the tensor cores: filter widths on both sides of four pixels, strides that do and do not
divide four, bands of one to 32 rows, rows wider than a tile, 16 to 256 output channels, lower clamps and shifts of
every form.  The layer's output equals the CPU oracle's, a batch's logits the plain kernels'."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv

pytestmark = pytest.mark.gpu

SHAPES = [  # (channels, h, w), c0, k, stride
    ((3, 24, 28), 64, 7, 2), ((3, 17, 20), 16, 3, 1), ((1, 9, 12), 96, 5, 1), ((4, 20, 23), 160, 5, 3), ((3, 33, 31), 48, 3, 2),
    ((2, 12, 16), 256, 1, 1), ((3, 30, 36), 64, 8, 4), ((3, 16, 300), 32, 7, 1), ((3, 10, 700), 32, 7, 1), ((3, 5, 4), 24, 5, 2), ((3, 19, 22), 16, 7, 5),
]


@pytest.mark.parametrize("shape,c0,k,stride", SHAPES)
@pytest.mark.parametrize("zp,shift_lo", [(-128, 2), (-40, 2), (9, 0)])
def test_stem_equals_the_oracle(shape, c0, k, stride, zp, shift_lo):
    rng = np.random.default_rng(c0 * k + stride)
    L = [_conv(rng, 0, shape[0], c0, k, stride, 1, 3, zp, shift_lo=shift_lo)]
    h, w = [(n + 2 * (k // 2) - k) // stride + 1 for n in shape[1:]]
    L.append(wl._gavgpool(1, c0, max(h * w, 2), zp))
    L.append(dict(_conv(rng, 2, c0, 9, 1, 1, 0, zp, 0), op=wl.OP_FC, pad=0))
    model = dict(in_shape=shape, n_classes=9, layers=L)
    gm, om = isc.Model(model), oracle.Model(model)
    gm.set_option("engine", 2)
    x = rng.integers(0, 256, shape).astype(np.uint8)
    for sample in (0, 5):
        got = gm.debug_tensor(x, 5, 1, 1, sample, 0.25, 1, oracle.tensor_size(om, 1))
        np.testing.assert_array_equal(got, oracle.forward(om, oracle.noisy_input(x, 5, 1, 1, sample, 0.25), dump_tensor=1)[1])
    many = gm.sample_counts(x, 5, 1, 1, 0, 700, 0.25, want_logits=True)
    gm.set_option("engine", 1)
    plain = gm.sample_counts(x, 5, 1, 1, 0, 700, 0.25, want_logits=True)
    np.testing.assert_array_equal(many[1], plain[1])
    np.testing.assert_array_equal(many[0], plain[0])


# bands beside bins of 10 and of 41 KB, beside the search's tables, without tables in shared memory; many items and few per CTA,
# and a CTA for each
@pytest.mark.parametrize("h,w,c0,k,stride,samples", [(224, 224, 64, 7, 2, 40), (301, 300, 64, 8, 2, 25), (32, 32, 64, 3, 1, 900), (75, 75, 64, 7, 2, 150), (40, 448, 48, 7, 2, 60)])
@pytest.mark.parametrize("sigma", [0.25, 1.0, 2.0, 4.6])
def test_noise_tables_beside_the_bands(h, w, c0, k, stride, samples, sigma):
    rng = np.random.default_rng(h + k)
    L = [_conv(rng, 0, 3, c0, k, stride, 1, 3, -128)]
    oh, ow = [(n + 2 * (k // 2) - k) // stride + 1 for n in (h, w)]
    L.append(wl._gavgpool(1, c0, oh * ow, -128))
    L.append(dict(_conv(rng, 2, c0, 9, 1, 1, 0, -128, 0), op=wl.OP_FC, pad=0))
    model = dict(in_shape=(3, h, w), n_classes=9, layers=L)
    gm, om = isc.Model(model), oracle.Model(model)
    x = rng.integers(0, 256, model["in_shape"]).astype(np.uint8)
    results = []
    for engine in (2, 1):
        gm.set_option("engine", engine)
        results.append(gm.sample_counts(x, 5, 1, 1, 0, samples, sigma, want_logits=True))
        got = gm.debug_tensor(x, 5, 1, 1, 3, sigma, 1, c0 * oh * ow)
        np.testing.assert_array_equal(got, oracle.forward(om, oracle.noisy_input(x, 5, 1, 1, 3, sigma), dump_tensor=1)[1])
    np.testing.assert_array_equal(results[0][1], results[1][1])
    np.testing.assert_array_equal(results[0][0], results[1][0])
