"""1 x 1 layers in tiles of 256 pixels x 128 channels, against the plain kernels: pixel counts that end in the first or in
the second half of a tile, one or several tiles of channels, with and without a residual operand (its term as a product;
the 64-bit term is in test_gpu_requant_range.py), lower clamps at and above -128, and batches on either side of the rule that
pairs tiles."""
import numpy as np
import pytest

import workloads as wl
import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hw,c0,c1", [((8, 8), 64, 128), ((7, 8), 128, 256), ((5, 4), 128, 384), ((9, 4), 192, 128)])
@pytest.mark.parametrize("zp,res_shift", [(-128, -1), (-128, 0), (17, 0), (-60, -1)])
def test_paired_tiles_equal_the_plain_kernels(hw, c0, c1, zp, res_shift):
    rng = np.random.default_rng(c1 + zp)
    L = [_conv(rng, 0, 3, c0, 3, 1, 1, 3, zp), _conv(rng, 1, c0, c1, 1, 1, 1, zp, zp), _conv(rng, 2, c1, c0, 1, 1, 1, zp, zp),
         _conv(rng, 3, c0, c1, 1, 1, 1, zp, zp, res=2, zp_res=zp), wl._gavgpool(4, c1, hw[0] * hw[1], zp)]
    L[3]["res_shift"] = res_shift
    L.append(dict(_conv(rng, 5, c1, 9, 1, 1, 0, zp, 0), op=wl.OP_FC, pad=0))
    model = dict(in_shape=(3,) + hw, n_classes=9, layers=L)
    x = rng.integers(0, 256, model["in_shape"]).astype(np.uint8)
    gm = isc.Model(model)
    pixels = hw[0] * hw[1]
    for n in (1, 30_000 // pixels, 60_000 // pixels + 1, 60_000 // pixels + 3):
        results = []
        for engine, copy in ((1, 1), (2, 1), (2, 0)):
            gm.set_option("engine", engine)
            gm.set_option("tensor_copy", copy)
            results.append(gm.sample_counts(x, 5, 1, 1, 0, n, 0.25, want_logits=True))
        for counts, logits in results[1:]:
            np.testing.assert_array_equal(logits, results[0][1])
            np.testing.assert_array_equal(counts, results[0][0])
