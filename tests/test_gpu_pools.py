"""Max-pool windows with and without padding, overlapping or not, on odd maps: every element of one sample's pooled
tensor equals the CPU oracle's, on both layer-by-layer engines."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hw,c,k,stride,pad", [((17, 20), 16, 3, 2, 1), ((9, 12), 40, 3, 1, 1), ((8, 8), 64, 2, 2, 0), ((11, 4), 32, 5, 3, 2), ((3, 4), 48, 3, 3, 0)])
@pytest.mark.parametrize("engine", [1, 2])
def test_max_pool(hw, c, k, stride, pad, engine):
    rng = np.random.default_rng(c + k)
    zp = int(rng.integers(-128, 40))
    h, w = [(n + 2 * pad - k) // stride + 1 for n in hw]
    L = [_conv(rng, 0, 3, c, 3, 1, 1, 3, zp, shift_lo=8), wl._maxpool(1, c, k, stride, pad, zp),
         wl._gavgpool(2, c, max(h * w, 2), zp)]
    L.append(dict(_conv(rng, 3, c, 9, 1, 1, 0, zp, 0), op=wl.OP_FC, pad=0))
    model = dict(in_shape=(3,) + hw, n_classes=9, layers=L)
    gm, om = isc.Model(model), oracle.Model(model)
    gm.set_option("engine", engine)
    x = rng.integers(0, 256, model["in_shape"]).astype(np.uint8)
    got = gm.debug_tensor(x, 5, 1, 1, 2, 0.25, 2, oracle.tensor_size(om, 2))
    np.testing.assert_array_equal(got, oracle.forward(om, oracle.noisy_input(x, 5, 1, 1, 2, 0.25), dump_tensor=2)[1])
    ec, el = oracle.sample_counts(om, x, 5, 1, 1, 0, 13, 0.25, want_logits=True)
    gc, gl = gm.sample_counts(x, 5, 1, 1, 0, 13, 0.25, want_logits=True)
    np.testing.assert_array_equal(gl, el)
    np.testing.assert_array_equal(gc, ec)
