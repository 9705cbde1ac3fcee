"""The layer-by-layer tensor-core kernels at the edges of their tiles: channel counts that fill no tile, output channels
in several tiles with a partial last one, maps of one pixel, of odd sizes and wider than a tile, strides, filters up to
5 x 5, batches that end inside a tile.  Every tensor of one sample and the logits of a batch equal the CPU oracle's; a
larger batch equals the plain layer-by-layer kernels'."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc

pytestmark = pytest.mark.gpu


def _conv(rng, in_tensor, cin, cout, k, stride, relu, zp_in, zp_out, res=-1, zp_res=0, shift_lo=2):
    return dict(op=wl.OP_CONV2D, in_tensor=in_tensor, res_tensor=res, cin=cin, cout=cout, kh=k, kw=k, stride=stride, pad=k // 2,
                relu=relu, zp_in=zp_in, zp_out=zp_out, zp_res=zp_res, w=rng.integers(-127, 128, (cout, cin, k, k)).astype(np.int8),
                bias=rng.integers(-4096, 4097, cout).astype(np.int32), mult=rng.integers(2 ** 30, 2 ** 31, cout).astype(np.int32),
                shift=rng.integers(shift_lo, 13, cout).astype(np.int8),
                res_mult=int(rng.integers(2 ** 30, 2 ** 31)) if res >= 0 else 0, res_shift=int(rng.integers(-1, 1)) if res >= 0 else 0)


def _net(rng, hw, c0, c1, k, stride, relu_zp, shift_lo):
    """stem -> conv k x k (the shape under test) -> the same with a residual add of its input -> pool -> FC"""
    h, w = hw
    z = [int(rng.integers(0, 256)), int(rng.integers(-128, 128)), int(rng.integers(-128, 128)), int(rng.integers(-128, 128))]
    if relu_zp:
        z[1] = z[2] = z[3] = -128
    L = [_conv(rng, 0, 3, c0, 3, 1, 1, z[0], z[1]),
         _conv(rng, 1, c0, c1, k, stride, 1, z[1], z[2], shift_lo=shift_lo),
         _conv(rng, 2, c1, c1, k, 1, int(relu_zp), z[2], z[3], res=2, zp_res=z[2], shift_lo=shift_lo)]
    side = ((h + 2 * (k // 2) - k) // stride + 1) * ((w + 2 * (k // 2) - k) // stride + 1)
    pool = dict(wl._gavgpool(3, c1, max(side, 2), z[3]))
    fc = dict(_conv(rng, 4, c1, 9, 1, 1, 0, z[3], 0), op=wl.OP_FC, pad=0)
    return dict(in_shape=(3, h, w), n_classes=9, layers=L + [pool, fc])


SHAPES = [  # (h, w), c0, c1, k, stride
    ((8, 8), 16, 16, 3, 1), ((9, 12), 24, 40, 3, 1), ((32, 32), 32, 32, 3, 1), ((17, 20), 48, 96, 3, 2), ((5, 4), 80, 112, 3, 1),
    ((1, 4), 64, 64, 3, 1), ((40, 40), 20, 48, 3, 1), ((13, 132), 16, 32, 3, 1), ((30, 28), 64, 64, 3, 1), ((14, 16), 128, 128, 3, 1),
    ((6, 8), 144, 272, 3, 1), ((7, 8), 256, 512, 3, 1), ((12, 12), 3, 5, 5, 1), ((11, 8), 48, 300, 1, 1), ((10, 12), 100, 33, 1, 2),
    ((16, 12), 33, 130, 3, 1), ((7, 36), 64, 128, 5, 2), ((3, 4), 512, 64, 3, 1),
]


@pytest.mark.parametrize("case", range(len(SHAPES)))
@pytest.mark.parametrize("relu_zp,shift_lo", [(True, 2), (False, 2), (False, 0)])
def test_layer_shapes_on_the_tensor_core_engine(case, relu_zp, shift_lo):
    hw, c0, c1, k, stride = SHAPES[case]
    rng = np.random.default_rng(7000 + case)
    model = _net(rng, hw, c0, c1, k, stride, relu_zp, shift_lo)
    gm, om = isc.Model(model), oracle.Model(model)
    gm.set_option("engine", 2)
    x = rng.integers(0, 256, model["in_shape"]).astype(np.uint8)
    a0 = oracle.noisy_input(x, 5, 1, 1, 2, 0.25)
    for t in range(1, om.n_layers + 1):
        got = gm.debug_tensor(x, 5, 1, 1, 2, 0.25, t, oracle.tensor_size(om, t))
        np.testing.assert_array_equal(got, oracle.forward(om, a0, dump_tensor=t)[1], err_msg=f"tensor {t}")
    ec, el = oracle.sample_counts(om, x, 5, 1, 1, 0, 13, 0.25, want_logits=True)
    gc, gl = gm.sample_counts(x, 5, 1, 1, 0, 13, 0.25, want_logits=True)
    np.testing.assert_array_equal(gl, el)
    np.testing.assert_array_equal(gc, ec)
    n = 1 + 400_000 // (hw[0] * hw[1])                  # several tiles for every SM
    many = gm.sample_counts(x, 5, 1, 1, 0, n, 0.25, want_logits=True)
    assert gm.get_info("engine") == 2
    gm.set_option("engine", 1)
    plain = gm.sample_counts(x, 5, 1, 1, 0, n, 0.25, want_logits=True)
    np.testing.assert_array_equal(many[1], plain[1])
    np.testing.assert_array_equal(many[0], plain[0])
