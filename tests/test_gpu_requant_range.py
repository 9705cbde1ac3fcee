"""Requantisation at the ends of its range: rounding addends whose sum with the product's high word needs more than 32 bits,
with accumulators of both signs; and the residual term in each of its forms, in every kernel.  Every tensor of one sample and the logits of a batch equal the CPU oracle's, or the
plain kernels'."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv

pytestmark = pytest.mark.gpu


def _wide(rng, *args, shift, mult=1_900_000_000, **kw):
    """A convolution whose channels' accumulators lie about 20 million above and below zero in turn."""
    layer = _conv(rng, *args, **kw)
    layer["bias"] = (layer["bias"] + 20_000_000 * (1 - 2 * (np.arange(layer["cout"]) & 1))).astype(np.int32)
    layer["mult"][:] = mult
    layer["shift"][:] = shift
    return layer


def _check(rng, shape, layers, engine, samples, pixels):
    """layers, then global pool -> FC, on `engine`"""
    c, zp = layers[-1]["cout"], layers[-1]["zp_out"]
    layers = layers + [wl._gavgpool(len(layers), c, max(2, pixels), zp)]
    layers = layers + [dict(_conv(rng, len(layers), c, 9, 1, 1, 0, zp, 0), op=wl.OP_FC, pad=0)]
    model = dict(in_shape=shape, n_classes=9, layers=layers)
    gm, om = isc.Model(model), oracle.Model(model)
    gm.set_option("engine", engine)
    x = rng.integers(0, 256, shape).astype(np.uint8)
    a0 = oracle.noisy_input(x, 5, 1, 1, 2, 0.25)
    for t in range(1, om.n_layers + 1 if engine != 3 else om.n_layers - 1):
        got = gm.debug_tensor(x, 5, 1, 1, 2, 0.25, t, oracle.tensor_size(om, t))
        np.testing.assert_array_equal(got, oracle.forward(om, a0, dump_tensor=t)[1], err_msg=f"tensor {t}")
    many = gm.sample_counts(x, 5, 1, 1, 0, samples, 0.25, want_logits=True)
    assert gm.get_info("engine") == engine
    gm.set_option("engine", 1)
    plain = gm.sample_counts(x, 5, 1, 1, 0, samples, 0.25, want_logits=True)
    np.testing.assert_array_equal(many[1], plain[1])
    np.testing.assert_array_equal(many[0], plain[0])


# (channels in, out, filter) of the layer with the residual operand: resident-tile filters, whole tiles single and paired, the
# general form
@pytest.mark.parametrize("cin,cout,k", [(32, 32, 3), (64, 128, 3), (256, 64, 1), (64, 128, 1), (48, 40, 1)])
# the addend of the product form lies 0.7 million above -2^31, 450 million above it (which fits), and far below it
@pytest.mark.parametrize("res_mult,zp_res,zp_out,shift", [(2032202290, 7, -20, 18), (2032202290, 7, -20, 17), (1798879234, -20, 5, 14)])
def test_residual_constants_leave_room_for_the_product(cin, cout, k, res_mult, zp_res, zp_out, shift):
    rng = np.random.default_rng(cin + cout + shift)
    layers = [_conv(rng, 0, 3, cin, 3, 1, 1, 3, -128), _conv(rng, 1, cin, cout, 1, 1, 0, -128, zp_res),
              _wide(rng, 1, cin, cout, k, 1, 0, -128, zp_out, res=2, zp_res=zp_res, shift=shift)]
    layers[2].update(res_mult=res_mult, res_shift=0)
    _check(rng, (3, 12, 8), layers, 2, 700, 96)


# first convolution, resident-tile filter, whole tiles by tensor copy and gathered, paired, the general form, FC; 2^(s - 1) + zp_out 2^s
# in 32 bits: fits with room for the product up to a shift of 24, without it at 25, not at all from 26 on
@pytest.mark.parametrize("zp", [-128, 127, 5])
@pytest.mark.parametrize("shift", [20, 24, 25, 26, 31])
def test_addends_of_wide_shifts(shift, zp):
    rng = np.random.default_rng(shift)
    relu = int(zp == -128)
    wide = lambda t, cin, cout, k, stride, z, **kw: _wide(rng, t, cin, cout, k, stride, relu, z, zp, shift=shift, **kw)
    layers = [wide(0, 3, 64, 3, 1, 3), wide(1, 64, 64, 3, 1, zp), wide(2, 64, 256, 1, 1, zp), wide(3, 256, 64, 1, 1, zp),
              wide(4, 64, 256, 1, 1, zp, res=3, zp_res=zp), wide(5, 256, 128, 1, 2, zp), wide(6, 128, 48, 1, 1, zp)]
    _check(rng, (3, 16, 12), layers, 2, 400, 48)


# a wide shift on one channel among ordinary ones
def test_one_channel_of_a_wide_shift():
    rng = np.random.default_rng(3)
    layers = [_conv(rng, 0, 3, 64, 3, 1, 1, 3, -128), _conv(rng, 1, 64, 64, 3, 1, 1, -128, -128), _conv(rng, 2, 64, 256, 1, 1, 0, -128, -128),
              _conv(rng, 3, 256, 64, 1, 1, 1, -128, -128)]
    for layer in layers:
        layer["shift"][7] = 27
    _check(rng, (3, 16, 12), layers, 2, 400, 192)


@pytest.mark.parametrize("res_mult,zp_res,zp_out,shift", [(2032202290, 7, -20, 18), (2032202290, 7, -20, 17), (1798879234, -20, 5, 14)])
def test_residual_constants_of_the_resident_engine(res_mult, zp_res, zp_out, shift):
    rng = np.random.default_rng(shift)
    layers = [_conv(rng, 0, 3, 16, 3, 1, 1, 3, -128), _conv(rng, 1, 16, 32, 3, 2, 0, -128, zp_res), _conv(rng, 2, 32, 32, 3, 1, 1, zp_res, -128),
              _wide(rng, 3, 32, 32, 3, 1, 0, -128, zp_out, res=2, zp_res=zp_res, shift=shift)]
    layers[3].update(res_mult=res_mult, res_shift=0)
    _check(rng, (3, 32, 32), layers, 3, 700, 256)


FORMS = [(1304428746, 0, 77), (1342155344, 0, 7), (1817091736, -1, 77), (1090259607, -1, -63),        # no product: the 64-bit term
         (1334892440, -1, -63), (2032202290, 0, 7), (1 << 30, 0, -128), (1435772024, -1, -128)]      # product


# resident-tile filter, whole tiles, paired tiles, the general form; paired tiles need enough of them for every SM
@pytest.mark.parametrize("cin,cout,k", [(32, 48, 3), (256, 64, 1), (64, 256, 1), (48, 40, 1)])
@pytest.mark.parametrize("res", FORMS)
@pytest.mark.parametrize("relu", [0, 1])
def test_both_forms_of_the_residual_term(cin, cout, k, res, relu):
    assert (isc.residual_product(*res) is None) == (FORMS.index(res) < 4)
    rng = np.random.default_rng(res[0] % 1000 + cin)
    layers = [_conv(rng, 0, 3, cin, 3, 1, 1, 3, -128), _conv(rng, 1, cin, cout, 1, 1, 0, -128, res[2]),
              _conv(rng, 1, cin, cout, k, 1, relu, -128, res[2], res=2, zp_res=res[2])]
    layers[2].update(res_mult=res[0], res_shift=res[1])
    _check(rng, (3, 12, 8), layers, 2, 700, 96)


@pytest.mark.parametrize("res", FORMS)
@pytest.mark.parametrize("relu", [0, 1])
def test_both_forms_on_the_resident_engine(res, relu):
    rng = np.random.default_rng(res[0] % 1000)
    layers = [_conv(rng, 0, 3, 16, 3, 1, 1, 3, res[2]), _conv(rng, 1, 16, 16, 3, 1, 1, res[2], -128),
              _conv(rng, 2, 16, 16, 3, 1, relu, -128, res[2], res=1, zp_res=res[2]), _conv(rng, 3, 16, 32, 3, 2, 1, res[2], res[2]),
              _conv(rng, 4, 32, 32, 3, 1, 1, res[2], -128), _conv(rng, 5, 32, 32, 3, 1, relu, -128, res[2], res=4, zp_res=res[2])]
    for layer in layers:
        layer.update(res_mult=res[0], res_shift=res[1])
    _check(rng, (3, 32, 32), layers, 3, 700, 256)
