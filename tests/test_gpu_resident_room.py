"""Networks that keep three 32 x 32 tensors on the resident engine, where shared memory has 6 KB left for a convolution's weights
and tables: every tensor of one sample equals the CPU oracle's, a batch's logits the plain kernels'."""
import numpy as np
import pytest

import paper_2108_09413_b200 as isc
from test_gpu_conv_shapes import _conv
from test_gpu_requant_range import _check


def three_tensors(kind, rng):
    """a residual block whose output has another zero-point than its skip operand, so that it cannot be written over it"""
    c = lambda t, cin, cout, k, zin, zout, res=-1, zres=0, stride=1: _conv(rng, t, cin, cout, k, stride, 0, zin, zout, res=res, zp_res=zres)
    if kind == "filters":
        return [c(0, 3, 16, 3, 3, -128), c(1, 16, 16, 3, -128, -128), c(2, 16, 16, 3, -128, -128), c(3, 16, 16, 3, -128, -123), c(4, 16, 16, 3, -123, 127, 3, -128)], 32
    if kind == "one by one":
        return [c(0, 3, 16, 3, 3, 121), c(1, 16, 16, 1, 121, 121), c(1, 16, 16, 1, 121, 121), c(2, 16, 16, 1, 121, -40), c(4, 16, 16, 1, -40, 121)], 32
    return [c(0, 3, 16, 3, 3, -128), c(1, 16, 16, 3, -128, -128), c(1, 16, 16, 1, -128, -128, stride=2), c(2, 16, 32, 3, -128, 0, stride=2),
            c(1, 16, 16, 3, -128, -128), c(3, 16, 64, 3, -128, -128, stride=2)], 8


KINDS = ["filters", "one by one", "branches"]


@pytest.mark.parametrize("kind", KINDS)
def test_they_have_a_plan(kind):
    layers, side = three_tensors(kind, np.random.default_rng(1))
    import workloads as wl
    n, cout, zp = len(layers), layers[-1]["cout"], layers[-1]["zp_out"]
    layers = layers + [wl._gavgpool(n, cout, side * side, zp), dict(_conv(np.random.default_rng(2), n + 1, cout, 9, 1, 1, 0, zp, 0), op=wl.OP_FC, pad=0)]
    assert isc.plan_resident(dict(in_shape=(3, 32, 32), n_classes=9, layers=layers))[0] == 1


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("seed", range(3))
def test_they_equal_the_oracle(kind, seed):
    rng = np.random.default_rng(seed)
    layers, side = three_tensors(kind, rng)
    _check(rng, (3, 32, 32), layers, 3, 1200, side * side)
