"""Calls at the limits of what an engine takes: whichever kernels they end up on, the results are the CPU oracle's."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc
from test_host_dispatch import _every_kernel_net, _hidden_layer_net

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout", [(24, 6912), (24, 6913), (64, 10112), (64, 10240)])
def test_layers_around_the_shared_memory_limit_of_the_tensor_core_kernel(cin, cout):
    model = _hidden_layer_net(wl, cin, cout)
    gm, om = isc.Model(model), oracle.Model(model)
    x = wl.images(1, shape=model["in_shape"], seed=3)[0]
    ec, el = oracle.sample_counts(om, x, 5, 1, 1, 0, 19, 0.25, want_logits=True)
    gc, gl = gm.sample_counts(x, 5, 1, 1, 0, 19, 0.25, want_logits=True)
    np.testing.assert_array_equal(gl, el)
    np.testing.assert_array_equal(gc, ec)
    np.testing.assert_array_equal(gm.sample_counts_static(x, 5, 1, 1, 0, 19, 0.25), ec)


@pytest.mark.parametrize("net", ["resident", "layerwise"])
def test_device_images_of_any_alignment(net):
    import torch
    model = wl.spread_model("resnet20") if net == "resident" else wl.resnet50(hw=64, blocks=(1, 1, 1, 1))
    gm = isc.Model(model)
    xs = wl.images(3, shape=model["in_shape"], seed=8)
    expected = gm.certify_batch(xs, 3, 7, 0, 20, 150, 0.25, 0.001)
    for offset in (0, 1, 2, 3, 5):
        buf = torch.zeros(xs.size + 16, dtype=torch.uint8, device="cuda")
        buf[offset:offset + xs.size] = torch.from_numpy(xs.ravel()).cuda()
        torch.cuda.synchronize()
        got = gm.certify_batch(None, 3, 7, 0, 20, 150, 0.25, 0.001, device_ptr=buf.data_ptr() + offset)
        for g, e in zip(got, expected):
            np.testing.assert_array_equal(g, e)


def test_static_entry_point_on_the_engine_it_is_told():
    gm = isc.Model(wl.spread_model("resnet20"))
    x = wl.spread_image()
    expected = gm.sample_counts(x, 9, 5, 1, 3, 1203, 0.25)
    for engine in (1, 2, 3):
        gm.set_option("engine", engine)
        np.testing.assert_array_equal(gm.sample_counts_static(x, 9, 5, 1, 3, 1203, 0.25), expected)


def test_stalled_layers_leave_through_their_abort_path():
    """One launch of every kernel of the layer-by-layer tensor-core engine whose weights are held back: the first
    convolution, the filter kernel with its weights resident and with a ring of them, the implicit GEMM.  Its waits run
    out after their own two seconds, the error word is up (ISC_ERR_TIMEOUT = -6), and the handle then computes the right
    logits.  Nothing here faults, traps or hangs the GPU."""
    model = _every_kernel_net(wl)
    gm, om = isc.Model(model), oracle.Model(model)
    gm.set_option("engine", 2)
    x = wl.images(1, shape=model["in_shape"])[0]
    for layer in (0, 2, 3, 4):
        rc, (err_word, ns) = gm.debug_stalled_launch(layer)
        assert rc == -6 and err_word >= 1, layer
        assert 1_900_000_000 <= ns
        got = gm.sample_counts(x, 11, 3, 1, 0, 3, 0.5, want_logits=True)
        exp = oracle.sample_counts(om, x, 11, 3, 1, 0, 3, 0.5, want_logits=True)
        np.testing.assert_array_equal(got[1], exp[1])
        np.testing.assert_array_equal(got[0], exp[0])
    assert gm.debug_stalled_launch(1)[0] == -3 and gm.debug_stalled_launch(len(model["layers"]))[0] == -1
