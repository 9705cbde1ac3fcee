"""The allocation-free entry point takes the handle's fastest engine; whichever it is, the counts are those of
isc_sample_counts: the resident engine, the layer-by-layer tensor-core kernels (several batches of the fixed array, a
ragged last one), and the plain kernels when they are asked for."""
import numpy as np
import pytest

import workloads as wl
import paper_2108_09413_b200 as isc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n", [("resnet20", 1), ("resnet20", 1777), ("wide", 1501), ("bottleneck", 203)])
def test_static_counts_on_every_engine(name, n):
    model = {"resnet20": lambda: wl.spread_model("resnet20"),
             "wide": lambda: wl.cifar_resnet(1, 3, n_classes=7, hw=24, widths=(24, 48, 96)),
             "bottleneck": lambda: wl.resnet50(5, n_classes=9, hw=64, blocks=(1, 1, 1, 1))}[name]()
    x = wl.spread_image() if name == "resnet20" else wl.images(1, shape=model["in_shape"], seed=8)[0]
    gm = isc.Model(model)
    for sigma in (0.25, 4.4):                    # 4.4: the table leaves no room for the guide
        expected = gm.sample_counts(x, 9, (7 << 32) | 5, 1, 33, n, sigma)
        for engine in (0, 1):
            gm.set_option("engine", engine)
            np.testing.assert_array_equal(gm.sample_counts_static(x, 9, (7 << 32) | 5, 1, 33, n, sigma), expected)
        gm.set_option("engine", 0)
