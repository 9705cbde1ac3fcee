"""The resident engine's noise and tail phases at the ends of their ranges: pooled maps of 8 x 8, 16 x 16 and 32 x 32
pixels, 16 to 64 channels (48 does not divide the CTA's threads), 1 to 4 input channels, 1 to 128 classes, sample counts
that leave a group partly empty."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_c,widths,classes", [(1, (16,), 1), (3, (16, 32, 48), 33), (4, (16, 32), 128), (2, (16,), 32), (3, (16, 32, 64), 100)])
def test_pooled_maps_and_classes(in_c, widths, classes):
    rng = wl.SplitMix64(77 + classes)
    Z = wl.RELU_ZP
    L = [wl._conv(rng, 0, in_c, widths[0], 3, 1, 1, True, 3, Z)]
    for i, w in enumerate(widths[1:]):
        L.append(wl._conv(rng, len(L), widths[i], w, 3, 2, 1, True, Z, Z))
    size = 32 >> (len(widths) - 1)
    L.append(wl._gavgpool(len(L), widths[-1], size * size, Z))
    L.append(wl._conv(rng, len(L), widths[-1], classes, 1, 1, 0, False, Z, 0, op=wl.OP_FC))
    model = dict(in_shape=(in_c, 32, 32), n_classes=classes, layers=L)
    x = wl.images(1, shape=model["in_shape"], seed=4)[0]
    gm, om = isc.Model(model), oracle.Model(model)
    assert gm.get_info("has_line_engine") == 1
    for n in (1, 37):
        counts, logits = gm.sample_counts(x, 5, 3, 1, 11, n, 0.5, want_logits=True)
        ecounts, elogits = oracle.sample_counts(om, x, 5, 3, 1, 11, n, 0.5, want_logits=True)
        np.testing.assert_array_equal(logits, elogits)
        np.testing.assert_array_equal(counts, ecounts)
