"""How a call's samples are cut into launches must not show: several images per launch, several pieces of a batch, and
launches that overlap on side streams give the counts of one image and one phase at a time."""
import numpy as np
import pytest

import workloads as wl
import paper_2108_09413_b200 as isc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_images,N0,N", [(1, 1, 1), (3, 100, 593), (5, 7, 18001), (9, 100, 4097)])
@pytest.mark.parametrize("launch", [0, 100, 1024, 30000])
def test_images_and_phases_share_launches(n_images, N0, N, launch):
    gm = isc.Model(wl.spread_model("tiny_cnn"))
    xs = np.stack([np.roll(wl.spread_image(), i, axis=2) for i in range(n_images)])
    image_id0 = (1 << 32) - 2                      # the ids of one launch cross 2^32
    gm.set_option("batch", launch)
    c0, c1 = gm.certify_batch(xs, n_images, 11, image_id0, N0, N, 0.25, 0.001)[2:]
    gm.set_option("batch", 0)
    for i in range(n_images):
        np.testing.assert_array_equal(c0[i], gm.sample_counts(xs[i], 11, image_id0 + i, 0, 0, N0, 0.25))
        np.testing.assert_array_equal(c1[i], gm.sample_counts(xs[i], 11, image_id0 + i, 1, 0, N, 0.25))
