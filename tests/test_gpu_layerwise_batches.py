"""How the layer-by-layer engine cuts a call's samples into batches must not show: several images and both phases in one
chain of launches give the counts of one image and one phase at a time, and the CPU oracle's for a call's first samples."""
import numpy as np
import pytest

import oracle
import workloads as wl
import paper_2108_09413_b200 as isc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [1, 2])
@pytest.mark.parametrize("n_images,N0,N", [(1, 1, 1), (3, 10, 53), (5, 7, 301), (2, 100, 9000)])
@pytest.mark.parametrize("batch", [0, 1, 64, 100])
def test_images_and_phases_share_batches(engine, n_images, N0, N, batch):
    if batch == 1 and N > 400:
        batch = 333
    model = wl.tiny_cnn()
    gm = isc.Model(model)
    gm.set_option("engine", engine)
    xs = wl.images(n_images, shape=model["in_shape"])
    image_id0 = (1 << 32) - 2                      # the ids of one chain cross 2^32
    gm.set_option("batch", batch)
    c0, c1 = gm.certify_batch(xs, n_images, 11, image_id0, N0, N, 0.25, 0.001)[2:]
    assert gm.get_info("engine") == engine
    gm.set_option("batch", 0)
    for i in range(n_images):
        np.testing.assert_array_equal(c0[i], gm.sample_counts(xs[i], 11, image_id0 + i, 0, 0, N0, 0.25))
        np.testing.assert_array_equal(c1[i], gm.sample_counts(xs[i], 11, image_id0 + i, 1, 0, N, 0.25))
    if N <= 53:
        om = oracle.Model(model)
        for i in range(n_images):
            for phase, n, got in ((0, N0, c0), (1, N, c1)):
                np.testing.assert_array_equal(got[i], oracle.sample_counts(om, xs[i], 11, image_id0 + i, phase, 0, n, 0.25))


@pytest.mark.parametrize("engine", [1, 2])
@pytest.mark.parametrize("classes", [1, 15, 16, 31, 32, 33, 63, 64, 100, 129, 511, 512, 1000, 1025])
def test_votes_and_logits_of_any_number_of_classes(engine, classes):
    rng = np.random.default_rng(classes)
    model = wl.tiny_cnn()
    fc = dict(model["layers"][-1], cout=classes, w=rng.integers(-3, 4, (classes, 32, 1, 1)).astype(np.int8), bias=np.zeros(classes, np.int32),
              mult=np.full(classes, 1 << 30, np.int32), shift=np.full(classes, 4, np.int8))            # small logits: ties for the first place
    model = dict(model, n_classes=classes, layers=model["layers"][:-1] + [fc])
    gm, om = isc.Model(model), oracle.Model(model)
    x = wl.images(1, shape=model["in_shape"])[0]
    gm.set_option("engine", engine)
    for n in (1, 3, 77):
        counts, logits = gm.sample_counts(x, 11, 2, 1, 5, n, 0.25, want_logits=True)
        want = oracle.sample_counts(om, x, 11, 2, 1, 5, n, 0.25, want_logits=True)
        np.testing.assert_array_equal(logits, want[1])
        np.testing.assert_array_equal(counts, want[0])
        np.testing.assert_array_equal(gm.sample_counts(x, 11, 2, 1, 5, n, 0.25), want[0])
    c0, c1 = gm.certify_batch(wl.images(2, shape=model["in_shape"]), 2, 11, 2, 9, 50, 0.25, 0.001)[2:] if classes > 1 else (None, None)
    if classes > 1:
        assert (c0.sum(1) == 9).all() and (c1.sum(1) == 50).all()
