"""The library's host code without a GPU: which kernels a call takes, and what it asks of the CUDA runtime for them.

Every test runs in a process of its own in which a stand-in for the CUDA runtime (host/fake_cudart.c) is preloaded:
device memory is host memory, kernels do nothing, launches are recorded and are refused for the reason for which the
real runtime refuses them (more dynamic shared memory than the kernel was granted on the current device)."""
import ctypes as C
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="session")
def fake_runtime(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libfakecudart.so")
    subprocess.run(["gcc", "-O1", "-Wall", "-shared", "-fPIC", "-pthread", "-I", "/usr/local/cuda/include", "-o", so,
                    os.path.join(HERE, "host", "fake_cudart.c")], check=True)
    return so


# ------------------------------------------------------------------ in the process with the stand-in

def _fake():
    f = C.CDLL(os.environ["LD_PRELOAD"])
    f.fake_launch_name.restype = C.c_char_p
    f.fake_allocated.restype = C.c_size_t
    f.fake_watch.argtypes = [C.c_void_p]
    f.fake_launch_word.restype = C.c_ulonglong
    f.fake_set_largest.argtypes = [C.c_size_t]
    return f


def _kernels(f):
    names = ("k_line", "k_stem", "k_halo", "k_igemm", "k_first_conv", "k_conv", "k_gavgpool", "k_maxpool", "k_votes")
    return [next(n for n in names if n in f.fake_launch_name(i).decode()) for i in range(f.fake_launches())]


def _hidden_layer_net(wl, cin, cout):
    """stem -> 1 x 1 convolution from `cin` to `cout` channels -> pool -> FC"""
    rng = wl.SplitMix64(5)
    L = [wl._conv(rng, 0, 3, cin, 3, 1, 1, True, 3, -128), wl._conv(rng, 1, cin, cout, 1, 1, 0, True, -128, -128),
         wl._gavgpool(2, cout, 16, -128), wl._conv(rng, 3, cout, 5, 1, 1, 0, False, -128, 0, op=wl.OP_FC)]
    return dict(in_shape=(3, 4, 4), n_classes=5, layers=L)


def layer_too_wide_for_shared_memory():
    """The implicit-GEMM kernel keeps a layer's constants in shared memory: a layer whose constants leave no room for two
    operand stages runs on the plain kernel, through every entry point."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    for cin, cout, kernel in ((24, 6912, "k_igemm"), (24, 6913, "k_conv"), (24, 8200, "k_conv"), (64, 10112, "k_igemm"), (64, 10240, "k_conv")):
        model = _hidden_layer_net(wl, cin, cout)
        gm = isc.Model(model)
        x = wl.images(1, shape=model["in_shape"])[0]
        for call in (gm.sample_counts, gm.sample_counts_static):
            f.fake_reset()
            call(x, 1, 0, 1, 0, 9, 0.25)
            assert _kernels(f) == ["k_stem", kernel, "k_gavgpool", "k_igemm", "k_votes"], (cin, cout, _kernels(f))


def _filter_net(wl):
    """a network whose kernels need more shared memory than a launch has by default: stem, resident filter, 1 x 1, FC"""
    rng = wl.SplitMix64(6)
    L = [wl._conv(rng, 0, 3, 96, 7, 1, 3, True, 3, -128), wl._conv(rng, 1, 96, 96, 3, 1, 1, True, -128, -128),
         wl._conv(rng, 2, 96, 256, 1, 1, 0, True, -128, -128), wl._gavgpool(3, 256, 24 * 36, -128),
         wl._conv(rng, 4, 256, 5, 1, 1, 0, False, -128, 0, op=wl.OP_FC)]
    return dict(in_shape=(3, 24, 36), n_classes=5, layers=L)


def first_calls_in_two_threads():
    """Two handles used for the first time at once: neither may launch before the kernels' shared-memory limits are raised,
    however long that takes the other."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    model = _filter_net(wl)
    x = wl.images(1, shape=model["in_shape"])[0]
    handles = [isc.Model(model) for _ in range(2)]
    f.fake_set_attribute_delay(200_000)
    failed = []

    def first_call(gm, wait_s):
        time.sleep(wait_s)
        try:
            gm.sample_counts(x, 1, 0, 1, 0, 9, 0.25)
        except isc.IscError as e:
            failed.append(e)
    threads = [threading.Thread(target=first_call, args=a) for a in zip(handles, (0.0, 0.1))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    assert sorted(set(_kernels(f))) == ["k_gavgpool", "k_halo", "k_igemm", "k_stem", "k_votes"]


def every_device():
    """Shared-memory limits are a property of each device: handles on two devices work in one process, and so does a handle
    that is used with another device current than before (its memory being visible there)."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    for model, kernels in ((_filter_net(wl), ["k_gavgpool", "k_halo", "k_igemm", "k_stem", "k_votes"]), (wl.resnet20(), ["k_line"])):
        x = wl.images(1, shape=model["in_shape"])[0]
        handles = []
        for device in (0, 1):
            f.fake_set_device(device)
            handles.append(isc.Model(model))
        for device, gm in ((0, handles[0]), (1, handles[1]), (2, handles[0]), (0, handles[0]), (3, handles[1])):
            f.fake_set_device(device)
            for call in (gm.sample_counts, gm.sample_counts_static):
                f.fake_reset()
                call(x, 1, 0, 1, 0, 9, 0.25)
                assert sorted(set(_kernels(f))) == kernels
                assert all(f.fake_launch_ok(i) and f.fake_launch_device(i) == device for i in range(f.fake_launches()))


def device_images_of_any_alignment():
    """The kernels read an image's rows as 32-bit words: device images are read in place where their address allows that,
    and from an aligned copy where it does not."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    for model in (wl.resnet20(), _filter_net(wl)):
        gm = isc.Model(model)
        size = int(np.prod(model["in_shape"]))
        room = np.zeros(2 * size + 64, np.uint8)
        base = (room.ctypes.data + 15) // 16 * 16
        for offset in (0, 1, 2, 3, 4, 7):
            f.fake_reset()
            f.fake_watch(base + offset)
            gm.certify_batch(None, 2, 1, 0, 5, 9, 0.25, 0.001, device_ptr=base + offset)
            assert any(f.fake_launch_watched(i) for i in range(f.fake_launches())) == (offset % 4 == 0), offset


def static_entry_point_takes_the_engine_it_is_told():
    """The allocation-free entry point takes the engine that isc_sample_counts takes under the same option, and refuses what
    that refuses, launching nothing."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    for model in (wl.resnet20(), _filter_net(wl)):
        gm = isc.Model(model)
        x = wl.images(1, shape=model["in_shape"])[0]
        for engine in (0, 1, 2, 3):
            gm.set_option("engine", engine)
            taken = []
            for call in (gm.sample_counts, gm.sample_counts_static):
                f.fake_reset()
                try:
                    call(x, 1, 0, 1, 0, 9, 0.25)
                except isc.IscError as e:
                    assert e.code == -3 and f.fake_launches() == 0
                taken.append(_kernels(f))
            assert taken[0] == taken[1], (engine, taken)
            assert ("k_line" in taken[1]) == (gm.get_info("has_line_engine") == 1 and engine in (0, 3))
            if taken[1]:
                assert gm.get_info("static_engine") == (engine or (3 if gm.get_info("has_line_engine") else 2))
            assert bool(taken[1]) == (engine != 3 or gm.get_info("has_line_engine") == 1)


def weights_are_on_the_device_once_per_kernel():
    """A filter layer's weights are uploaded for the plain kernel and for the one tensor-core kernel that takes the layer."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    rng = wl.SplitMix64(6)
    L = [wl._conv(rng, 0, 3, 256, 3, 1, 1, True, 3, -128), wl._conv(rng, 1, 256, 256, 3, 1, 1, True, -128, -128),
         wl._gavgpool(2, 256, 24 * 24, -128), wl._conv(rng, 3, 256, 5, 1, 1, 0, False, -128, 0, op=wl.OP_FC)]
    gm = isc.Model(dict(in_shape=(3, 24, 24), n_classes=5, layers=L))
    assert 2.0 <= f.fake_allocated() / L[1]["w"].size < 2.3
    gm.close()


def side_streams_keep_the_callers_priority():
    """Short launches are dealt to side streams of the engine's own: with the priority of the stream that the call is on."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    gm = isc.Model(wl.tiny_cnn())
    gm.set_option("batch", 64)
    x = wl.images(1)[0]
    for device, priority in ((0, 0), (0, -5), (0, -5), (0, -1), (1, -1), (0, None)):
        f.fake_set_device(device)
        stream = C.c_void_p()
        if priority is not None:
            f.cudaStreamCreateWithPriority(C.byref(stream), 1, priority)
        f.fake_reset()
        gm.sample_counts(x, 1, 0, 1, 0, 500, 0.25, stream=stream.value)
        assert f.fake_launches() == 8
        for i in range(8):
            assert (f.fake_launch_priority(i), f.fake_launch_stream_device(i)) == (priority or 0, device)


def _every_kernel_net(wl):
    """stem, max-pool, 3 x 3 with resident weights, 3 x 3 with a ring of them, 1 x 1, pool, FC"""
    rng = wl.SplitMix64(6)
    L = [wl._conv(rng, 0, 3, 64, 5, 1, 2, True, 3, -128), wl._maxpool(1, 64, 3, 2, 1, -128), wl._conv(rng, 2, 64, 64, 3, 1, 1, True, -128, -128),
         wl._conv(rng, 3, 64, 256, 3, 1, 1, True, -128, -128), wl._conv(rng, 4, 256, 64, 1, 1, 0, True, -128, -128),
         wl._gavgpool(5, 64, 100, -128), wl._conv(rng, 6, 64, 7, 1, 1, 0, False, -128, 0, op=wl.OP_FC)]
    return dict(in_shape=(3, 20, 20), n_classes=7, layers=L)


def stalled_launches_reach_every_kernel():
    """The probe of the bounded waits launches the kernel that runs the layer, and refuses layers without one."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    gm = isc.Model(_every_kernel_net(wl))
    gm.set_option("engine", 2)
    x = wl.images(1, shape=(3, 20, 20))[0]
    gm.sample_counts(x, 1, 0, 1, 0, 9, 0.25)
    taken = _kernels(f)
    assert taken == ["k_stem", "k_maxpool", "k_halo", "k_halo", "k_igemm", "k_gavgpool", "k_igemm", "k_votes"]
    for layer, kernel in enumerate(taken[:-1]):
        f.fake_reset()
        tensor_cores = kernel in ("k_stem", "k_halo", "k_igemm")
        assert gm.debug_stalled_launch(layer)[0] == (0 if tensor_cores else -3)      # 0: the stand-in's kernels raise no error word
        assert _kernels(f) == ([kernel] if tensor_cores else [])


def bins_hold_the_levels_of_the_search():
    """The noise law's table of bins against the search in its cumulative table: every boundary between two levels and the
    uniforms beside it, both ends, the middle, the edges of all bins, and random ones."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    gm = isc.Model(wl.tiny_cnn())
    x = wl.images(1)[0]
    rng = np.random.default_rng(1)
    sizes = {}
    for noise in (0, 1):
        gm.set_option("noise", noise)
        for sigma in (1e-4, 0.001, 0.003, 0.01, 0.12, 0.25, 0.4, 0.5, 0.65, 0.7, 1.0, 1.31, 1.32, 2.0, 40.0):
            f.fake_reset()
            gm.sample_counts(x, 1, 0, 1, 0, 1, sigma)
            word = [f.fake_launch_word(0, k) for k in range(20)]
            bits = sizes[noise, sigma] = word[19] & 0xFFFFFFFF if word[18] else 0
            if not bits:
                continue
            cum = isc.noise_table(sigma, rounded=bool(noise)).astype(np.int64)
            T = cum.size // 2
            side = (10 << bits) + 2
            bins = np.frombuffer(C.string_at(word[18], 16 * side), np.uint32).astype(np.int64).reshape(2, side, 2)
            # distances from the end at which bins begin
            edges = np.concatenate([((1 << bits) + np.arange(1 << bits)) << (21 + o - bits) for o in range(10)]) - 2 ** 21
            near = np.concatenate([cum, edges, 2 ** 32 - 1 - edges, [0, 2 ** 31, 2 ** 31 - 2 ** 21, 2 ** 31 + 2 ** 21, 2 ** 32 - 1]])
            u = np.clip(np.concatenate([near + d for d in (-1, 0, 1)] + [rng.integers(0, 2 ** 32, 200_000)]), 0, 2 ** 32 - 1)
            want = np.minimum(np.searchsorted(cum, u, side="right"), 2 * T) - T
            upper = (u >> 31).astype(int)
            sums = np.where(upper == 1, 2 ** 32 - 1 - u, u) + 2 ** 21
            e = np.frexp(sums.astype(np.float64))[1] - 1
            at = ((e - 21) << bits) + (sums >> (e - bits)) - (1 << bits)
            bound, level = bins[upper, at, 0], bins[upper, at, 1]
            level = np.where(level >= 2 ** 31, level - 2 ** 32, level)
            known = level != 1 << 30
            np.testing.assert_array_equal((level + (u >= bound))[known], want[known])
            assert known[-200_000:].mean() > 1 - 2 ** -10
    assert {s: b for (n, s), b in sizes.items() if n == 0} == {1e-4: 6, 0.001: 6, 0.003: 6, 0.01: 6, 0.12: 6, 0.25: 6, 0.4: 7, 0.5: 7, 0.65: 7, 0.7: 8, 1.0: 8, 1.31: 8, 1.32: 0, 2.0: 0, 40.0: 0}


def batches_shrink_to_the_memory_there_is():
    """A call whose default batch the device's memory does not hold takes a smaller one, and later calls do not try in vain."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    model = _filter_net(wl)
    per_sample = 24 * 36 * 256                                    # the largest activation tensor
    x = wl.images(1, shape=model["in_shape"])[0]
    for engine in (1, 2):
        gm = isc.Model(model)
        gm.set_option("engine", engine)
        launches = lambda: sum(k in ("k_stem", "k_first_conv") for k in _kernels(f))
        cap = 3 * 2 ** 30 // (24 * 36 * (96 + 256))               # 3 GiB of two buffers
        def call(n):
            f.fake_reset()
            gm.sample_counts(x, 1, 0, 1, 0, n, 0.25)
            return launches()
        f.fake_set_largest(2 ** 62)
        assert call(500) == 1
        f.fake_set_largest(1000 * per_sample)
        assert call(5000) == -(-5000 // 625) and f.fake_refused() == 3       # 5,000, 2,500 and 1,250 do not fit
        assert call(5000) == 8 and call(100) == 1 and f.fake_refused() == 3
        gm.certify_batch(wl.images(3, shape=model["in_shape"]), 3, 1, 0, 100, 900, 0.25, 0.001)
        assert f.fake_refused() == 3
        f.fake_set_largest(2 ** 62)
        gm.set_option("batch", 0)
        assert call(5000) == -(-5000 // cap) < 8
        gm.close()
        gm = isc.Model(model)
        gm.set_option("engine", engine)
        f.fake_set_largest(per_sample - 1)
        with pytest.raises(isc.IscError) as e:
            gm.sample_counts(x, 1, 0, 1, 0, 5, 0.25)
        assert e.value.code == -4


def resident_plans_order_rows_of_other_bands():
    """Maps of 16 x 16 lie in two bands whose edge rows are copied into each other's padding.  Only a stacked filter on the
    output of the convolution before it waits, through its rows above and below, for those copies' readers and writers
    one by one; any other convolution has to wait for all of the one before."""
    import paper_2108_09413_b200 as isc
    import workloads as wl
    f = _fake()
    rng = wl.SplitMix64(6)

    def record(at, count, dtype=np.uint32):
        return np.frombuffer(C.string_at(int(at), count * np.dtype(dtype).itemsize), dtype)

    def blobs(layers, side):
        n, c = len(layers), layers[-1]["cout"]
        layers = layers + [wl._gavgpool(n, c, side * side, -128), wl._conv(rng, n + 1, c, 5, 1, 1, 0, False, -128, 0, op=wl.OP_FC)]
        gm = isc.Model(dict(in_shape=(3, 32, 32), n_classes=5, layers=layers))
        gm.set_option("engine", 3)
        f.fake_reset()
        gm.sample_counts(wl.images(1)[0], 1, 0, 1, 0, 9, 0.25)
        params = np.array([f.fake_launch_word(0, k) for k in range(5)], np.uint64)       # phase table, blobs' sources, counts, (barriers, phases), (convolutions, ..)
        for k in range(int(params[4] & 0xFFFFFFFF)):
            yield int(record(int(params[1]) + 32 * k, 1, np.uint64)[0])

    def wait_for_all(layers, side):
        """per convolution: whether each issuing thread's first record waits for all of the convolution before"""
        out = []
        for blob in blobs(layers, side):
            n_ops, _, ops = record(blob + 112, 3)
            assert n_ops >= 3
            out.append([bool(record(blob + int(ops) + 32 * r + 30, 1, np.uint16)[0] & 1) for r in range(3)])
        assert all(len(set(w)) == 1 for w in out)
        return [w[0] for w in out]

    conv = lambda t, cin, cout, k, stride=1, res=-1: wl._conv(rng, t, cin, cout, k, stride, k // 2, True, 3 if t == 0 else -128, -128, res, -128)
    stem = [conv(0, 3, 16, 3), conv(1, 16, 32, 3, 2)]                        # tensor 2: 32 x 16 x 16, in two bands
    # 1 x 1 in place over tensor 3; a filter on an older tensor than the last, over the last one's input
    assert wait_for_all(stem + [conv(2, 32, 32, 3), conv(3, 32, 32, 3), conv(4, 32, 32, 1, res=3), conv(5, 32, 32, 3)], 16)[3:] == [False, True, False]
    assert wait_for_all(stem + [conv(2, 32, 32, 3), conv(3, 32, 32, 3), conv(2, 32, 32, 3, res=4)], 16)[3:] == [False, True]
    # one band: rows above and below the map are padding
    assert wait_for_all([conv(0, 3, 16, 3), conv(1, 16, 16, 3), conv(2, 16, 16, 1)], 32)[1:] == [False, False]
    # basic blocks need no such wait
    assert not any(wait_for_all(wl.resnet20()["layers"][:-2], 8))
    # a residual term without the form of a product, or whose constant has no room beside the product, keeps the fast pass
    for res_mult, zp, shift, flags in ((1304428746, 77, 9, 2 | 4), (1798879234, -20, 14, 2 | 4), (1798879234, -20, 9, 2), (1304428746, -128, 9, 2)):
        layers = [conv(0, 3, 16, 3), conv(1, 16, 16, 3), conv(2, 16, 16, 3, res=1)]
        for layer in layers:
            layer.update(zp_in=3 if layer is layers[0] else zp, zp_out=zp, zp_res=zp, relu=0, shift=np.full(16, shift, np.int8))
        layers[2].update(res_mult=res_mult, res_shift=0)
        layers = layers + [dict(conv(3, 16, 32, 3, 2), zp_in=zp)]
        assert [int(record(blob, 1)[0]) & (2 | 4 | 16) for blob in blobs(layers, 16)][2] == flags


# ------------------------------------------------------------------ the tests

SCENARIOS = [layer_too_wide_for_shared_memory, first_calls_in_two_threads, every_device, device_images_of_any_alignment,
             static_entry_point_takes_the_engine_it_is_told, weights_are_on_the_device_once_per_kernel,
             side_streams_keep_the_callers_priority, resident_plans_order_rows_of_other_bands,
             batches_shrink_to_the_memory_there_is, bins_hold_the_levels_of_the_search, stalled_launches_reach_every_kernel]


@pytest.mark.parametrize("scenario", [s.__name__ for s in SCENARIOS])
def test_host_code(scenario, fake_runtime):
    r = subprocess.run([sys.executable, os.path.abspath(__file__), scenario], cwd=ROOT, timeout=300, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=fake_runtime, PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]


if __name__ == "__main__":
    globals()[sys.argv[1]]()
