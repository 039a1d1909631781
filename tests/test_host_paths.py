"""Host-side paths of the library that need no GPU: per-device state, fallbacks
and launch plans, against a stand-in for the CUDA runtime (fake_cudart.cpp)."""
import ctypes
import shutil

import numpy as np
import pytest

from paper_2108_08591_gb300 import _lib

pytestmark = pytest.mark.skipif(not shutil.which("g++"), reason="g++ not found")


@pytest.fixture(scope="module")
def linked(tmp_path_factory):
    from _fakecuda import Fake, link
    out = tmp_path_factory.mktemp("fake") / "libmdf_fake.so"
    link(out)
    return Fake(out)


@pytest.fixture
def fake(linked):
    linked.lib.fake_reset()
    linked.new_device()
    return linked


def test_kernel_attributes_are_set_on_every_device(fake):
    """Shared memory and cluster sizes beyond the defaults are a device's own:
    a handle on a second GPU of the process launches as on the first."""
    lib = fake.lib
    conv = [np.zeros(8 * 8 * 64 * 64, np.float32) for _ in range(3)]
    x, w, y = ((a.ctypes.data + 63) // 64 * 64 for a in conv)
    got = []
    for dev in (fake.device, fake.new_device()):
        lib.fake_set_device(dev)
        for shape, q in (((64, 64), 0), ((40, 60), 4), ((60, 60, 200), 0), ((60, 60, 200), 6)):
            h = fake.lattice(shape, q=q)
            assert lib.mdf_step(h, 6) == _lib.OK, (dev, shape, lib.mdf_last_error(h))
            lib.mdf_destroy(h)
        b = fake.batch([65, 97, 129])
        assert lib.mdf_batch_step(b, 10) == _lib.OK, (dev, lib.mdf_batch_last_error(b))
        lib.mdf_batch_destroy(b)
        for which in (2, 1):
            assert lib.mdf_nn_set_conv_kernel(which) == _lib.OK
            assert lib.mdf_nn_conv_fwd(x, w, None, y, None, 1, 64, 64, 32, 32, 0, None) == _lib.OK, (dev, which)
        assert lib.mdf_nn_set_conv_kernel(2) == _lib.OK
        assert lib.mdf_nn_set_halo_tile(2, 16) == _lib.OK
        assert lib.mdf_nn_conv_fwd(x, w, None, y, None, 1, 64, 64, 32, 32, 0, None) == _lib.OK, dev
        assert lib.mdf_nn_set_halo_tile(0, 0) == _lib.OK
        assert lib.mdf_nn_conv_wgrad(x, x, y, w, 1, 64, 64, 32, 32, None) == _lib.OK, dev
        got.append([(n, *rest) for n, d, *rest in fake.launches() if d == dev])
    assert got[0] == got[1]
    for kernel in ("k_resident2d", "k_update_fused3d", "k_batch_resident", "k_conv_fwd_pers", "k_conv_fwd_halo",
                   "k_conv_fwd_tc", "k_conv_wgrad_tma"):
        assert any(kernel in n for n, *_ in got[1]), kernel


def _step_kernels(fake, b):
    fake.launches()
    assert fake.lib.mdf_batch_step(b, 8) == _lib.OK, fake.lib.mdf_batch_last_error(b)
    return {n for n, *_ in fake.launches() if "batch_tick" not in n}


def test_batch_falls_back_where_its_faster_path_cannot_be_set_up(fake):
    """A cluster query or an allocation that only the fused launches need does
    not fail the creation of a batch: it goes by fused launches, or by the
    persistent kernel."""
    lib = fake.lib
    b = fake.batch([65, 97])
    assert all("k_batch_resident" in n for n in _step_kernels(fake, b))
    lib.mdf_batch_destroy(b)
    lib.fake_fail_clusters(1)
    b = fake.batch([65, 97])
    assert all("k_batch_fused" in n for n in _step_kernels(fake, b))
    lib.mdf_batch_destroy(b)
    lib.fake_fail_clusters(0)
    side, Re = (ctypes.c_int * 2)(65, 97), (ctypes.c_double * 2)(100.0, 100.0)
    got = []
    for k in range(1, 40):  # the k-th allocation fails
        lib.fake_fail_malloc(k)
        b = ctypes.c_void_p()
        st = lib.mdf_batch_create(ctypes.byref(b), 2, 2, side, Re, 0.1, None)
        lib.fake_fail_malloc(0)
        if st != _lib.OK:
            assert st == _lib.ENOMEM
            got.append("refused")
            continue
        kinds = _step_kernels(fake, b)
        got.append(next(n for n in ("chunk", "fused", "resident") if any(n in x for x in kinds)))
        lib.mdf_batch_destroy(b)
    # the state's own, the lists of fused launches, the seats on chip, none
    order = [g for k, g in enumerate(got) if k == 0 or g != got[k - 1]]
    assert order == ["refused", "chunk", "fused", "resident"], got


class _Items(ctypes.Structure):  # of the fused batch kernel: lists, their lengths
    _fields_ = [("list", ctypes.c_void_p * 3), ("n", ctypes.c_int * 3), ("wave", ctypes.c_int)]


@pytest.mark.parametrize("sides", [[300] * 4, [240, 175], [113, 267, 56], [870, 600], [61, 1100], [1921, 2]])
@pytest.mark.parametrize("K", [2, 4])
def test_fused_batch_items_cover_every_box_once(fake, sides, K):
    """Each list of a fused launch of K updates covers every node once, with no
    strip (64 columns less the K lost on each side) beyond its box."""
    lib, out = fake.lib, {2: 60, 4: 56}[K]
    lib.fake_clusters(0)  # boxes that would fit on chip as well
    b = fake.batch(sides)
    lib.fake_watch(b"k_batch_fusedILi%d" % K, 1, ctypes.sizeof(_Items))
    # 16 updates make launches of the batch's depth, a period of 6 one of the other
    assert lib.mdf_batch_step(b, 18) == _lib.OK
    st = [np.zeros(len(sides), t) for t in (np.int64, np.int32, np.float64)]
    lib.mdf_batch_run(b, 1e-8, 6, 6, *(v.ctypes.data for v in st))
    it = fake.watched(_Items)
    assert it.n[0] > 0
    for l in range(3):
        items = np.ctypeslib.as_array((ctypes.c_int * (4 * it.n[l])).from_address(it.list[l])).reshape(-1, 4)
        cover = [np.zeros((N, N), np.int8) for N in sides]
        for c, s, y0, y1 in items:
            assert s * out < sides[c], (l, c, s)
            assert 0 <= y0 < y1 <= sides[c]
            cover[c][y0:y1, s * out:(s + 1) * out] += 1
        assert all((v == 1).all() for v in cover), l
    lib.mdf_batch_destroy(b)


@pytest.mark.parametrize("storage", ["f16eq", "bf16eq"])
@pytest.mark.parametrize("shape,walled,open_", [((2050, 1998), 64, 96), ((2098, 40), 64, 96), ((1024, 64), 64, 64)])
def test_walled_2d_equilibrium_shifted_rows_keep_their_block(fake, storage, shape, walled, open_):
    got = []
    for wall in (True, False):
        h = fake.lattice(shape, storage, wall=wall)
        fake.launches()
        assert fake.lib.mdf_step(h, 1) == _lib.OK
        got += [threads for n, _, _, threads, _ in fake.launches() if "k_update_eq" in n]
        fake.lib.mdf_destroy(h)
    assert got == [walled, open_]


@pytest.mark.parametrize("sides,kernel,per_update,arg", [([300, 240], "k_batch_fused", 2 * 5.0, -1),
                                                         ([65, 97, 129], "k_batch_resident", 5.0, 4)])
def test_batch_autotune_weighs_warm_kernels(fake, sides, kernel, per_update, arg):
    """The first launch of a kernel loads it.  That does not count against the
    fused or on-chip launches, which stay in use when they are the faster ones,
    also after a schedule of the caller's own."""
    lib = fake.lib
    lib.fake_cost(kernel.encode(), per_update, 1e5, arg)
    lib.fake_cost(b"k_batch_chunk", 10.0, 1e5, 2)  # us per update
    b = fake.batch(sides)
    assert lib.mdf_batch_autotune(b, 20, None, None, None) == _lib.OK
    assert all(kernel in n for n in _step_kernels(fake, b))
    assert lib.mdf_batch_set_schedule(b, 64, 0, 3) == _lib.OK
    assert all("k_batch_chunk" in n for n in _step_kernels(fake, b))
    assert lib.mdf_batch_autotune(b, 20, None, None, None) == _lib.OK
    assert all(kernel in n for n in _step_kernels(fake, b))
    lib.mdf_batch_destroy(b)


def test_batch_autotune_keeps_the_persistent_kernel_where_it_is_faster(fake):
    lib = fake.lib
    lib.fake_cost(b"k_batch_fused", 2 * 12.0, 0.0, -1)
    lib.fake_cost(b"k_batch_chunk", 10.0, 0.0, 2)
    b = fake.batch([300, 240])
    assert all("k_batch_fused" in n for n in _step_kernels(fake, b))
    assert lib.mdf_batch_autotune(b, 20, None, None, None) == _lib.OK
    assert all("k_batch_chunk" in n for n in _step_kernels(fake, b))
    lib.mdf_batch_destroy(b)
