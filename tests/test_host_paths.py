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
    Re = (ctypes.c_double * 2)(100.0, 100.0)
    # the state's own allocations, then the seats on chip or the item lists, then none
    for sides, want in (((65, 97), ["refused", "fused", "resident"]), ((300, 240), ["refused", "chunk", "fused"])):
        got = []
        for k in range(1, 40):  # the k-th allocation fails
            lib.fake_fail_malloc(k)
            b = ctypes.c_void_p()
            st = lib.mdf_batch_create(ctypes.byref(b), 2, 2, (ctypes.c_int * 2)(*sides), Re, 0.1, None)
            lib.fake_fail_malloc(0)
            if st != _lib.OK:
                assert st == _lib.ENOMEM
                got.append("refused")
                continue
            kinds = _step_kernels(fake, b)
            got.append(next(n for n in ("chunk", "fused", "resident") if any(n in x for x in kinds)))
            lib.mdf_batch_destroy(b)
        assert [g for k, g in enumerate(got) if k == 0 or g != got[k - 1]] == want, got


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


def _count(fake, step):
    """(update kernels launched, threads of the last) of a call."""
    fake.launches()
    assert step() == _lib.OK
    return [(n, threads) for n, _, _, threads, _ in fake.launches() if "set_clock" not in n]


@pytest.mark.parametrize("shape,storage,opts", [
    ((64, 64), "f32", {}), ((1200, 16), "f32", {}), ((129, 130), "f32", {"q": 4}), ((300, 300), "f32", {}),
    ((1003, 751), "f32", {}), ((400001, 2), "f32", {}), ((250001, 3), "f32", {}), ((1003, 751), "f32", {"vx": 1}),
    ((1003, 751), "f32", {"inplace": 1}), ((1003, 751), "f16", {}), ((64, 64), "f64", {}), ((60, 60, 200), "f32", {}),
    ((64, 64, 64), "f32", {}), ((60, 60, 200), "f16eq", {}), ((119, 121, 151), "f32", {"q": 6, "wall": True})])
def test_plan_is_what_a_step_launches(fake, shape, storage, opts):
    h = fake.lattice(shape, storage, **opts)
    kernels = {0: "k_update", 1: "k_update_fused", 2: "k_resident2d"}
    for n in (0, 1, 2, 3, 4, 7, 70):
        p = _lib.Plan()
        assert fake.lib.mdf_plan(h, n, ctypes.byref(p)) == _lib.OK
        got = _count(fake, lambda: fake.lib.mdf_step(h, n))
        assert p.launches == len(got), n
        assert p.updates * p.launches >= n
        if n:
            assert kernels[p.path] in got[0][0] and got[0][1] == p.threads, (n, got)
            assert ("fused" in got[0][0]) == (p.path == 1)
    p = _lib.Plan()
    assert fake.lib.mdf_plan(h, 10**12, ctypes.byref(p)) == _lib.OK and p.launches * p.updates >= 10**12
    assert fake.lib.mdf_plan(h, -1, ctypes.byref(p)) == _lib.EINVAL
    assert fake.lib.mdf_plan(h, 1, None) == _lib.EINVAL
    fake.lib.mdf_destroy(h)


def test_plan_of_a_long_run_on_chip(fake):
    h = fake.lattice((64, 64))
    p = _lib.Plan()
    assert fake.lib.mdf_plan(h, 40001, ctypes.byref(p)) == _lib.OK
    assert (p.path, p.updates, p.launches, p.threads) == (2, 16384, 3, 256)
    assert len(_count(fake, lambda: fake.lib.mdf_step(h, 40001))) == 3
    fake.lib.mdf_destroy(h)


def test_plan_struct_matches_the_header(tmp_path):
    """As tests/test_abi.py checks the other structs."""
    import os
    import subprocess
    src = tmp_path / "layout.c"
    src.write_text('#include <stdio.h>\n#include <stddef.h>\n#include "mdf.h"\nint main(void) {\n'
                   + "".join(f'printf("%zu ", offsetof(mdf_plan_t, {f}));' for f, _ in _lib.Plan._fields_)
                   + 'printf("%zu", sizeof(mdf_plan_t)); return 0; }\n')
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include")
    subprocess.run(["gcc", "-std=c99", "-I", inc, str(src), "-o", str(tmp_path / "layout")], check=True)
    out = subprocess.run([str(tmp_path / "layout")], check=True, capture_output=True, text=True).stdout
    assert [int(v) for v in out.split()] == [getattr(_lib.Plan, f).offset for f, _ in _lib.Plan._fields_] + [
        ctypes.sizeof(_lib.Plan)]


@pytest.mark.parametrize("sides,path,updates,kernel", [([300, 240], 1, 2, "k_batch_fused"), ([700] * 2, 1, 4, "k_batch_fused"),
                                                       ([65, 97], 2, 0, "k_batch_resident")])
def test_batch_path_is_reported_and_can_be_chosen(fake, sides, path, updates, kernel):
    lib = fake.lib
    b = fake.batch(sides)

    def now():
        p, k = ctypes.c_int(), ctypes.c_int()
        assert lib.mdf_batch_get_path(b, ctypes.byref(p), ctypes.byref(k)) == _lib.OK
        kinds = _step_kernels(fake, b)
        assert all(("k_batch_chunk" if p.value == _lib.PATH_PERSISTENT else kernel) in n for n in kinds)
        return p.value, k.value

    default, persistent = (path, updates), (_lib.PATH_PERSISTENT, 0)
    assert now() == default
    for away in (lambda: lib.mdf_batch_set_schedule(b, 64, 0, 3), lambda: lib.mdf_batch_set_path(b, _lib.PATH_PERSISTENT)):
        assert away() == _lib.OK and now() == persistent
        assert lib.mdf_batch_set_path(b, _lib.PATH_DEFAULT) == _lib.OK and now() == default
    assert lib.mdf_batch_set_timeout(b, 1000) == _lib.OK and now() == persistent
    assert lib.mdf_batch_set_path(b, _lib.PATH_DEFAULT) == _lib.OK and now() == persistent  # the limit stays
    assert lib.mdf_batch_set_timeout(b, 4_000_000_000) == _lib.OK and now() == default
    for bad in (-2, 0, 1, 2, 4):
        assert lib.mdf_batch_set_path(b, bad) == _lib.EINVAL
    lib.mdf_batch_destroy(b)


@pytest.mark.parametrize("shape,storage,own", [((29, 124, 157), "f16", (4, 96)), ((190, 40, 20), "bf16eq", (2, 96)),
                                               ((700, 700), "f32", (4, 96)), ((64, 64), "f64", (2, 64))])
def test_autotune_weighs_the_shape_in_use(fake, shape, storage, own):
    """The launch shape of a handle is a candidate of its own, and stays where no
    other is faster (here all take no time)."""
    h = fake.lattice(shape, storage)
    info = _lib.Info()
    assert fake.lib.mdf_info(h, ctypes.byref(info)) == _lib.OK and (info.vx, info.block) == own
    fake.launches()
    v, b = ctypes.c_int(), ctypes.c_int()
    assert fake.lib.mdf_autotune(h, 2, ctypes.byref(v), ctypes.byref(b)) == _lib.OK
    assert own[1] in {threads for _, _, _, threads, _ in fake.launches()}
    assert (v.value, b.value) == own
    assert fake.lib.mdf_info(h, ctypes.byref(info)) == _lib.OK and (info.vx, info.block) == own
    fake.lib.mdf_destroy(h)
