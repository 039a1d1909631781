"""Loads the library's host code linked against fake_cudart.cpp in the place of
the CUDA runtime, so that plans, dispatch and error paths are tested without a
GPU."""
import ctypes
import glob
import os
import subprocess

from paper_2108_08591_gb300 import _build, _lib

HERE = os.path.dirname(os.path.abspath(__file__))


def link(out):
    """Link the built objects with the stand-in into `out`."""
    _build.build()
    objs = sorted(glob.glob(os.path.join(_build.BUILD, "mdf_*.o")))
    if len(objs) != len(_build._sources()):
        _build.build(force=True)
        objs = sorted(glob.glob(os.path.join(_build.BUILD, "mdf_*.o")))
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build._nvcc()))), "include")
    # every other symbol is local: the process may hold the real library as well,
    # whose templates' statics (kernel handles) the dynamic linker would share
    script = str(out) + ".map"
    with open(script, "w") as fh:
        fh.write("{ global: mdf_*; fake_*; local: *; };\n")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", f"-Wl,--version-script={script}", "-I", inc,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", str(out)], check=True)


class Fake:
    """The library on the stand-in.  What the library keeps per device stays for
    the life of the process, so every test starts on a device of its own."""

    def __init__(self, linked):
        self.device = -1
        self.lib = ctypes.CDLL(str(linked))
        for name, (res, args) in _lib.SIGNATURES.items():
            fn = getattr(self.lib, name)
            fn.restype, fn.argtypes = res, args
        self.lib.fake_launch.restype = ctypes.c_char_p
        self.lib.fake_watched.restype = ctypes.c_void_p
        self.lib.fake_cost.argtypes = [ctypes.c_char_p, ctypes.c_double, ctypes.c_double, ctypes.c_int]

    def new_device(self):
        """Make a device that nothing has been launched on the current one."""
        self.device += 1
        self.lib.fake_set_device(self.device)
        return self.device

    def launches(self):
        """Recorded launches as (kernel, device, blocks, threads, cluster)."""
        out = []
        for k in range(self.lib.fake_launches()):
            v = [ctypes.c_uint() for _ in range(4)]
            name = self.lib.fake_launch(k, *(ctypes.byref(x) for x in v)).decode()
            out.append((name, *(x.value for x in v)))
        self.lib.fake_clear()
        return out

    def watched(self, ctype):
        return ctype.from_buffer_copy(ctypes.string_at(self.lib.fake_watched(), ctypes.sizeof(ctype)))

    def lattice(self, shape, storage="f32", **opts):
        h = ctypes.c_void_p()
        g = _lib.Grid(*shape, *([1] if len(shape) == 2 else []))
        r = _lib.Rates(1.0, 1.7, -1.0)
        o = _lib.Opts(_lib.STORAGE[storage], 1, None, *(opts.get(k, 0) for k in ("vx", "block", "q", "inplace")))
        bc = _lib.BC()
        bc.wall[:] = [int(opts.get("wall", False) and k < len(shape)) for k in range(3)]
        st = self.lib.mdf_create(ctypes.byref(h), ctypes.byref(g), len(shape), ctypes.byref(r), ctypes.byref(bc),
                                 ctypes.byref(o))
        assert st == _lib.OK, self.lib.mdf_last_error(None)
        return h

    def batch(self, sides):
        h = ctypes.c_void_p()
        side = (ctypes.c_int * len(sides))(*sides)
        Re = (ctypes.c_double * len(sides))(*[100.0] * len(sides))
        st = self.lib.mdf_batch_create(ctypes.byref(h), 2, len(sides), side, Re, 0.1, None)
        assert st == _lib.OK, self.lib.mdf_batch_last_error(None)
        return h
