"""The library's host code on a stand-in CUDA runtime (fake_cudart.cpp): which kernels a call launches and
what it allocates, without a device.  ``fake_lib()`` links the library's own objects against it."""
import ctypes as C
import os
import re
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


def fake_lib(tmp):
    from paper_1008_0135_gb300 import _abi, build_ext
    build_ext.build()
    objs = [os.path.join(build_ext.BUILD, s + ".o") for s in build_ext.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build_ext.build(force=True)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    so = os.path.join(str(tmp), "libvr_fake.so")
    r = subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-Wl,-Bsymbolic", f"-I{cuda}/include",
                        os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", so, "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(so)
    for name, (res, args) in _abi.SIGNATURES.items():
        fn = getattr(L, name)
        fn.restype, fn.argtypes = res, args
    L.fake_launches.restype = C.c_char_p
    L.fake_reserved.restype = C.c_size_t
    L.fake_limit.argtypes = [C.c_size_t]
    L.fake_device_alloc.restype, L.fake_device_alloc.argtypes = C.c_void_p, [C.c_size_t]
    return L


def launches(L):
    """[(kernel, template arguments)] launched (and copies made) since the last call."""
    out = []
    names = subprocess.run(["c++filt"], input=L.fake_launches().decode(), capture_output=True, text=True, check=True).stdout
    for name in names.splitlines():
        k = re.search(r"\b(k_\w+)(?:<([^(]*)>)?\(", name.replace("(anonymous namespace)::", ""))
        args = (k.group(2) or "").replace("true", "1").replace("false", "0").split(", ") if k else []
        out.append((k.group(1) if k else name, tuple(int(x) for x in args if x.isdigit())))
    return out


class Host:
    """A context of the library on the stand-in runtime, by the C calls."""

    def __init__(self, L, cache=0):
        self.L, self.h = L, C.c_void_p()
        L.fake_reset()
        assert L.vr_create(C.byref(self.h), 0, cache) == 0
        lut = np.linspace(0, 1, 8, dtype=np.float32).reshape(2, 4).copy()
        self.ok(L.vr_set_transfer_function(self.h, lut.ctypes.data, 2, 0.0, 1.0))
        self.ok(L.vr_set_full_rect(self.h, 1))        # (no kernel fills the bricks' value ranges)

    def ok(self, rc):
        assert rc == 0, (rc, self.L.vr_last_error_message())

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.L.vr_destroy(self.h)

    def load(self, n):
        """A resident cube of nx, ny, nz voxels."""
        cube, cid = np.zeros(n[::-1], np.float32), C.c_int()
        self.ok(self.L.vr_load_cube(self.h, cube.ctypes.data, 0, *n, 0, None, None, C.byref(cid)))
        return cid.value

    def brick(self, cid, brick, layouts=9, storage=0):
        self.ok(self.L.vr_set_brick_layouts(self.h, cid, layouts))
        return self.L.vr_set_bricking(self.h, cid, *brick, 1, storage)

    def camera(self, view, proj=0, param=64.0, W=32, H=24, mode=0, step=0.7):
        v = np.ascontiguousarray(view, np.float32)
        self.ok(self.L.vr_set_camera(self.h, v.ctypes.data, proj, param, W, H))
        self.ok(self.L.vr_set_render_params(self.h, mode, step, 0.99))
        self.out = np.zeros((H, W, 4), np.float32)

    def frame(self, cid):
        return self.L.vr_render_frame(self.h, cid, self.out.ctypes.data, 0, None)
