"""The library's host code against a CUDA runtime that runs nothing (fake_cuda_runtime.cpp): which
kernels a call launches, with what attributes, on which device.  CPU only."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2503_17491_gb300 import _lib
from paper_2503_17491_gb300 import build as product_build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def library_file(tmp_path_factory):
    """The library's objects linked with the fake runtime in place of CUDA's."""
    product_build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(product_build.nvcc())))
    objs = [os.path.join(product_build.BUILD, u.replace(".cu", ".o")) for u in product_build.UNITS]
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                    "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cuda_runtime.cpp"), *objs, "-o", so], check=True)
    return so


class Host:
    """One fresh copy of the library (its statics included), with the calls the tests make."""

    def __init__(self, so):
        self.lib = ctypes.CDLL(so)
        for name, (args, res) in _lib.SIGNATURES.items():
            getattr(self.lib, name).argtypes = args
            getattr(self.lib, name).restype = res
        self.lib.fake_launch.restype = ctypes.c_char_p

    def create(self, n, views=1, rows=16, cols=64, **cap):
        cfg = _lib.splat_render_config()
        self.lib.splat_default_config(ctypes.byref(cfg))
        self.n, self.pixels = n, views * rows * cols
        c = _lib.splat_capacity(n, views, self.pixels, cap.get("max_pairs", 1 << 16), 0)
        self.ctx = ctypes.c_void_p()
        r = self.lib.splat_ctx_create(ctypes.byref(cfg), ctypes.byref(c), ctypes.byref(self.ctx))
        if r:
            return r
        T = np.ascontiguousarray(np.stack([np.eye(4)] * views))
        intr = (_lib.splat_lidar_intrinsics * views)(
            *[_lib.splat_lidar_intrinsics(rows, cols, -0.3, 0.3)] * views)
        assert self.lib.splat_set_views(self.ctx, views, T.ctypes.data, intr) == 0
        self.buf = np.zeros(16 * max(n, self.pixels) + 16, np.float32)   # stands for every buffer
        self.p = (self.buf.ctypes.data + 15) // 16 * 16
        self.g = _lib.splat_gaussians(self.p, self.p, self.p, n)
        return 0

    def render(self):
        return self.lib.splat_render_views(self.ctx, ctypes.byref(self.g), self.p, self.p, self.p,
                                           None)

    def backward(self):
        return self.lib.splat_render_views_backward(self.ctx, ctypes.byref(self.g), self.p, self.p,
                                                    self.p, self.p, self.p, self.p, 0, None)

    def launches(self):
        out = []
        for k in range(self.lib.fake_launches()):
            grid, block = (ctypes.c_uint * 3)(), ctypes.c_uint()
            shared, chained = ctypes.c_uint(), ctypes.c_int()
            name = self.lib.fake_launch(k, grid, ctypes.byref(block), ctypes.byref(shared),
                                        ctypes.byref(chained)).decode()
            out.append(dict(name=name, grid=tuple(grid), block=block.value, shared=shared.value,
                            chained=bool(chained.value)))
        return out


@pytest.fixture
def host(library_file, tmp_path):
    so = str(tmp_path / "lib.so")
    with open(library_file, "rb") as f, open(so, "wb") as g:
        g.write(f.read())
    return Host(so)


def test_shared_memory_limits_on_a_second_device(host):
    """Kernels above 48 KB have their limit raised on every device they are launched on, and a
    failure to raise it is not remembered."""
    host.lib.fake_fail_attributes(1)
    assert host.create(5000) != 0
    for device in (0, 1):
        host.lib.fake_set_device(device)
        assert host.create(5000) == 0, device
        assert host.render() == 0, device
        assert host.backward() == 0, device
    names = [x["name"] for x in host.launches() if x["shared"] > 48 << 10]
    assert len(names) == 6 and len(set(names)) == 3   # lists, forward, backward on either device


@pytest.mark.parametrize("n,views", [(1 << 18, 2), ((1 << 18) + 1, 2), (1 << 19, 1),
                                     ((1 << 19) + 1, 1)])
def test_chained_launches_follow_the_size(host, n, views):
    """A call of up to 2^19 pairs chains every kernel, a larger one none but the parameter
    gradients, which go by the primitives."""
    assert host.create(n, views) == 0
    host.lib.fake_clear()
    assert host.render() == 0 and host.backward() == 0
    last = [x["chained"] for x in host.launches() if "k_param_grads" in x["name"]]
    rest = {x["chained"] for x in host.launches() if "k_param_grads" not in x["name"]}
    assert last == [n <= 1 << 19] and rest == {n * views <= 1 << 19}


def test_stage_times_of_a_profiled_render_add_up(host):
    """Every stage of a profiled render has a time (the two that the binning no longer has take
    none), so that the values can be summed; what was not recorded gives -1."""
    assert host.create(100) == 0
    ms = (ctypes.c_float * 7)()
    assert host.lib.splat_stage_times(host.ctx, ms) == 0 and list(ms) == [-1.0] * 7
    assert host.lib.splat_set_profiling(host.ctx, 1) == 0 and host.render() == 0
    assert host.lib.splat_stage_times(host.ctx, ms) == 0
    assert list(ms) == [1.0, 0.0, 1.0, 1.0, 0.0, -1.0, -1.0]
