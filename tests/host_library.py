"""The library's host side over a stand-in CUDA runtime (fake_runtime.cpp, fake_launchers.cu): the
same C ABI, every step launch logged with its stream, no GPU."""
import concurrent.futures as cf
import ctypes
import os
import re
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1411_3133_gb300", "csrc")


def build_host_library(out_dir):
    """Compile and link it under out_dir; the bound ctypes library."""
    from paper_1411_3133_gb300 import build, lbgm as L
    srcs = [os.path.join(CSRC, f) for f in ("api.cu", "batch.cu", "geometry.cpp")] + [
        os.path.join(HERE, f) for f in ("fake_launchers.cu", "fake_runtime.cpp")]

    def compile_one(src):
        obj = os.path.join(out_dir, os.path.basename(src) + ".o")
        cmd = [build._nvcc()] + build.ARCH + ["-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return obj

    with cf.ThreadPoolExecutor(len(srcs)) as ex:
        objs = list(ex.map(compile_one, srcs))
    path = os.path.join(out_dir, "libhost.so")
    # -Bsymbolic: a real CUDA runtime in the process must not take the calls
    r = subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", path] + objs, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(path)
    for name, (res, args) in L.SIGNATURES.items():
        if hasattr(lib, name):
            getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    lib.fake_take_log.restype = ctypes.c_char_p
    lib.fake_stream.restype = ctypes.c_void_p
    lib.fake_capture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.fake_set_costs.argtypes = [ctypes.c_double] * 5
    return lib


class Host:
    """One context of the host library."""

    def __init__(self, lib, metric, size, batch, precision, periodic3=True, priority=0, stream=None, old_forcing=0):
        from paper_1411_3133_gb300 import lbgm as L
        self.lib, self.L = lib, L
        desc = L.make_desc(1.0, 1.0 / 0.975, *size, periodic3=periodic3)
        self.stream = stream or lib.fake_stream(priority)
        self.ctx = ctypes.c_void_p()
        self.batch, self.dtype = batch, {"fp64": np.uint64, "fp32": np.uint32}.get(precision, np.uint16)
        self.ok(lib.lb_create_geometry(L.METRICS[metric], ctypes.byref(desc), batch, L.PRECISIONS[precision],
                                       ctypes.c_void_p(self.stream), None, ctypes.byref(self.ctx)))
        self.init(old_forcing)

    def init(self, old_forcing=0):
        p = (self.L.lb_params * self.batch)(*[self.L.make_params(0.6, 1e-5, old_forcing, 1, 0.0, False)] * self.batch)
        self.ok(self.lib.lb_init(self.ctx, p))

    def ok(self, status):
        assert status == self.L.LB_OK, (status, self.lib.lb_last_error(self.ctx))

    def option(self, opt, value):
        self.ok(self.lib.lb_set_option(self.ctx, opt, value))

    def step(self, n):
        self.ok(self.lib.lb_step(self.ctx, n))

    def counts(self):
        """Steps every instance has taken."""
        n = self.lib.lb_state_bytes(self.ctx)
        buf = np.zeros(n // np.dtype(self.dtype).itemsize, self.dtype)
        self.ok(self.lib.lb_get_state(self.ctx, buf.ctypes.data_as(ctypes.c_void_p), n, 0))
        return buf.reshape(self.batch, -1)[:, 0]

    def close(self):
        self.lib.lb_destroy(self.ctx)


def take_log(lib):
    """Logged calls since the last one: dicts (kind, and the line's fields)."""
    out = []
    for line in lib.fake_take_log().decode().splitlines():
        kind, *rest = line.split()
        out.append(dict({k: int(v, 16 if k == "first" else 10) for k, v in (x.split("=") for x in rest)}, kind=kind))
    return out


def launches(lib):
    return [x for x in take_log(lib) if re.match(r"f|h|b|list|tma|shift", x["kind"])]
