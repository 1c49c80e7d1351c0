"""The library's own objects linked with a CUDA runtime in host memory (``native/fake_cuda.cpp``): every entry point runs
its host code here, with no GPU. Allocations count against a limit and can be made to fail; launches are recorded and run
nothing."""
import ctypes
import os
import shutil
import subprocess

import paper_1709_03565_gb300 as skis
from paper_1709_03565_gb300 import _binding, _build

HERE = os.path.dirname(os.path.abspath(__file__))
NATIVE = os.path.join(HERE, "native")
OUT = os.path.join(NATIVE, "_build")
_fk = None


def build() -> str:
    skis.build()
    os.makedirs(OUT, exist_ok=True)
    nvcc = _build._nvcc()
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    objs = sorted(os.path.join(_build.OBJ, f) for f in os.listdir(_build.OBJ) if f.endswith(".o"))
    deps = [os.path.join(_build.CSRC, "skis_internal.cuh"), os.path.join(_build.INCLUDE, "skis.h")]
    mine = []
    for name, cmd in (("fake_cuda.cpp", [shutil.which("g++") or "g++", "-std=c++17", "-O1", "-fPIC", "-I", cuda]),
                      ("sketch_fields.cu", [nvcc, *_build.ARCH, *_build.FLAGS])):
        src, obj = os.path.join(NATIVE, name), os.path.join(OUT, name.split(".")[0] + ".o")
        if _build._stale(obj, [src] + deps):
            subprocess.run([*cmd, "-c", src, "-o", obj], check=True)
        mine.append(obj)
    lib = os.path.join(OUT, "libskis_fake.so")
    if _build._stale(lib, objs + mine):
        tmp = lib + f".{os.getpid()}.tmp"
        subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", tmp, *objs, *mine], check=True)
        os.replace(tmp, lib)
    return lib


def lib():
    global _fk
    if _fk is None:
        h = ctypes.CDLL(build())
        for name, res, args in _binding._SIGNATURES:
            f = getattr(h, name)
            f.restype, f.argtypes = res, args
        P, U64, S = ctypes.c_void_p, ctypes.c_uint64, ctypes.c_char_p
        for name, res, args in (("fk_start", None, [U64]), ("fk_fail_at", None, [ctypes.c_int64, ctypes.c_int]),
                                ("fk_allocs", U64, []), ("fk_used", U64, []),
                                ("fk_script", None, [P, P, ctypes.c_int]), ("fk_set_W", None, [P, U64]),
                                ("fk_value", U64, [P, S]), ("fk_bytes", U64, [P, S]), ("fk_cursor", U64, [P]),
                                ("fk_first_bad", U64, [P]), ("fk_events", ctypes.c_int, [P]),
                                ("fk_launch", ctypes.c_int, [U64, P, U64, P, P])):
            f = getattr(h, name)
            f.restype, f.argtypes = res, args
        _fk = h
    return _fk


class Sketch:
    """A sketch of an edgeless graph of n vertices (no kernel runs, so its samples are empty)."""

    def __init__(self, n, lt=False, limit=280 << 30, arena=0):
        self.fk = fk = lib()
        self.before = fk.fk_used()  # held by sketches of tests that failed
        fk.fk_start(self.before + limit)
        self.g, self.s = ctypes.c_void_p(), ctypes.c_void_p()
        load = fk.skis_load_graph_lt if lt else fk.skis_load_graph
        assert load(ctypes.byref(self.g), n, 0, None, None, None, skis.SKIS_W_WC, 0, skis.SKIS_MEM_HOST, None) == 0
        fk.fk_set_W(self.g, 1)
        assert fk.skis_sketch_create(ctypes.byref(self.s), self.g, 1, arena, None) == 0

    def option(self, opt, value):
        assert self.fk.skis_sketch_set_option(self.s, opt, value) == 0

    def sample(self, count):
        return self.fk.skis_sample(self.s, count, None, None)

    def script(self, *passes):
        flat = [x for p in passes for x in p]
        self.fk.fk_script(self.s, (ctypes.c_uint64 * len(flat))(*flat), len(passes))

    def value(self, field):
        return self.fk.fk_value(self.s, field.encode())

    def bytes(self, field):
        return self.fk.fk_bytes(self.s, field.encode())

    def launches(self):
        out, name = [], ctypes.create_string_buffer(512)
        grid, block = ctypes.c_uint(), ctypes.c_uint()
        while self.fk.fk_launch(len(out), name, 512, ctypes.byref(grid), ctypes.byref(block)):
            out.append((name.value.decode(), grid.value, block.value))
        return out

    def close(self):
        if self.s:
            self.fk.skis_sketch_free(self.s)
        self.fk.skis_graph_free(self.g)
        assert self.fk.fk_used() == self.before
