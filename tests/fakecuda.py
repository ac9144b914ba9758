"""The library linked against a CUDA runtime that needs no GPU (fake_cudart.c):
what the host code allocates, asks of its kernels and launches, and where."""
from __future__ import annotations

import ctypes as C
import glob
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
PATCHED_STATUS = 144  # bytes of the status block a call reads back


class Fake:
    def __init__(self):
        from paper_1910_02611_gb300 import build
        from paper_1910_02611_gb300.rambo import SIGNATURES

        lib = build.build()
        objs = [os.path.join(build.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
        if not all(os.path.exists(o) for o in objs):
            build.build(force=True)
        os.makedirs(os.path.join(HERE, "_build"), exist_ok=True)
        out = os.path.join(HERE, "_build", "librambo_fake.so")
        src = os.path.join(HERE, "fake_cudart.c")
        if not os.path.exists(out) or os.path.getmtime(out) < max(map(os.path.getmtime, [lib, src, *objs])):
            subprocess.check_call(["gcc", "-O1", "-fPIC", "-w", "-c", src, "-o", out + ".o"])
            subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic,-z,defs", "-o", out, *objs, out + ".o"])
        self.lib = C.CDLL(out)
        for name, (res, args) in SIGNATURES.items():
            f = getattr(self.lib, name)
            f.restype, f.argtypes = res, args
        self.lib.fake_used.restype = C.c_size_t
        self.lib.fake_event.restype = C.c_char_p
        for dev in (0, 1):
            self.budget(dev, 64 << 30)

    def budget(self, dev: int, n: int):
        self.lib.fake_budget(dev, C.c_size_t(n))

    def used(self, dev: int = 0) -> int:
        return self.lib.fake_used(dev)

    def device(self, dev: int):
        self.lib.cudaSetDevice(dev)

    def status(self, offset: int | None = None, value: int = 0):
        """The status blocks that calls read back hold `value` at `offset` (None: as the host left them)."""
        self.lib.fake_patch(C.c_uint64(0 if offset is None else PATCHED_STATUS), C.c_uint64(offset or 0), C.c_uint64(value))

    def clear(self):
        self.lib.fake_clear()

    def events(self, kinds: str = "LFM") -> list[dict]:
        """Launches (L), other uses of a kernel (F) and device allocations (M) since clear()."""
        out = []
        kind, dev, grid, smem, size = C.c_char(), C.c_int(), C.c_uint(), C.c_size_t(), C.c_size_t()
        for i in range(self.lib.fake_events()):
            name = self.lib.fake_event(i, C.byref(kind), C.byref(dev), C.byref(grid), C.byref(smem), C.byref(size)).decode()
            if kind.value.decode() in kinds:
                out.append(dict(kind=kind.value.decode(), name=name, device=dev.value, grid=grid.value, smem=smem.value,
                                bytes=size.value))
        return out

    def create(self, K, B, R, m, eta=2, seed=1):
        h = C.c_void_p()
        assert self.lib.rambo_create(K, B, R, m, eta, seed, C.byref(h)) == 0
        return h

    def config(self, h):
        from paper_1910_02611_gb300.rambo import QueryConfig

        cfg = QueryConfig()
        assert self.lib.rambo_get_query_config(h, cfg) == 0
        return cfg

    def query(self, h, data: np.ndarray, offsets: np.ndarray, on_device: bool, k: int = 31) -> int:
        """The arena call, for keys or (bytes) sequences; `device` memory is host memory here."""
        ids, off = C.c_void_p(), C.c_void_p()
        n, tail = offsets.size - 1, (int(on_device), C.byref(ids), C.byref(off), None)
        if data.dtype == np.uint8:
            return self.lib.rambo_query_seq_batch(h, data.ctypes.data, offsets.ctypes.data, n, k, *tail)
        return self.lib.rambo_query_batch(h, data.ctypes.data, offsets.ctypes.data, n, *tail)

    def plan(self, h, kind: int, max_queries: int, max_items: int, max_ids: int, k: int = 31):
        """(return code, plan)"""
        p = C.c_void_p()
        return self.lib.rambo_plan_create(h, kind, max_queries, max_items, max_ids, k, C.byref(p)), p

    def noalloc(self, h, data: np.ndarray, offsets: np.ndarray, k: int = 31) -> int:
        n = offsets.size - 1
        ids, off, need = np.zeros(1 << 10, np.uint32), np.zeros(n + 1, np.uint64), C.c_uint64()
        self.status(0, 2**64 - 1)  # no error: the kernel that clears the status block does not run
        try:
            return self.lib.rambo_query_seq_batch_noalloc(h, data.ctypes.data, offsets.ctypes.data, n, k, ids.ctypes.data,
                                                          ids.size, off.ctypes.data, C.byref(need), None)
        finally:
            self.status()
