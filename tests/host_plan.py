"""The library's host side (bookkeeping, planner, launches) compiled with g++ against recording_runtime.cpp: what a
sequence of calls launches, with which descriptors, without a GPU."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np

from paper_2608_10402_b200 import tide

DECODE, TILE, UMMA, MERGE, APPEND, MOVE, TABLE, UPLOAD, COPY_PAGES, READ, FETCH = range(11)
INT_MAX = 2 ** 31 - 1
_TESTS = os.path.dirname(os.path.abspath(__file__))


def build(folder):
    """The shared object, built in `folder`."""
    so = os.path.join(str(folder), "libhostplan.so")
    host = os.path.join(os.path.dirname(_TESTS), "paper_2608_10402_b200", "csrc", "tide_host.cu")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I/usr/local/cuda/include", "-x", "c++", host,
                           os.path.join(_TESTS, "recording_runtime.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    lib.launch_at.restype = ctypes.c_void_p
    return lib


class Handle:
    """One tide_kv_t of the recorded library.  Streams are plain numbers; calls return the status code."""

    def __init__(self, lib, Hq=28, Hkv=4, D=128, S=16, num_pages=4096, max_tasks=16, max_pages=2048, max_rows=16, max_tokens=8192, layers=1):
        self.lib = lib
        cfg = tide.make_config(Hq, Hkv, D, S, num_pages, max_tasks, max_pages, max_rows, max_tokens, layers)
        pb, wb = ctypes.c_size_t(0), ctypes.c_size_t(0)
        assert lib.tide_kv_required_bytes(ctypes.byref(cfg), ctypes.byref(pb), ctypes.byref(wb)) == 0
        self._ws = np.zeros(wb.value + 256, np.uint8)
        cfg.pool, cfg.pool_bytes = 1 << 40, pb.value                       # never touched: kernels do not run
        cfg.workspace, cfg.workspace_bytes = (self._ws.ctypes.data + 255) // 256 * 256, wb.value
        self.h = ctypes.c_void_p(0)
        assert lib.tide_kv_create(ctypes.byref(cfg), ctypes.byref(self.h)) == 0
        self.cfg, self.mp = cfg, max_pages

    def close(self):
        self.lib.tide_kv_destroy(self.h)

    def _list(self, counts):
        ids = np.array(list(counts), np.int32)
        ip = np.concatenate([[0], np.cumsum(list(counts.values()))]).astype(np.int32)
        return ids, ip

    def alloc(self, *tasks):
        for t in tasks:
            assert self.lib.tide_kv_alloc(self.h, t, ctypes.c_int64(0)) == 0

    def append(self, counts, stream=0):
        """counts: {task: new tokens}"""
        ids, ip = self._list(counts)
        return self.lib.tide_kv_append(self.h, 0, len(ids), ids.ctypes.data_as(ctypes.c_void_p), ip.ctypes.data_as(ctypes.c_void_p),
                                       ctypes.c_void_p(4096), ctypes.c_void_p(4096), ctypes.c_void_p(stream))

    def extend(self, counts, stream=0):
        ids, ip = self._list(counts)
        return self.lib.tide_kv_extend(self.h, len(ids), ids.ctypes.data_as(ctypes.c_void_p), ip.ctypes.data_as(ctypes.c_void_p),
                                       ctypes.c_void_p(stream))

    def write(self, layer, counts, stream=0):
        ids, ip = self._list(counts)
        return self.lib.tide_kv_write(self.h, layer, len(ids), ids.ctypes.data_as(ctypes.c_void_p), ip.ctypes.data_as(ctypes.c_void_p),
                                      ctypes.c_void_p(4096), ctypes.c_void_p(4096), ctypes.c_void_p(stream))

    def fork(self, parent, child, stream=0):
        return self.lib.tide_kv_fork(self.h, 0, parent, child, ctypes.c_void_p(stream))

    def prune(self, task, keep, tail, stream=0):
        return self.lib.tide_kv_prune(self.h, 0, task, keep, tail, ctypes.c_void_p(stream))

    def truncate(self, task, n):
        return self.lib.tide_kv_truncate(self.h, task, n)

    def attend(self, rows, stream=0, scale=0.125):
        p = ctypes.c_void_p(4096)
        return self.lib.tide_attend(self.h, 0, len(rows), tide.rows_array(rows), None, p, ctypes.c_float(scale), p, None, ctypes.c_void_p(stream))

    def step_begin(self, rows, stream=0):
        return self.lib.tide_step_begin(self.h, len(rows), tide.rows_array(rows), ctypes.c_void_p(stream))

    def step_layer(self, layer, stream=0, new_k=1 << 30, new_v=2 << 30, q=3 << 30, out=4 << 30, lse=None):
        p = ctypes.c_void_p
        return self.lib.tide_step_layer(self.h, layer, p(new_k), p(new_v), p(q), ctypes.c_float(0.125), p(out), p(lse), p(stream))

    def step_host(self, rows):
        """A host-buffer step on stream 0 with (empty) host buffers."""
        kv_row, q_row = 2 * self.cfg.num_kv_heads * self.cfg.head_dim, 2 * self.cfg.num_q_heads * self.cfg.head_dim
        tokens = sum(n for _, n, _ in rows)
        k, q, o = (np.zeros(tokens * b, np.uint8) for b in (kv_row, q_row, q_row))
        a = lambda x: x.ctypes.data_as(ctypes.c_void_p)
        return self.lib.tide_step_host(self.h, 0, len(rows), tide.rows_array(rows), a(k), a(k), a(q), ctypes.c_float(0.125), a(o), None, None)

    def fix_grids(self, *caps):
        return self.lib.tide_step_fix_grids(self.h, *caps)

    def tune(self, knob, value):
        assert self.lib.tide_tune(self.h, knob, ctypes.c_int64(value)) == 0

    def plan(self):
        v = [ctypes.c_int64(0) for _ in range(4)]
        assert self.lib.tide_last_plan(self.h, *[ctypes.byref(x) for x in v]) == 0
        return dict(zip(("decode_items", "prefill_items", "merge_rows", "kernel_launches"), (x.value for x in v)))

    def forget(self):
        self.lib.forget()

    def launches(self):
        """What was launched since forget(): dicts, attention kernels with their segments' task and first live key."""
        out = []
        for i in range(self.lib.recorded()):
            v, s = (ctypes.c_int * 7)(), (ctypes.c_int * 20)()
            stream = self.lib.launch_at(i, v)
            segs = []
            for j in range(v[5]):
                self.lib.segment_at(i, j, s)
                segs.append({"task": s[0] // self.mp, "n": s[2], "p": s[3], "n_splits": s[6], "chunk": s[7], "live_from": s[9], "causal": s[10],
                             "origin": s[11], "partial": s[12]})
            out.append({"kind": v[0], "run_ahead": v[1], "overlapped": v[2], "items": v[3], "early": v[4], "writes": v[6], "stream": stream or 0, "segs": segs})
        return out

    def live(self, rows, stream=0):
        """First live key per task of the attention of `rows` (the producers run ahead below it)."""
        self.forget()
        assert self.attend(rows, stream) == 0
        found = {}
        for l in self.launches():
            if l["kind"] in (DECODE, UMMA):
                for s in l["segs"]:
                    f = s["live_from"] if l["run_ahead"] else 0
                    found[s["task"]] = min(found.get(s["task"], INT_MAX), f)
        return found
