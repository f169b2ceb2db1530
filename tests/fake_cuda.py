"""The library's host code on a CPU: its object files linked with a stand-in for the CUDA runtime (fake_cuda.c) that writes down
what is queued on which stream, runs nothing, and makes any chosen call fail."""
import ctypes
import os
import subprocess

import torch

from paper_2608_03676_b200.binding import TaotParams, _Outputs
from paper_2608_03676_b200.build import OBJ, SOURCES, build

LAUNCH, RECORD, WAIT, COPY, SET, STREAM_CREATE, EVENT_CREATE, DEVICE_ALLOC = range(1, 9)
CALLER = 0x77                                    # the stream that the caller passes
DEVICE = 1 << 40                                 # where "device memory" begins: nothing follows these addresses


class Entry(ctypes.Structure):
    _fields_ = [("kind", ctypes.c_int), ("stream", ctypes.c_long), ("obj", ctypes.c_long), ("grid", ctypes.c_long),
                ("name", ctypes.c_char * 96), ("arg", ctypes.c_ubyte * 256)]


def load(folder):
    build()
    here = os.path.dirname(os.path.abspath(__file__))
    obj, lib = os.path.join(folder, "fake_cuda.o"), os.path.join(folder, "libtaot_fake.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["gcc", "-O1", "-fPIC", "-I", os.path.join(cuda, "include"), "-c", os.path.join(here, "fake_cuda.c"), "-o", obj], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib, obj] + [os.path.join(OBJ, src.replace(".cu", ".o")) for src in SOURCES], check=True)
    so = ctypes.CDLL(lib)
    so.fake_entry.restype = ctypes.POINTER(Entry)
    so.fake_capturing.argtypes = [ctypes.c_int]
    return so


class SinkArgs(ctypes.Structure):
    """The argument of the Phase-1 kernels (sinkhorn_common.cuh)."""
    _fields_ = [("pointers", ctypes.c_void_p * 8), ("R", ctypes.c_int32), ("kcap", ctypes.c_int32), ("inv_eps", ctypes.c_double),
                ("eps0", ctypes.c_float), ("max_iters", ctypes.c_int32), ("tol", ctypes.c_float), ("check_every", ctypes.c_int32),
                ("early", ctypes.c_int32), ("only_marked", ctypes.c_int32), ("skip_solved", ctypes.c_int32)]


class FakePlanner:
    """A handle of the library over the fake runtime, with made-up device addresses."""

    def __init__(self, so, L, R, E, K, k, T, C, e2r=None, eps=1.0, max_iters=100, tol=0.0, ablation=0):
        self.so, self.L, self.R, self.T, self.k = so, L, R, T, k
        p = TaotParams(ctypes.sizeof(TaotParams), L, R, E, K, k, T, eps, max_iters, tol, 1, 1e-8, 0.1, 0, ablation)
        e2r = (torch.arange(E) * R // E).int() if e2r is None else e2r.int().contiguous()
        C = C.float().contiguous()
        self.handle = ctypes.c_void_p()
        rc = so.taot_create(ctypes.byref(self.handle), ctypes.byref(p), ctypes.c_void_p(e2r.data_ptr()), ctypes.c_void_p(C.data_ptr()), None)
        assert rc == 0
        self.stream = ctypes.c_void_p(CALLER)

    def plan(self, topk=DEVICE):
        o = _Outputs(*[DEVICE + (i + 1) * (1 << 34) for i in range(14)])
        return self.so.taot_plan(self.handle, ctypes.c_void_p(topk), ctypes.byref(o), ctypes.c_void_p(DEVICE + (1 << 39)), self.stream)

    def plan_host_block(self):
        at = lambda i: ctypes.c_void_p(i << 36)
        return self.so.taot_plan_host_block(self.handle, at(1), at(2), at(3), ctypes.c_void_p(DEVICE), self.stream)

    def host_block_layout(self):
        off, n = (ctypes.c_size_t * 14)(), ctypes.c_size_t()
        return self.so.taot_host_block_layout(self.handle, off, ctypes.byref(n))

    def sinkhorn(self, B):
        at = lambda i: ctypes.c_void_p(DEVICE + (i << 34))
        return self.so.taot_sinkhorn(self.handle, at(1), at(2), ctypes.c_int32(B), at(3), at(4), at(5), at(6), at(7), self.stream)

    def close(self):
        self.so.taot_destroy(self.handle)


def log(so):
    return [so.fake_entry(i).contents for i in range(so.fake_count())]


def kernels(so):
    return [e.name.decode() for e in log(so) if e.kind == LAUNCH]


def not_joined(entries):
    """Operations (launches, copies, sets) on any stream that the end of the caller's stream does not wait for."""
    seen = {CALLER: set()}                       # per stream, the operations that its end comes after
    events = {}
    work = []
    for i, e in enumerate(entries):
        mine = seen.setdefault(e.stream, set())
        if e.kind in (LAUNCH, COPY, SET):
            mine.add(i)
            work.append(i)
        elif e.kind == RECORD:
            events[e.obj] = set(mine)
        elif e.kind == WAIT:
            mine |= events.get(e.obj, set())
    return [i for i in work if i not in seen[CALLER]]
