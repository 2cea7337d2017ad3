"""The library linked against tests/fake_cudart.cpp: what it launches, waits for and
synchronises, as a list of log entries (no GPU)."""
import collections
import ctypes as C
import os
import subprocess

from paper_2603_24027_gb300 import _capi as A
from paper_2603_24027_gb300 import build as B
from paper_2603_24027_gb300 import fdtd as F

HERE = os.path.dirname(os.path.abspath(__file__))
# what: launch, graph, wait, record, sync, h2d, d2h, symbol; a: the stream; b: the event
# (wait, record), the bytes (copies) or whether a capture is on (launch)
Entry = collections.namedtuple("Entry", "what name a b grid")


def load(tmp):
    B.build()
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    out = os.path.join(str(tmp), "libfdtd_fake.so")
    home = os.path.dirname(os.path.dirname(B.nvcc()))
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-O1", "-Wl,-Bsymbolic", "-o", out,
                    "-I" + os.path.join(home, "include"), os.path.join(HERE, "fake_cudart.cpp")]
                   + objs, check=True)
    L = C.CDLL(out)
    for name, (res, args) in A._PROTOS.items():
        getattr(L, name).restype, getattr(L, name).argtypes = res, args
    L.fake_log.restype = C.c_char_p
    return L


def entries(L):
    out = []
    for ln in L.fake_log().decode().splitlines():
        p = ln.split()
        out.append(Entry(p[0], p[1], int(p[2]), int(p[3]), tuple(int(x) for x in p[4:7])))
    L.fake_clear()
    return out


class Runner:
    """Simulations with an invented workspace on the logged library."""

    def __init__(self, L, monkeypatch):
        self.L = L
        monkeypatch.setattr(A, "_lib", L)
        self.next = 0x100000000000

    def sim(self, w, rec, options=None):
        sim = F.Simulation(w)
        for k, v in (options or {}).items():
            sim.set_option(k, v)
        n = sim.workspace_bytes(rec)
        A.check(self.L.fdtd_bind_workspace(sim.h, self.next, n), sim.h)
        self.next += (n + (1 << 20)) & ~0xff
        return sim

    def forward(self, sim, rec):
        v = C.c_double()
        A.check(self.L.fdtd_forward(sim.h, 0x1000, C.byref(rec), C.byref(v)), sim.h)
        return entries(self.L)

    def backward(self, sim):
        A.check(self.L.fdtd_backward(sim.h, 1.0, 0x1000), sim.h)
        return entries(self.L)

    def group_forward(self, sims, rec):
        n = len(sims)
        hs = (C.c_void_p * n)(*[s.h for s in sims])
        eps = (C.c_void_p * n)(*([0x1000] * n))
        v = (C.c_double * n)()
        A.check(self.L.fdtd_group_forward(hs, n, eps, C.byref(rec), v))
        return entries(self.L)
