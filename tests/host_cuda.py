"""The library's host code on the runtime of host_cuda.c: the objects of the build linked
against it, and the words that the host waits for written by `publish` in the kernels' place.
For faults of the host code that need a failing allocation or launch, or two devices."""
import ctypes
import glob
import os
import subprocess

import pytest

from paper_0905_2200_gb300 import build as fembuild

HERE = os.path.dirname(os.path.abspath(__file__))
# words of a published plan (fem_internal.cuh)
PLAN_EDGES, PLAN_SLABS, PLAN_PARTS_MIN, PLAN_WORDS = 10, 11, 12, 15
ON_LAUNCH = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.POINTER(ctypes.c_void_p))


class Publish(ctypes.Structure):
    _fields_ = [("host", ctypes.POINTER(ctypes.c_uint32)), ("err", ctypes.POINTER(ctypes.c_uint32)),
                ("seq", ctypes.c_uint32)]


def link(tmp):
    fembuild.build()
    names = [os.path.basename(s)[:-3] + ".o" for s in glob.glob(os.path.join(fembuild.CSRC, "*.cu"))]
    objs = [os.path.join(fembuild.OUT_DIR, n) for n in names]
    if not all(os.path.exists(o) for o in objs):
        pytest.skip("the build's objects are not kept here")
    # (one library that binds to itself: a process may hold the real runtime's names)
    rt, lib = os.path.join(tmp, "host_cuda.o"), os.path.join(tmp, "libfem_host.so")
    subprocess.check_call(["gcc", "-c", "-fPIC", "-O1", "-o", rt, os.path.join(HERE, "host_cuda.c")])
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,--wrap=_Znwm", "-o", lib] + objs + [rt])
    return lib


class Host:
    """The loaded library; `launches` are the names of the kernels launched so far."""

    def __init__(self, tmp):
        self.lib = self.rt = ctypes.CDLL(link(tmp))
        self.launches = []
        self.plan = {}     # words of the next plans
        self.error = 0     # error word that the next counts publish
        self.publish_seq = True  # else plans and validations publish it everywhere but in its place
        self.on_launch = ON_LAUNCH(self._launched)
        ctypes.c_void_p.in_dll(self.rt, "host_on_launch").value = ctypes.cast(self.on_launch,
                                                                              ctypes.c_void_p).value

    def number(self, name, kind=ctypes.c_int):
        return kind.in_dll(self.rt, name)

    def _launched(self, name, args):
        name = name.decode()
        self.launches.append(name)

        def arg(k, kind):
            return ctypes.cast(args[k], ctypes.POINTER(kind))[0]

        if "k_publish_load" in name:
            t_last, k, host = (arg(i, kind) for i, kind in
                               ((1, ctypes.POINTER(ctypes.c_uint32)), (3, ctypes.c_uint32),
                                (4, ctypes.POINTER(ctypes.c_uint32))))
            first = arg(7, ctypes.POINTER(ctypes.c_uint32))
            host[0], host[1], host[258] = 0, t_last[0] if t_last else 0, first[0] if t_last else 0
            for a in range(k):
                host[2 + a] = 0
            host[arg(5, ctypes.c_uint32)] = arg(6, ctypes.c_uint32)
        elif "k_plan_scan" in name:
            p = arg(3, Publish)
            self._words(p, PLAN_WORDS, self.plan)
        elif "k_publish_info" in name:
            self._words(arg(2, Publish), 3, {w: self.plan.get(("info", w), 0) for w in range(3)})
        elif "k_publish_count" in name:
            p = arg(1, Publish)
            p.host[0], p.host[1], p.host[2] = 0, self.error, p.seq

    def _words(self, p, n, values):
        if not self.publish_seq:
            for w in range(PLAN_WORDS):
                p.host[w] = p.seq
            return
        for w in range(n):
            p.host[w] = values.get(w, 0)
        p.host[PLAN_WORDS], p.host[PLAN_WORDS + 1] = 0, p.seq
