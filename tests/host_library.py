"""The library's host code on a machine without a GPU: its own translation units
linked with a fake CUDA runtime (fake_cudart.cpp), loaded through the package's
binding. Kernels do nothing; device memory is guarded host memory whose
overruns are recorded. Imported only by tests."""
import concurrent.futures as cf
import contextlib
import ctypes as C
import os
import subprocess

import numpy as np

from paper_2302_04180_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
FAKE = os.path.join(HERE, "fake_cudart.cpp")
OUT = os.path.join(B.OUT, "host")
LIB = os.path.join(OUT, "librbs_host.so")
HOOK = C.CFUNCTYPE(C.c_int, C.c_char_p, C.c_char_p, C.c_uint64)


def build():
    """No device code for any GPU (PTX only): the kernels never run."""
    files = B._deps() + [FAKE, os.path.abspath(__file__)]
    if os.path.exists(LIB) and all(os.path.getmtime(f) <= os.path.getmtime(LIB) for f in files):
        return LIB
    os.makedirs(OUT, exist_ok=True)
    arch = ["-gencode", "arch=compute_103a,code=compute_103a"]
    sources = [os.path.join(B.CSRC, s) for s in B.SOURCES] + [FAKE]
    objs = [os.path.join(OUT, f"{os.path.basename(s)}.{os.getpid()}.o") for s in sources]

    def one(s, o):
        return subprocess.run([B.nvcc(), *arch, *B.NVCC_FLAGS, "-c", s, "-o", o], capture_output=True, text=True)
    try:
        with cf.ThreadPoolExecutor(max_workers=len(sources)) as ex:
            for r in ex.map(one, sources, objs):
                assert r.returncode == 0, r.stderr[-3000:]
        tmp = f"{LIB}.{os.getpid()}"
        r = subprocess.run([B.nvcc(), *arch, "-cudart", "none", "-shared", "-Xlinker", "-Bsymbolic", "-o", tmp, *objs],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        os.replace(tmp, LIB)
    finally:
        for o in objs:
            if os.path.exists(o):
                os.remove(o)
    return LIB


class DeviceArray:
    """A numpy array's copy in the fake device memory, as the binding takes tensors."""
    is_cuda = False

    def __init__(self, host, a, room=None):
        self.host, self.shape, self.dtype, self.nbytes = host, a.shape, a.dtype, a.nbytes
        self.p = C.c_void_p()
        assert host.fake.cudaMalloc(C.byref(self.p), C.c_size_t(a.nbytes)) == 0
        host.fake.fake_data(self.p)
        C.memmove(self.p.value, a.ctypes.data, a.nbytes)

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return self.p.value

    def numel(self):
        return int(np.prod(self.shape))


class Host:
    """The binding on the fake library; events: every call the hook saw, in order, as
    (call, what, bytes). fail: names of calls or launched kernels to refuse, with
    the error, or a function of (call, what, bytes) that answers it."""

    def __init__(self, rbs, fake):
        self.rbs, self.fake = rbs, fake
        self.events, self.fail = [], None
        fake.fake_faults.restype = C.c_char_p
        fake.fake_find.restype = C.c_void_p
        fake.fake_find.argtypes = [C.c_size_t]
        fake.fake_where.argtypes = [C.c_void_p, C.c_size_t]
        for f in ("fake_state_bytes", "fake_state_done", "fake_state_iter"):
            getattr(fake, f).restype = C.c_size_t

        def hook(call, what, n):
            e = (call.decode(), what.decode(), n if n < 1 << 63 else n - (1 << 64))
            self.events.append(e)
            return int(self.fail(*e) or 0) if self.fail else 0
        self._hook = HOOK(hook)
        fake.fake_hook(self._hook)

    def device(self, a):
        return DeviceArray(self, np.ascontiguousarray(a))

    def csr(self, A):
        return self.rbs.DeviceCSR(A.n, self.device(A.rowptr), self.device(A.col), self.device(A.val))

    def launched(self):
        return [what for call, what, _ in self.events if call == "launch"]

    def faults(self):
        return self.fake.fake_faults().decode()


@contextlib.contextmanager
def host_library():
    import paper_2302_04180_gb300 as rbs
    saved, path = rbs._lib, build()
    rbs._lib = None
    try:
        rbs.load(path)
        h = Host(rbs, rbs._lib)
        yield h
        rbs.rbs_release()
    finally:
        if rbs._lib is not None:
            rbs._lib.fake_hook(None)
            rbs._lib.fake_clear_faults()
        rbs._lib = saved
