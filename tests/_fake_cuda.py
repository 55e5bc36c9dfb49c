"""Host-code tests without a device: runs a script in a process of its own whose libhv.so
calls tests/fake_cudart.cpp instead of the CUDA runtime, and orders what that writes down."""
import functools
import json
import os
import subprocess
import sys
import tempfile

from paper_2508_03911_gb300 import build

TESTS = os.path.dirname(os.path.abspath(__file__))

PRELUDE = """
import ctypes as C, json, sys
sys.path.insert(0, %(root)r)
fake = C.CDLL(%(fake)r, mode=C.RTLD_GLOBAL)
fake.fake_log.restype = C.c_char_p
fake.fake_fail_malloc.argtypes = [C.c_size_t, C.c_size_t, C.c_int]
fake.fake_fail_launch.argtypes = [C.c_char_p, C.c_int]
from paper_2508_03911_gb300 import hv

def log():
    return [[int(x) if x.isdigit() else x for x in l.split()] for l in fake.fake_log().decode().splitlines()]

class Dev:  # a device array of which only the address matters
    is_cuda = True
    def __init__(self, shape, size):
        self.shape, self.size, p = shape, size, C.c_void_p()
        assert fake.cudaMalloc(C.byref(p), C.c_size_t(self.numel() * size)) == 0
        self.p = p.value
    def numel(self):
        n = 1
        for s in self.shape: n *= s
        return n
    def element_size(self): return self.size
    def is_contiguous(self): return True
    def data_ptr(self): return self.p
"""


@functools.lru_cache(None)
def _library():
    out = os.path.join(tempfile.mkdtemp(prefix="fake_cudart_"), "fake_cudart.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{build.CSRC}", f"-I{build.INCLUDE}", f"-I{cuda}",
                    os.path.join(TESTS, "fake_cudart.cpp"), "-o", out], check=True)
    return out


def run(script):
    """What the script prints as its last line, from JSON."""
    pre = PRELUDE % dict(root=build.ROOT, fake=_library())
    r = subprocess.run([sys.executable, "-c", pre + script], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return json.loads(r.stdout.splitlines()[-1])


def unordered_copies(log):
    """Pairs of copies into overlapping memory that nothing orders: vector clocks over the
    streams' events and the host's waits."""
    clock, event, host, copies, bad = {}, {}, {}, [], []

    def merge(a, b):
        for k, v in b.items():
            a[k] = max(a.get(k, 0), v)

    for op in log:
        what = op[0]
        if what in ("copy", "kernel", "record", "wait", "graph"):
            s = op[1]
            c = clock.setdefault(s, {})
            merge(c, host)
            c[s] = c.get(s, 0) + 1
            if what == "record":
                event[op[2]] = dict(c)
            elif what == "wait":
                merge(c, event.get(op[2], {}))
            elif what == "copy":
                _, s, dst, src, n = op
                for t, at, d, m in copies:
                    if dst < d + m and d < dst + n and c.get(t, 0) < at:
                        bad.append([d, m, dst, n])
                copies.append((s, c[s], dst, n))
        elif what == "host_stream":
            merge(host, clock.get(op[1], {}))
        elif what == "host_event":
            merge(host, event.get(op[1], {}))
        elif what in ("sync", "malloc", "free"):
            for c in clock.values():
                merge(host, c)
    return bad
