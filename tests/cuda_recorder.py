"""The library's host code on a recording stand-in for the CUDA runtime (cuda_recorder.cpp): no GPU, no kernels."""
import ctypes
import glob
import os
import subprocess
import tempfile
from contextlib import contextmanager

HERE = os.path.dirname(os.path.abspath(__file__))


def _link(out: str) -> None:
    from paper_1708_00033_gb300 import _build
    _build.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc())))
    include = [d for d in glob.glob(os.path.join(cuda, "targets", "*", "include")) + [os.path.join(cuda, "include")]
               if os.path.exists(os.path.join(d, "cuda_runtime_api.h"))]
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include[0], "-o", out,
                    os.path.join(HERE, "cuda_recorder.cpp")] + glob.glob(os.path.join(_build.OUT, "*.o")), check=True)


@contextmanager
def recorded(stream: int = 8):
    """(lib, ctx): the library on the stand-in, bound as hf's library for the block's duration, and a context of
    ``stream``.  Objects made in the block are closed in it."""
    from paper_1708_00033_gb300 import hf
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "libhf_recorded.so")
        _link(path)
        saved = hf._lib, hf.LIB_PATH
        hf._lib, hf.LIB_PATH = None, path
        try:
            lib = hf.load_library()
            lib.rec_log.restype = ctypes.c_char_p
            lib.rec_live_bytes.restype = lib.rec_peak_bytes.restype = ctypes.c_ulonglong
            lib.rec_set_limit.argtypes = [ctypes.c_ulonglong]
            lib.rec_launch.argtypes = [ctypes.c_ulonglong, ctypes.c_char_p]
            lib.rec_read_words.argtypes = [ctypes.c_int, ctypes.c_ulonglong]
            ctx = hf.Context(0, stream=stream)
            try:
                yield lib, ctx
            finally:
                ctx.close()
        finally:
            hf._lib, hf.LIB_PATH = saved


def log(lib):
    """[(operation, stream, argument)] in the order of the calls; what a graph captured is left out."""
    out, depth = [], 0
    for line in lib.rec_log().decode().splitlines():
        op, stream, what = line.split(" ", 2)
        if op == "capture":
            depth += 1
        elif op == "captured":
            depth -= 1
        elif not depth:
            out.append((op, int(stream), what))
    return out


def happens_before(ops):
    """For each operation, the set of earlier operations that streams, events and host waits order before it."""
    streams, events, host, out = {}, {}, set(), []
    for i, (op, s, what) in enumerate(ops):
        here = streams.setdefault(s, set())
        if op == "wait":
            here |= events.get(what, set())
        elif op == "record":
            events[what] = set(here)
        elif op == "sync":
            host |= here
        elif op == "eventsync":
            host |= events.get(what, set())
        else:
            here |= host
            out.append(set(here))
            here.add(i)
            continue
        out.append(set())
    return out
