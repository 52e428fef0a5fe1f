"""What the library's host code asks of the CUDA runtime, without a GPU: the
library's objects linked with tests/fake_cudart.cpp.  Each check runs in a
process of its own (`python tests/host_calls.py NAME`): a CPU access to device
memory ends it."""
from __future__ import annotations

import ctypes
import os
import subprocess
import sys
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from paper_1507_07039_gb300 import build as b  # noqa: E402

FAKE = os.path.join(b.OBJ_DIR, "libpanda_host_calls.so")


class Opts(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("prec", "diag", "normalize", "t0", "graph_iters")]


class Record(ctypes.Structure):
    _fields_ = [("what", ctypes.c_char * 128)] + [(n, ctypes.c_uint64) for n in ("dst", "src", "bytes", "stream")] + [
        ("async_", ctypes.c_int), ("grid", ctypes.c_int), ("arg", ctypes.c_uint64 * 16)]


def link() -> str:
    """The stand-in library, linked again when an object or the stand-in is newer."""
    src = os.path.join(ROOT, "tests", "fake_cudart.cpp")
    b.build()
    objs = [os.path.join(b.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in b.sources()]
    if not all(os.path.exists(o) for o in objs):
        b.build(force=True)
    if not os.path.exists(FAKE) or os.path.getmtime(FAKE) <= max(os.path.getmtime(p) for p in [src, *objs]):
        with tempfile.TemporaryDirectory(dir=b.OBJ_DIR) as tmp:
            out = os.path.join(tmp, "fake.so")
            subprocess.run([b.nvcc(), *b.ARCH, "-std=c++17", "-shared", "-cudart", "none", "-Xcompiler", "-fPIC",
                            "-Xlinker", "-Bsymbolic", "-o", out, src, *objs, "-ldl", "-lpthread"],
                           check=True, capture_output=True)
            os.replace(out, FAKE)
    return FAKE


def load():
    lib = ctypes.CDLL(link())
    vp, i, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_size_t
    for name, res, args in (("fake_alloc", vp, [i, sz]), ("fake_shadow", vp, [vp]),
                            ("fake_record", ctypes.POINTER(Record), [i]), ("fake_count", i, []),
                            ("panda_last_error", ctypes.c_char_p, [vp]), ("panda_destroy", None, [vp]),
                            ("panda_stream", vp, [vp])):
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    return lib


def records(lib):
    return [lib.fake_record(k).contents for k in range(lib.fake_count())]


def networks(T, G):
    rng = np.random.default_rng(T + G)
    W = rng.standard_normal((T, G)).astype(np.float32)
    return W, np.eye(T, dtype=np.float32), np.eye(G, dtype=np.float32)


def p(a):
    return ctypes.c_void_p(a.ctypes.data if isinstance(a, np.ndarray) else a)


def create(lib, T, G, prec, nets=None, normalize=0):
    ctx, o, nets = ctypes.c_void_p(), Opts(prec, 0, normalize, 0, 8), nets or networks(T, G)
    rc = lib.panda_create(ctypes.byref(ctx), T, G, *(p(x) for x in nets), ctypes.byref(o))
    assert rc == 0, (rc, lib.panda_last_error(None))
    return ctx


def check_stream_order():
    """Nothing that a context's or a set's kernels read is sent by a copy or a
    memset that their stream does not wait for."""
    lib = load()
    T, G = 60, 3000
    for prec in range(4):
        lib.fake_clear()
        ctx = create(lib, T, G, prec)
        stream = lib.panda_stream(ctx)
        for r in records(lib):
            if r.what in (b"copy", b"set"):
                assert r.async_ and r.stream == stream, (prec, r.what, r.bytes, r.stream)
        lib.panda_destroy(ctx)
    nets = networks(T, G)
    for prec in range(4):
        batch, o = ctypes.c_void_p(), Opts(prec, 0, 0, 0, 8)
        arr = [(ctypes.c_void_p * 2)(*[x.ctypes.data] * 2) for x in nets]
        lib.fake_clear()
        rc = lib.panda_batch_create(ctypes.byref(batch), 2, (ctypes.c_int * 2)(T, T), (ctypes.c_int * 2)(G, G), *arr,
                                    ctypes.byref(o))
        assert rc == 0, lib.panda_last_error(None)
        for r in records(lib):
            if r.what in (b"copy", b"set"):
                assert r.async_ and r.stream, (prec, r.what, r.bytes)
        lib.panda_batch_destroy(batch)


def check_another_gpu():
    """Arrays in another GPU's memory are copied, never handed to a kernel and
    never touched by the CPU: create, set_state, get and the static step."""
    lib = load()
    T, G = 40, 300

    def foreign():
        out = []
        for x in networks(T, G):
            a = lib.fake_alloc(1, x.nbytes)
            ctypes.memmove(lib.fake_shadow(a), x.ctypes.data, x.nbytes)
            out.append(a)
        return out

    def no_kernel_sees(arrays, what):
        for r in records(lib):
            if r.what not in (b"copy", b"set", b"sync"):  # StateIn, StateOut, or a pointer comes first
                words = 9 if b"k_load" in r.what or b"k_norms" in r.what else 14 if b"k_store" in r.what else 1
                assert not set(arrays) & set(r.arg[:words]), (what, r.what)

    def copied(arrays, field, what):
        sizes = [4 * T * G, 4 * T * T, 4 * G * G]
        for a, n in zip(arrays, sizes):
            assert sum(r.bytes for r in records(lib) if r.what == b"copy" and getattr(r, field) == a) >= n, what

    for prec in range(4):
        nets, out = foreign(), foreign()
        ctx, o = ctypes.c_void_p(), Opts(prec, 0, 0, 0, 8)
        lib.fake_clear()
        rc = lib.panda_create_device(ctypes.byref(ctx), T, G, *(p(a) for a in nets), ctypes.byref(o), p(0x5550))
        assert rc == 0, lib.panda_last_error(None)
        copied(nets, "src", "create")
        no_kernel_sees(nets, "create")
        lib.fake_clear()
        assert lib.panda_set_state(ctx, *(p(a) for a in nets), 3) == 0, lib.panda_last_error(ctx)
        copied(nets, "src", "set_state")
        no_kernel_sees(nets, "set_state")
        lib.fake_clear()
        assert lib.panda_get_device(ctx, *(p(a) for a in out)) == 0, lib.panda_last_error(ctx)
        copied(out, "dst", "get")
        no_kernel_sees(out, "get")
        lib.panda_destroy(ctx)
    nets = foreign()
    lib.fake_clear()
    rc = lib.panda_step_static(T, G, *(p(a) for a in nets), ctypes.c_float(0.1), 1, 0, None, None)
    assert rc == 0, lib.panda_last_error(None)
    copied(nets, "src", "static")
    copied(nets, "dst", "static")
    no_kernel_sees(nets, "static")
    # in host memory too (kernels read it only on machines that share their page tables)
    nets = networks(T, G)
    rc = lib.panda_step_static(T, G, *(p(a) for a in nets), ctypes.c_float(0.1), 1, 0, None, None)
    assert rc == 0, lib.panda_last_error(None)
    no_kernel_sees([a.ctypes.data for a in nets], "static, host")
    # on this device they are read and written where they lie
    here = [lib.fake_alloc(0, x.nbytes) for x in networks(T, G)]
    lib.fake_clear()
    assert lib.panda_step_static(T, G, *(p(a) for a in here), ctypes.c_float(0.1), 1, 0, None, None) == 0
    assert not any(r.what == b"copy" and (r.src in here or r.dst in here) for r in records(lib))


def check_other_device():
    """On a GPU without tcgen05 every mode, the default one and the static step
    included, is refused before it touches the device."""
    lib = load()
    assert [lib.panda_precision_supported(k) for k in range(-1, 5)] == [0, 1, 1, 1, 1, 0]
    lib.fake_capability(9, 0)
    assert [lib.panda_precision_supported(k) for k in range(4)] == [0, 0, 0, 0]
    nets = networks(8, 20)
    for prec in range(4):
        ctx, o = ctypes.c_void_p(), Opts(prec, 0, 0, 0, 8)
        lib.fake_clear()
        rc = lib.panda_create(ctypes.byref(ctx), 8, 20, *(p(x) for x in nets), ctypes.byref(o))
        assert (rc, ctx.value, lib.fake_count()) == (-8, None, 0), (prec, rc)
    here = [lib.fake_alloc(0, x.nbytes) for x in nets]
    lib.fake_clear()
    rc = lib.panda_step_static(8, 20, *(p(a) for a in here), ctypes.c_float(0.1), 1, 0, None, None)
    assert (rc, lib.fake_count()) == (-8, 0), rc


if __name__ == "__main__":
    globals()["check_" + sys.argv[1]]()
    print("ok")
