"""The library linked against the fake CUDA runtime of _fake_cudart.cpp (test helper)."""
import contextlib
import ctypes as C
import glob
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import paper_2412_14973_gb300 as T
from paper_2412_14973_gb300 import build as B
from paper_2412_14973_gb300 import tlr_mdd as M

_SO = None


def _build():
    global _SO
    if _SO is None:
        if not (shutil.which(B._nvcc()) or os.path.exists(B._nvcc())) or not shutil.which("g++"):
            pytest.skip("no compiler")
        B.build()   # the objects (nothing to do when they are there)
        objs = [os.path.join(B.BUILD, os.path.basename(s)[:-3] + ".o") for s in glob.glob(os.path.join(B.CSRC, "*.cu"))]
        out = os.path.join(tempfile.mkdtemp(prefix="fakecuda"), "libtlr_fake.so")
        inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(B._nvcc()) or B._nvcc()))), "include")
        src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_fake_cudart.cpp")
        r = subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc, src, *objs, "-o", out],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        _SO = out
    return _SO


@contextlib.contextmanager
def fake():
    """The binding on the fake runtime; yields the fake's own entry points."""
    so = _build()
    was, path = M._LIB, M.lib_path
    M._LIB, M.lib_path = None, lambda: so
    try:
        F = T.lib()
        F.fake_fail.argtypes = [C.c_char_p, C.c_int, C.c_int]
        F.fake_launches.argtypes = [C.c_char_p]
        F.fake_last_upload_block.restype = C.c_void_p
        for f in ("fake_stale_uploads", "fake_uploads", "fake_default_pool_most", "fake_launches"):
            getattr(F, f).restype = C.c_longlong
        yield F
    finally:
        F.fake_fail(b"", 0, 0)
        M._LIB, M.lib_path = was, path


def handle(precision, nr=64, ns=48, b=16, rank=3, stream=None, **kw):
    """A handle on host arrays standing for device memory."""
    g = np.random.default_rng(1)
    D = (g.standard_normal((ns, nr)) + 1j * g.standard_normal((ns, nr))).astype(np.complex64)
    d = T.desc(nr, ns, b, rank=rank, nx=nr // 8, ny=8, precision=precision, diag_mode=T.TLR_DIAG_LOWRANK, **kw)
    return T.tlr_mdd_create(d, D, D, stream), D
