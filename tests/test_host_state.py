"""What the host side keeps from call to call, with the CUDA runtime replaced by one that has no device (fake_runtime.cpp): no
test here needs a GPU, and failures, captures and expired waits are planted in the replacement."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2510_18546_b200 import build as enl_build
from paper_2510_18546_b200 import enl

HERE = os.path.dirname(os.path.abspath(__file__))
SOURCES = ["enl_host.cu", "enl_static_scratch.cu", "enl_decode_cluster_sm100.cu"]


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    """The host code and the fake runtime in one library (device code is compiled, but never loaded)."""
    path = str(tmp_path_factory.mktemp("host") / "libhost.so")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=compute_100a", "-std=c++17", "-O1",
                    "-cudart", "none", "-Xcompiler", "-fPIC", "-shared", "-Xlinker", "-Bsymbolic", "-t", "4", "-o", path,
                    os.path.join(HERE, "fake_runtime.cpp")] + [os.path.join(enl_build.CSRC, s) for s in SOURCES], check=True)
    return path


@pytest.fixture
def host(built, tmp_path):
    """A library of its own for every test (a copy: what is kept per process starts anew)."""
    path = str(tmp_path / "libhost.so")
    with open(built, "rb") as f, open(path, "wb") as g:
        g.write(f.read())
    L = ctypes.CDLL(path)
    L.fake_capture.argtypes = [ctypes.c_ulonglong]
    L.fake_bytes.restype = ctypes.c_longlong
    return L


def static_args(D=128, lens=(90, 40, 300), n_new=7, base=1 << 20):
    """Arguments of enl_attend_static; the pointers are never followed."""
    a = enl.StaticArgs()
    seg = np.asarray(lens, np.int32)
    a.n_q_heads, a.n_kv_heads, a.head_dim, a.n_seg, a.n_new = 32, 8, D, len(seg), n_new
    a.seg_len, a.held = seg.ctypes.data, seg
    a.q, a.k, a.v, a.out, a.group_mass = (base * i for i in range(1, 6))
    return a


@pytest.mark.parametrize("D", [64, 128])
def test_static_call_uses_no_heap(host, D):
    """enl_attend_static promises it of every call, the first one on a device included."""
    a = static_args(D)
    for call in range(3):
        host.fake_heap()
        assert host.enl_attend_static(ctypes.byref(a), None) == enl.ENL_OK
        assert host.fake_heap() == 0, f"call {call}"
    assert host.fake_launches() == 3 and host.fake_kind(0) == ord("c")


def test_static_call_that_gave_up_is_reported(host):
    """An expired wait shows once in the status call, whichever head_dim launched the kernel, and not in later ones."""
    assert host.enl_static_status() == enl.ENL_OK               # before any call
    for D in (64, 128):
        a = static_args(D)
        assert host.enl_attend_static(ctypes.byref(a), None) == enl.ENL_OK
        assert host.enl_static_status() == enl.ENL_OK
        host.fake_expire(1)
        assert host.enl_attend_static(ctypes.byref(a), None) == enl.ENL_OK
        host.fake_expire(0)
        assert host.enl_attend_static(ctypes.byref(a), None) == enl.ENL_OK      # a later call does not hide it
        assert host.enl_static_status() == enl.ENL_E_TIMEOUT
        assert host.enl_static_status() == enl.ENL_OK
