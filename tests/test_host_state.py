"""What the host side keeps from call to call, with the CUDA runtime replaced by one that has no device (fake_runtime.cpp): no
test here needs a GPU, and failures, captures and expired waits are planted in the replacement."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2510_18546_b200 import build as enl_build
from paper_2510_18546_b200 import enl
from tests.test_gpu_halves import CASES as HALVES

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


class Cache:
    """A cache on the fake device: two groups of 64 rows and one of `long` rows, and calls over them that take each of the routes."""
    ROUTES = dict(short=("a", [0, 1], 20, 0), prefill=("a", [0, 2], 300, 0), cluster=("c", [0, 1], 1, 0), stream=("d", [0, 2], 1, 8),
                  masses=("m", [0, 2], 40, 0))

    def __init__(self, host, long=4000):
        self.host, self.h = host, ctypes.c_void_p()
        d = enl.CacheDesc(2, 8, 2, 128, 0, 4, long + 200, enl.ENL_BF16, 0, 4, 512, 0)
        assert host.enl_cache_create(ctypes.byref(d), ctypes.byref(self.h)) == enl.ENL_OK
        for g, n in enumerate((64, 64, long)):
            self.store(g, n)

    def store(self, group, n):
        for layer in range(2):
            assert self.host.enl_group_store(self.h, group, layer, n, ctypes.c_void_p(1 << 20), ctypes.c_void_p(1 << 21), 0, None) == enl.ENL_OK

    def attend(self, route, layer=0):
        """Return code, and what was launched: (kind, wait_first) of every launch."""
        kind, sel, n_q, split = self.ROUTES[route]
        ids = np.asarray(sel, np.int32)
        a = enl.AttendArgs()
        a.layer, a.batch, a.n_sel, a.n_q, a.n_new, a.split_hint = layer, 1, len(ids), n_q, n_q, split
        a.sel_ids, a.mass_stride = ids.ctypes.data, len(ids) + 1
        a.q, a.k_new, a.v_new, a.out, a.group_mass = ((1 << 20) * i for i in range(1, 6))
        a.flags = enl.ENL_MASS_ONLY if route == "masses" else 0
        self.host.fake_clear()
        rc = self.host.enl_attend(self.h, ctypes.byref(a), None)
        return rc, [(chr(self.host.fake_kind(i)), self.host.fake_wait_first(i)) for i in range(self.host.fake_launches())]

    def waits(self, route, layer=0):
        """wait_first of a call that goes through, and whether it wrote the gather plan."""
        rc, log = self.attend(route, layer)
        assert rc == enl.ENL_OK
        (first,) = [w for k, w in log if k == self.ROUTES[route][0]]
        return first, any(k in "wp" for k, _ in log)


@pytest.mark.parametrize("refused", ["launch", "map"])
@pytest.mark.parametrize("route", sorted(Cache.ROUTES))
def test_refused_launch_settles_nothing(host, route, refused):
    """The pages stored before a call whose launch was refused may still be on their way in the call after it."""
    c = Cache(host)
    host.fake_fail(ord(Cache.ROUTES[route][0] if refused == "launch" else "e"))
    assert c.attend(route)[0] == enl.ENL_E_CUDA
    host.fake_fail(0)
    assert c.waits(route)[0] == 1
    assert c.waits(route, layer=1) == (0, False)
    c.store(1, 60)
    assert c.waits(route)[0] == 1


@pytest.mark.parametrize("route", sorted(Cache.ROUTES))
def test_captured_call_settles_nothing_outside_its_graph(host, route):
    """A captured call has run when its graph runs, if it does: calls outside the graph go by what was launched outside it, and a
    graph brings its gather plan along, however often and after whatever it runs."""
    inside = route == "short"                                   # such a call carries its plan in its own parameters
    c = Cache(host)
    host.fake_capture(7)
    assert c.waits(route) == (1, not inside)
    assert c.waits(route, layer=1) == (0, False)                # behind the first one in the same graph
    host.fake_capture(0)
    assert c.waits(route) == (1, not inside)                    # the stores are still to be waited for, the plan to be written
    if inside:
        assert c.waits(route, layer=1) == (0, False)
    else:
        assert c.waits(route, layer=1) == (1, True)             # the graph may have run in between and written its own plan there
    host.fake_capture(8)
    assert c.waits(route) == (1, not inside)
    c.store(1, 60)
    assert c.waits(route)[0] == 1
    host.fake_capture(0)
    assert c.waits(route) == (1, not inside)


def test_captured_plan_of_any_size_is_part_of_the_graph(host):
    """A plan too large for one launch's parameters is copied from a buffer that the next plan overwrites; a graph may run later
    than that, so it takes the plan along in pieces.  The next plan does not wait for what was captured."""
    c = Cache(host, long=90000)
    assert [k for k, _ in c.attend("prefill")[1]][:2] == ["p", "a"]
    host.fake_capture(7)
    rc, log = c.attend("prefill")
    assert rc == enl.ENL_OK and [k for k, _ in log][:3] == ["w", "w", "a"]
    assert 28672 == host.fake_bytes(0) >= host.fake_bytes(1) > 0
    host.fake_capture(0)
    c.store(2, 89000)
    assert c.waits("prefill") == (1, True)


@pytest.mark.parametrize("all_layers", [False, True])
@pytest.mark.parametrize("route", sorted(Cache.ROUTES))
def test_captured_store_is_waited_for_whenever_its_graph_may_have_run(host, route, all_layers):
    """A captured store writes the pool when its graph runs, however often that is: calls outside the graph and in other graphs cannot
    know, so their launches read nothing of the pool before what the stream holds has ended."""
    c = Cache(host)
    assert c.waits(route)[0] == 1 and c.waits(route, layer=1) == (0, False)
    host.fake_capture(7)
    if all_layers:
        rows = (ctypes.c_void_p * 2)(1 << 20, 1 << 20)
        assert host.enl_group_store_all_layers(c.h, 1, 64, rows, rows, 0, None) == enl.ENL_OK
    else:
        c.store(1, 64)
    host.fake_capture(0)
    for layer in (0, 1, 0, 1):                                  # the graph may have run before each of these
        assert c.waits(route, layer)[0] == 1
    c.store(1, 60)
    for layer in (0, 1):
        assert c.waits(route, layer)[0] == 1
    host.fake_capture(8)                                        # a graph's first launch waits for all that ran before the graph
    assert c.waits(route)[0] == 1 and c.waits(route, layer=1) == (0, False)
    host.fake_capture(0)
    assert c.waits(route)[0] == 1


@pytest.mark.parametrize("heads", [(1, 1), (2, 1), (4, 1), (8, 1), (16, 1), (8, 2), (32, 8)])
@pytest.mark.parametrize("D", [64, 128])
def test_no_cta_without_keys(host, heads, D):
    """The attention kernel writes nothing for a range of keys without a step of 64: no plan has one, in whichever form."""
    hq, hkv = heads
    h = ctypes.c_void_p()
    d = enl.CacheDesc(1, hq, hkv, D, 0, 4, 8192, enl.ENL_BF16, 0, 4, 2048, 0)
    assert host.enl_cache_create(ctypes.byref(d), ctypes.byref(h)) == enl.ENL_OK
    halves = 0
    for n in (1, 16, 60, 70, 130, 1000):
        assert host.enl_group_store(h, 0, 0, n, ctypes.c_void_p(1 << 20), ctypes.c_void_p(1 << 21), 0, None) == enl.ENL_OK
        for n_q in (2, 17, 63, 64, 65, 127, 128, 129, 255, 256, 257, 500):
            for prior in (0, 1, 63, 64, 65, 127, 128, 129):
                for hint in (0, 64):
                    for n_sel in (0, 1):
                        ids = np.zeros(1, np.int32)
                        a = enl.AttendArgs()
                        a.batch, a.n_sel, a.n_q, a.n_new, a.split_hint, a.sel_ids = 1, n_sel, n_q, n_q + prior, hint, ids.ctypes.data
                        a.q, a.k_new, a.v_new, a.out, a.group_mass = ((1 << 20) * i for i in range(1, 6))
                        a.mass_stride, a.flags = 2, enl.ENL_PLAN_ONLY
                        assert host.enl_attend(h, ctypes.byref(a), None) == enl.ENL_OK
                        out = [ctypes.c_int32() for _ in range(4)]
                        assert host.enl_plan_inspect(h, 0, None, None, ctypes.byref(out[0]), 0, None, None, *(ctypes.byref(x) for x in out[1:])) == enl.ENL_OK
                        _, n_splits, n_items, kind = (x.value for x in out)
                        tile = 128 // (hq // hkv)
                        if n_items != -(-n_q // (2 * tile)) * hkv * n_splits or kind == 3:
                            if kind == 3 or n_items == 0:
                                continue
                            assert n_items == -(-n_q // tile) * hkv * n_splits
                            halves += 1
                        first = min(tile, n_q)                  # the fewest rows a first block may have
                        pages = -(-n // 16) if n_sel else 0
                        assert n_splits <= -(-pages // 4) + (prior + first - 1) // 64 + 1, (n, n_q, prior, hint, n_sel)
    assert halves > 0
    host.enl_cache_free(h)


@pytest.mark.parametrize("want_mass", [True, False])
@pytest.mark.parametrize("name", sorted(HALVES))
def test_form_of_the_calls_that_test_halves(host, name, want_mass):
    """The calls whose results are checked on the GPU as calls with few CTAs are planned as such: the walkers share the steps, with the
    splits on top that the case says."""
    c = HALVES[name]
    n = len(c["pool"])
    lens = [x for pool in c["pool"] for x in pool]
    h = ctypes.c_void_p()
    d = enl.CacheDesc(1, c["Hq"], c["Hkv"], c["D"], 0, len(lens), sum(lens), enl.ENL_BF16, 0, n, sum(c["n_q"]), 0)
    assert host.enl_cache_create(ctypes.byref(d), ctypes.byref(h)) == enl.ENL_OK
    for g, x in enumerate(lens):
        assert host.enl_group_store(h, g, 0, x, ctypes.c_void_p(1 << 20), ctypes.c_void_p(1 << 21), 0, None) == enl.ENL_OK
    ids = np.arange(len(lens), dtype=np.int32)
    cu = [np.concatenate([[0], np.cumsum(x)]).astype(np.int32) for x in ([len(x) for x in c["pool"]], c["n_q"], c["n_new"])]
    a = enl.AttendArgs()
    a.batch, a.n_sel, a.n_q, a.n_new = n, len(ids), sum(c["n_q"]), sum(c["n_new"])
    a.sel_ids, a.mass_stride = ids.ctypes.data, max(len(x) for x in c["pool"]) + 1
    a.cu_sel, a.cu_q, a.cu_new = (x.ctypes.data for x in cu)
    a.q, a.k_new, a.v_new, a.out = ((1 << 20) * i for i in range(1, 5))
    a.group_mass = (1 << 20) * 5 if want_mass else None
    host.fake_clear()
    assert host.enl_attend(h, ctypes.byref(a), None) == enl.ENL_OK
    (i,) = [i for i in range(host.fake_launches()) if chr(host.fake_kind(i)) == "a"]
    assert host.fake_halves(i) == 1
    out = [ctypes.c_int32() for _ in range(4)]
    assert host.enl_plan_inspect(h, 0, None, None, ctypes.byref(out[0]), 0, None, None, *(ctypes.byref(x) for x in out[1:])) == enl.ENL_OK
    assert (out[1].value > 1) == c["splits"]
    host.enl_cache_free(h)
