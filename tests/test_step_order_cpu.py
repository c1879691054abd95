"""The order that the host code of the step calls gives to their launches and copies, checked without a GPU.

The library's host code is linked with a device that only keeps vector clocks (tests/host_order/fake_device.cpp):
operations that touch the same memory, one of them writing, without an order between them are reported."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2601_01204_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
H, D = 4, 64
FRAME = H * 256 * D * 2                       # bytes between two tensors of a pool


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    build.build()
    import paper_2601_01204_b200.xkv as xkv
    out = tmp_path_factory.mktemp("host_order")
    nvcc = build._nvcc()
    include = ["-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC]
    so = str(out / "libfake.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-shared", "-cudart", "none",
                    "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic", *include, os.path.join(build.CSRC, "xkv_host.cu"),
                    os.path.join(HERE, "host_order", "fake_device.cpp"), "-o", so], check=True)
    fake = C.CDLL(so)
    for name in xkv.EXPORTED:
        getattr(fake, name).restype = getattr(xkv.lib, name).restype
        getattr(fake, name).argtypes = getattr(xkv.lib, name).argtypes
    fake.fake_report.restype = C.c_char_p
    return fake


class Stack:
    """Caches on addresses that nobody ever reads."""
    bump = 1 << 40

    def __init__(self, lib, layers, budget, n, bits=4, once=0, tail=0, stream=None):
        import paper_2601_01204_b200.xkv as xkv
        self.lib, self.xkv, self.n, self.stream = lib, xkv, n, stream
        self.p = xkv.Params(n_heads=H, budget=budget, max_frame_tokens=n, kv_bits=bits, key_mode=once).c()
        self.caches = []
        for _ in range(layers):
            size = lib.xkv_workspace_bytes(C.byref(self.p))
            h = C.c_void_p()
            assert lib.xkv_create(C.byref(self.p), Stack.take(size), size, stream, C.byref(h)) == 0
            assert lib.xkv_set_unquantised_tail(h, tail) == 0
            self.caches.append(h.value)

    @classmethod
    def take(cls, size):
        at, cls.bump = cls.bump, cls.bump + (size + 4095) // 4096 * 4096
        return at

    def info(self, i):
        x = self.xkv.xkv_info()
        assert self.lib.xkv_get_info(self.caches[i], C.byref(x)) == 0
        return x

    def tensors(self, count):
        return [Stack.take(FRAME) for _ in range(count)]

    def step(self, which, host=False, q=None, k=None, v=None, out=None):
        """One step of the caches with these numbers, in this order; returns the status."""
        n, stream = len(which), self.stream
        arr = lambda xs: (C.c_void_p * n)(*xs)
        q, k, v, out = (x or self.tensors(n) for x in (q, k, v, out))
        caches = arr([self.caches[i] for i in which])
        if host:
            size = self.lib.xkv_stream_step_host_bytes(C.byref(self.p), self.n)
            return self.lib.xkv_stream_step_host(caches, n, arr(q), arr(k), arr(v), arr(out), self.n, Stack.take(size), size, stream)
        return self.lib.xkv_stream_step(caches, n, arr(q), arr(k), arr(v), arr(out), self.n, D, self.n * D, stream)

    def races(self):
        report = self.lib.fake_report().decode()
        self.lib.fake_clear()
        return report


FORMS = [dict(bits=4, once=0), dict(bits=4, once=1), dict(bits=8, once=1), dict(bits=16, once=0), dict(bits=4, once=0, tail=1)]


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("form", FORMS)
def test_a_cache_that_comes_twice_waits_for_its_head_means(lib, form, host):
    s = Stack(lib, 3, 1000, 200, **form)
    for _ in range(9):                        # growing, then evicting
        for order in ([0, 1, 1], [0, 1, 0], [1, 2, 0, 2, 1, 1]):
            assert s.step(order, host) == 0
    assert s.info(1).last_evicted > 0
    assert s.races() == ""


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("form", FORMS)
def test_steps_of_different_layers_are_ordered(lib, form, host):
    """Also with caches long enough that the host-buffer step takes two layers at a time."""
    for layers, budget, n in ((5, 1000, 200), (6, 10700, 250), (31, 600, 130)):
        s = Stack(lib, layers, budget, n, **form)
        for _ in range(budget // n + 3 if layers == 6 else 6):
            assert s.step(range(layers), host) == 0
        assert s.races() == "", (layers, budget, n)


def test_captured_steps_wait_on_nothing_from_before(lib):
    for form in FORMS:
        s = Stack(lib, 2, 1000, 200, **form)
        for _ in range(7):
            assert s.step([0, 1]) == 0
        lib.fake_begin_capture()
        assert s.step([0, 1]) == 0
        assert s.races() == "", form


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("launch", [b"maintenance", b"regroup", b"attention", b"head means"])
@pytest.mark.parametrize("form", FORMS)
def test_a_launch_that_fails(lib, form, launch, host):
    """The caches of a failed launch take no further frame before a reset.  Without their head means, which
    only the next frame needs, regrouped and 16-bit caches go on and compute them anew."""
    s = Stack(lib, 2, 1000, 200, **form)
    for _ in range(7):
        assert s.step([0, 1], host) == 0
    if launch == b"regroup" and (form["bits"] != 4 or form["once"]):
        return
    lib.fake_fail_next(launch)
    assert s.step([0, 1], host) == s.xkv.XKV_E_CUDA
    goes_on = launch == b"head means" and not form["once"]
    status = s.step([0], host)
    assert status == (0 if goes_on else s.xkv.XKV_E_STATE)
    assert lib.xkv_reset(s.caches[0], None) == 0
    assert s.step([0], host) == 0
    assert s.races() == ""


@pytest.mark.parametrize("host", [False, True])
def test_a_step_that_is_not_supported_leaves_the_caches_alone(lib, host):
    """The unquantised tail is not built for 8-bit codes: refused before anything is launched, for every
    layer that would have shared the launch."""
    s = Stack(lib, 3, 1000, 200, bits=8, once=1, tail=1)
    assert s.step([0, 1, 2], host) == s.xkv.XKV_E_UNSUPPORTED
    assert [(s.info(i).frames, s.info(i).stage) for i in range(3)] == [(0, 0)] * 3
    assert lib.fake_ops(b"maintenance") == 0
    for c in s.caches:
        lib.xkv_set_unquantised_tail(c, 0)
    assert s.step([0, 1, 2], host) == 0
    assert s.races() == ""


@pytest.mark.parametrize("launch", [b"maintenance", b"attention", b"head means"])
@pytest.mark.parametrize("nth", [1, 2])
def test_a_step_of_other_caches_in_the_middle_of_one(lib, launch, nth):
    """As when two threads drive different caches on streams of their own."""
    ours, theirs = Stack(lib, 1, 1000, 200, stream=0x11), Stack(lib, 2, 1000, 200, stream=0x22)
    hook = C.CFUNCTYPE(None)(lambda: theirs.step([0, 1]))
    for _ in range(7):
        assert ours.step([0]) == 0 and theirs.step([0, 1]) == 0
        new = Stack(lib, 1, 1000, 200, bits=16, stream=0x11)     # its first frame: no head means behind its attention
        ours.caches[1:] = new.caches
        lib.fake_hook(launch, nth, hook)
        assert ours.step([0, 1]) == 0
        lib.fake_hook(b"", 0, C.CFUNCTYPE(None)())
        assert ours.step([0]) == 0
    assert ours.info(0).last_evicted > 0 and theirs.info(0).last_evicted > 0
    assert ours.races() == ""
