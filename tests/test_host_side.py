"""The host side of the library's calls on a stand-in for the CUDA runtime (tests/fake_cudart.cpp):
per-device and per-context set-up, for which a second GPU or a device reset would be needed."""
import ctypes
import glob
import os
import subprocess

import pytest

from paper_2609_33614_gb300 import build, eat

HERE = os.path.dirname(os.path.abspath(__file__))
KEYS = ("w_router", "w_gate", "w_up", "w_down", "ws_gate", "ws_up", "ws_down", "w_gate_scale",
        "w_up_scale", "w_down_scale", "ws_gate_scale", "ws_up_scale", "ws_down_scale")


@pytest.fixture(scope="module")
def objects(tmp_path_factory):
    build.build()
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.cu.o")))
    if len(objs) != len(build._sources()):
        build.build(force=True)
        objs = sorted(glob.glob(os.path.join(build.BUILD, "*.cu.o")))
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    out = str(tmp_path_factory.mktemp("fake"))
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-I", inc, "-c",
                        os.path.join(HERE, "fake_cudart.cpp"), "-o", out + "/fake.o"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return objs, out


@pytest.fixture
def lib(objects, request):
    """A library of its own per test, so that nothing is set up yet."""
    objs, out = objects
    so = f"{out}/{abs(hash(request.node.name))}.so"
    r = subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, out + "/fake.o"] + objs,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(so, mode=os.RTLD_LOCAL | os.RTLD_NOW)
    for name, (res, args) in eat._SIGS.items():
        getattr(L, name).restype, getattr(L, name).argtypes = res, args
    L.fake_launches.restype = L.fake_setups.restype = ctypes.c_longlong
    return L


def _layer_calls(lib, wdt, xdt, Ts, view=True):
    # (no address is read: they only have to be aligned)
    at = {n: 1 << (20 + i) for i, n in enumerate(KEYS)}
    if not view:  # gate and up in one tensor have no interleaved view
        at["w_up"], at["ws_up"] = at["w_gate"], at["ws_gate"]
    if wdt != eat.EAT_FP8_E4M3:
        at.update({n: None for n in KEYS if n.endswith("scale")})
    base = dict(d_model=256, n_experts=8, d_ff=256, n_shared=1, d_ff_shared=256, max_tokens=max(Ts),
                wdtype=wdt, xdtype=xdt, b_router=None, opd_scale=None, **at)
    desc = eat.eat_layer_desc(*[base[n] for n, _ in eat.eat_layer_desc._fields_])
    p = eat.eat_default_params(2)
    h = ctypes.c_void_p()
    assert lib.eat_create(ctypes.byref(desc), ctypes.byref(p), ctypes.byref(h)) == eat.EAT_OK
    before = lib.fake_setups()
    for T in Ts:
        n = lib.fake_launches()
        r = lib.eat_moe_forward(h, 4096, T, 0, 8192, None, None, None, None)
        assert r == eat.EAT_OK, (T, lib.eat_last_error(h))
        assert lib.fake_launches() > n
    assert lib.eat_destroy(h) == eat.EAT_OK
    return lib.fake_setups() - before


@pytest.mark.parametrize("wdt,xdt", [(eat.EAT_BF16, eat.EAT_BF16), (eat.EAT_FP8_E4M3, eat.EAT_BF16),
                                     (eat.EAT_F32, eat.EAT_F32)])
def test_handles_on_two_devices(lib, wdt, xdt):
    """A kernel's shared-memory limit holds for one device: creating a handle sets it for the
    handle's device, for every kernel that its calls may launch."""
    Ts = (1, 17, 40, 64, 100, 128, 129, 200, 600, 5000)
    for dev in (0, 1):
        lib.fake_set_device(dev)
        for view in (True, False):
            assert _layer_calls(lib, wdt, xdt, Ts, view) == 0  # nothing is left to a handle's calls


def _route_noalloc(lib, T):
    p = eat.eat_default_params(4)
    a = [4096 * i for i in range(1, 9)]
    return lib.eat_route_noalloc(a[0], T, 2048, 64, eat.EAT_BF16, a[1], None, a[2], a[3], a[4],
                                 ctypes.byref(p), 0, a[5], a[6], a[7], None)


def test_noalloc_set_up_by_the_first_call_of_a_context(lib):
    """The first eat_route_noalloc call on a device, of any size, leaves no set-up to later ones (a
    stream capture may follow it), and so does the first one after the device was reset, which takes
    the kernels' shared-memory limits."""
    for dev in (0, 1):
        lib.fake_set_device(dev)
        for _ in range(2):
            assert _route_noalloc(lib, 8) == eat.EAT_OK
            done = lib.fake_setups()
            for T in (128, 300, 2048, 1):
                assert _route_noalloc(lib, T) == eat.EAT_OK, lib.eat_last_error(None)
            assert lib.fake_setups() == done
            lib.fake_reset_device()
