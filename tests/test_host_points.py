"""A plan whose point storage could not be allocated refuses its calls: the library's own objects, linked
with a CUDA runtime stand-in in which allocations are made to fail (no GPU)."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2111_02912_gb300 import _abi, build
    build.build()
    objs = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    d = tmp_path_factory.mktemp("fake")
    rt, so = str(d / "rt.o"), str(d / "libfake.so")
    subprocess.run(["gcc", "-c", "-fPIC", "-w", os.path.join(HERE, "fake_cudart.c"), "-o", rt], check=True)
    subprocess.run(["g++", "-shared", "-o", so] + objs + [rt, "-Wl,-Bsymbolic", "-lpthread"], check=True)
    L = ctypes.CDLL(so)
    vp, i64 = ctypes.c_void_p, ctypes.c_int64
    L.nufft_plan.argtypes = [ctypes.POINTER(vp), ctypes.POINTER(_abi.nufft_opts), i64, vp, vp]
    L.nufft_set_points.argtypes = [vp, i64, vp, vp]
    L.nufft_destroy.argtypes = [vp]
    L.nufft_launch_count.restype = i64
    L.nufft_cg_work_bytes.restype = ctypes.c_size_t
    L.nufft_cg_work_bytes.argtypes = [vp, ctypes.c_int, ctypes.c_int]
    return L, _abi


def _calls(L, h):
    """One of each call of the plan (every pointer non-NULL; nothing runs), as (name, status)."""
    q = ctypes.c_void_p(ctypes.addressof(_calls.buf))
    work = L.nufft_cg_work_bytes(h, 2, 0)
    return [("sort", L.nufft_sort_points(h, None)),
            ("forward", L.nufft_forward(h, 2, q, None, q, None)),
            ("adjoint", L.nufft_adjoint(h, 2, q, None, q, None)),
            ("jvp", L.nufft_jvp_omega(h, 2, q, None, q, q, q, None)),
            ("vjp", L.nufft_vjp_omega_x(h, 2, q, None, q, q, q, None)),
            ("cg", L.nufft_cg_normal(h, 2, q, None, ctypes.c_float(1.0), 1, q, q, ctypes.c_size_t(work), None))]


_calls.buf = ctypes.create_string_buffer(64)


@pytest.mark.parametrize("spread,det,nalloc", [(0, 0, 12), (0, 1, 13), (2, 0, 7)])   # strips, deterministic, tiles
def test_calls_after_a_failed_growth_are_refused(fake, spread, det, nalloc):
    L, abi = fake
    for f in (L.nufft_forward, L.nufft_adjoint, L.nufft_jvp_omega, L.nufft_vjp_omega_x, L.nufft_cg_normal,
              L.nufft_sort_points):
        f.argtypes = None
    o = abi.nufft_default_opts(2, (64, 64))
    o.max_coils, o.spread_variant, o.deterministic = 2, spread, det
    om = ctypes.c_void_p(ctypes.addressof(_calls.buf))
    before = L.fake_live()
    h = ctypes.c_void_p()
    assert L.nufft_plan(ctypes.byref(h), ctypes.byref(o), 1000, om, None) == 0
    assert all(st == 0 for _, st in _calls(L, h))
    held = L.fake_live()
    for k in range(1, nalloc + 1):
        L.fake_fail_malloc(k)
        assert L.nufft_set_points(h, 100000 * k, om, None) == -3   # NUFFT_ERR_OOM
        assert L.fake_fail_left() == 0
        assert L.fake_live() == held - nalloc                      # what the growth had got is given back
        n = L.nufft_launch_count()
        assert [c for c in _calls(L, h) if c[1] != -3] == []
        assert L.nufft_launch_count() == n                         # and nothing was launched
        if k % 3 == 0:   # no points at all need the (smallest) storage too
            assert L.nufft_set_points(h, 0, None, None) == 0
            assert all(st == 0 for _, st in _calls(L, h))
        assert L.nufft_set_points(h, 700, om, None) == 0           # a set_points that succeeds mends the plan
        assert L.fake_live() == held
        assert all(st == 0 for _, st in _calls(L, h))
    L.fake_fail_malloc(nalloc + 1)
    assert L.nufft_set_points(h, 1000000 * nalloc, om, None) == 0  # nalloc is the number of allocations
    assert L.fake_fail_left() == 1
    L.fake_fail_malloc(0)
    L.nufft_destroy(h)
    assert L.fake_live() == before
