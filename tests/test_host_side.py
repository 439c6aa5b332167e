"""The host side of the solver on a CUDA runtime of host memory (fake_cuda.cpp): which kernels
a call launches on which arrays, also after an allocation that fails and in graphs."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1901_00682_gb300", "csrc")


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1901_00682_gb300 import _lib, build
    nvcc = subprocess.run(["which", build._nvcc()], capture_output=True, text=True).stdout.strip()
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    so = str(tmp_path_factory.mktemp("host") / "libhost.so")
    # (-Bsymbolic: its own runtime, whichever other one the process has loaded)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include, "-x", "c++",
                    os.path.join(HERE, "fake_cuda.cpp"), os.path.join(CSRC, "dd_tv.cu"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for name, (res, args) in _lib.SIGNATURES.items():
        if hasattr(lib, name):
            getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_fail_allocations.argtypes = [ctypes.c_size_t]
    return lib


@pytest.fixture
def lib(fake):
    yield fake
    fake.fake_fail_allocations(0)
    fake.fake_fail_allocation(0)
    fake.fake_fail_prepare(0)
    fake.fake_chain(0)


class Handle:
    def __init__(self, lib, *args, **kw):
        from paper_1901_00682_gb300 import _lib
        self.lib, self.h = lib, ctypes.c_void_p()
        d = _lib.Params()
        lib.dd_tv_default_params(ctypes.byref(d))
        for k, v in dict(alpha=10.0, **kw).items():
            setattr(d, k, v)
        d.height, d.width, d.sub_rows, d.sub_cols = args
        self.shape = args[:2]
        self.rc = lib.dd_tv_create(ctypes.byref(self.h), ctypes.byref(d))

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.lib.dd_tv_destroy(self.h)

    def load(self, f, mask=None):
        return self.lib.dd_tv_load(self.h, f.ctypes.data, None if mask is None else mask.ctypes.data)

    def launches(self, n_outer):
        """The launches of n_outer outer iterations."""
        self.lib.fake_clear_log()
        assert self.lib.dd_tv_iterate(self.h, n_outer) == 0
        return self.lib.fake_log().decode().split("\n")[:-1]

    def u(self):
        out = np.empty(self.shape, np.float32)
        assert self.lib.dd_tv_get_u(self.h, out.ctypes.data) == 0
        return out


@pytest.mark.parametrize("path,kernels", [(0, {"interface", "local"}), (2, {"full"})])
def test_load_that_fails_leaves_the_handle_as_it_was(lib, path, kernels):
    """The first masked load finds no memory for the mask: the captured loop of the unmasked
    problem goes on, and a later masked load does not replay it."""
    H, W = 96, 64
    f, g, m = np.zeros((H, W), np.float32), np.ones((H, W), np.float32), np.ones((H, W), np.uint8)
    with Handle(lib, H, W, 2, 1, path=path) as s:
        assert s.load(f) == 0
        lib.fake_fail_allocations(m.nbytes)
        assert s.load(g, m) == 2   # ENOMEM
        lib.fake_fail_allocations(0)
        assert s.u()[-1, -1] == 0
        assert set(s.launches(8)) == kernels
        assert s.load(g, m) == 0
        masked = [k for k in s.launches(8) if k != "interface"]
        assert masked and all(k.endswith(" masked") for k in masked)
        assert s.load(f) == 0
        assert set(s.launches(8)) == kernels


@pytest.mark.parametrize("K", [1, 7, 10, 15])
@pytest.mark.parametrize("n_outer", [1, 2, 3])
@pytest.mark.parametrize("before", [0, 1, 5])
def test_full_dimension_iterations_replay_from_a_callers_graph(lib, K, n_outer, before):
    """Outer iterations captured into a caller's graph advance the iterate at every replay,
    whichever set of arrays held it, and the handle goes on from there."""
    H, W = 70, 60
    f = np.zeros((H, W), np.float32)
    with Handle(lib, H, W, 1, 1, path=2, inner_iters=K) as s:
        assert s.load(f) == 0
        s.launches(before)
        graph, run, out = ctypes.c_void_p(), ctypes.c_void_p(), np.empty_like(f)
        assert lib.cudaStreamBeginCapture(None, 0) == 0
        assert lib.dd_tv_iterate(s.h, n_outer) == 0
        assert lib.dd_tv_get_u(s.h, ctypes.c_void_p(out.ctypes.data)) == 0
        assert lib.cudaStreamEndCapture(None, ctypes.byref(graph)) == 0
        assert lib.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)) == 0
        lib.cudaGraphDestroy(graph)
        for r in (1, 2, 3):
            assert lib.cudaGraphLaunch(run, None) == 0
            assert out[0, 0] == K * (before + r * n_outer)
        lib.cudaGraphExecDestroy(run)
        s.launches(6)
        assert s.u()[0, 0] == K * (before + 3 * n_outer + 6)


HALF_STEPS = ["ustep", "pstep"]


def test_full_dimension_without_room_for_the_second_set(lib):
    """Only then the path runs a launch per half-step in place; state and results as otherwise."""
    H, W, K = 70, 60, 3
    f = np.zeros((H, W), np.float32)
    lib.fake_fail_allocations(2 * 4 * H * W)   # more than any single array
    with Handle(lib, H, W, 1, 1, path=2, inner_iters=K) as s:
        assert s.rc == 0
        lib.fake_fail_allocations(0)
        assert s.load(f) == 0
        assert s.launches(1) == HALF_STEPS * K
        assert s.launches(6) == HALF_STEPS * (6 * K)
        assert s.u()[0, 0] == 7 * K
    with Handle(lib, H, W, 1, 1, path=2, inner_iters=K) as s:
        assert s.load(f) == 0
        assert s.launches(7) == ["full"] * 7


@pytest.mark.parametrize("path", [0, 2])
def test_create_reports_a_kernel_set_up_that_fails(lib, path):
    lib.fake_fail_prepare(98)   # cudaErrorInvalidDeviceFunction
    with Handle(lib, 70, 60, 1, 1, path=path) as s:
        assert s.rc == 3 and not s.h.value   # ECUDA
        assert b"set-up" in lib.dd_tv_last_error(None)


@pytest.mark.parametrize("path,n", [(0, 9), (1, 16), (2, 12)])
def test_create_reports_each_allocation_that_fails(lib, path, n):
    """Every allocation of a new handle in turn finds no memory."""
    codes = []
    for k in range(1, 40):
        lib.fake_fail_allocation(k)
        with Handle(lib, 70, 60, 2, 2, path=path) as s:
            codes.append(s.rc)
            assert (s.rc == 0) == bool(s.h.value)
            if s.rc:
                assert b"cudaMalloc" in lib.dd_tv_last_error(None)
    assert codes.count(2) >= n and set(codes) == {0, 2}


@pytest.mark.parametrize("H,W,K,half_steps", [(70, 61, 1, True), (70, 60, 1, False), (70, 61, 2, False),
                                              (2047, 2049, 1, True), (2049, 2049, 1, False)])
def test_single_full_dimension_iterations_of_unaligned_rows_run_half_steps(lib, H, W, K, half_steps):
    f = np.zeros((H, W), np.float32)
    with Handle(lib, H, W, 1, 1, path=2, inner_iters=K) as s:
        assert s.load(f) == 0
        assert s.launches(5) == (HALF_STEPS if half_steps else ["full"]) * 5


def _operations(lib, call):
    before = lib.fake_operations()
    assert call() == 0
    return lib.fake_operations() - before


@pytest.mark.parametrize("sub", [(2, 2), (3, 1), (1, 3), (1, 1)])
def test_chained_update_costs_loads_and_set_state_nothing(lib, sub):
    """The arrays that the local solves' own multiplier update needs are set without more copies
    and launches than a handle without it takes (one for what follows from the strips)."""
    H, W = 70, 60
    f, ops = np.ones((H, W), np.float32), []
    P1, P2 = np.zeros((H + sub[0], W), np.float32), np.zeros((H, W + sub[1]), np.float32)
    lam = np.zeros(4 * (H + W), np.float32)
    for chain in (0, 1):
        lib.fake_chain(chain)
        with Handle(lib, H, W, *sub) as s:
            state = [a.ctypes.data for a in (f, P1, P2, lam, lam, P1, P2)]
            ops.append((_operations(lib, lambda: s.load(f)), _operations(lib, lambda: lib.dd_tv_set_state(s.h, *state, 3))))
    assert ops[1][0] == ops[0][0]
    assert ops[1][1] <= ops[0][1] + (sub != (1, 1))
    assert ops[1][1] <= 3 + (sub[0] > 1) + (sub[1] > 1) + 2


def test_second_set_of_arrays_takes_no_allocation_of_its_own(lib):
    """Creating a full-dimension handle allocates no more often with it than without."""
    n = []
    for W in (60, 61):   # two sets; one (single iterations of unaligned rows)
        before = lib.fake_allocations()
        with Handle(lib, 70, W, 1, 1, path=2, inner_iters=1) as s:
            assert s.rc == 0
            n.append(lib.fake_allocations() - before)
    assert n[0] <= n[1]
