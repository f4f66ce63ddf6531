"""The library's host code against a stand-in for the CUDA runtime with two devices
(fake_cudart.cpp): what it allocates, waits for and frees, and on which device.  No GPU."""
import ctypes as ct
import glob
import os
import subprocess
import threading
import time

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2112_15562_gb300 import _lib, build

    def objects():
        return [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]

    build.build(force=not all(os.path.exists(o) for o in objects()))
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))))
    include = [d for d in (os.path.join(cuda, "include"), *glob.glob(os.path.join(cuda, "targets", "*", "include")))
               if os.path.exists(os.path.join(d, "cuda_runtime_api.h"))]
    out = str(tmp_path_factory.mktemp("fake") / "libgj_fake.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", include[0],
                    os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objects(), "-o", out], check=True)
    real, _lib._lib, path, _lib.LIB_PATH = _lib._lib, None, _lib.LIB_PATH, out
    try:
        yield _lib.load()
    finally:
        _lib._lib, _lib.LIB_PATH = real, path


def solver(lib, kmax=5):
    """A solver over 4 x 4 x 2 cells in FP64; returns (handle, operators, keep-alive)."""
    from paper_2112_15562_gb300 import _lib as L
    from paper_2112_15562_gb300.api import solver_params

    z = (ct.c_double * 3)(0.0, 10.0, 20.0)
    g = L.Grid(4, 4, 4, 4, 2, 10.0, 10.0, ct.cast(z, ct.POINTER(ct.c_double)), 0.0, 0, 0)
    mag = L.Mag(50000.0, 60.0, 10.0)
    ops = (ct.c_void_p * 2)()
    for i in range(2):
        h = ct.c_void_p()
        assert lib.gj_bttb_setup(ct.byref(g), 1 + i, ct.byref(mag), 0, 0, 0, None, ct.byref(h)) == 0
        ops[i] = h.value
    keep = [(ct.c_double * n)(*([1.0] * n)) for n in (16, 16, 2, 32) for _ in range(2)]
    pair = lambda k: (ct.c_void_p * 2)(*[ct.addressof(x) for x in keep[2 * k:2 * k + 2]])
    P = solver_params(kmax=kmax)
    h = ct.c_void_p()
    assert lib.gj_rrcg_create(ops, ct.byref(P), pair(0), pair(1), None, pair(2), None, pair(3), None, None, ct.byref(h)) == 0
    return h, ops, keep


@pytest.mark.parametrize("current", [0, 1])
def test_a_solver_is_freed_after_its_own_device_is_done(lib, current):
    """Its block is pool memory, which is given back without waiting: destroying it while another
    device is current has to wait for the device that it was made on, and leaves the caller's
    device current."""
    before, blocks = lib.fake_early_frees(), lib.fake_pool_blocks()
    assert lib.cudaSetDevice(0) == 0
    h, ops, keep = solver(lib)
    n = lib.fake_launches()
    assert lib.gj_rrcg_iterate(h, 2, 0, None) == 0 and lib.fake_launches() > n
    assert lib.fake_pool_blocks() == blocks + 1
    lib.cudaSetDevice(current)
    lib.gj_rrcg_destroy(h)
    dev = ct.c_int(-1)
    lib.cudaGetDevice(ct.byref(dev))
    assert dev.value == current
    assert lib.fake_pool_blocks() == blocks
    assert lib.fake_early_frees() == before
    lib.cudaSetDevice(0)
    for op in ops:
        lib.gj_op_destroy(op)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dz", [10.0, 400.0])
def test_a_recomputing_operator_keeps_one_layer(lib, dz, prec):
    """Beside its intermediates (workspace_bytes) and the one spectrum plane, an operator that
    rebuilds its spectra holds the work buffers of one layer's build: more layers add a few depths,
    also when layers forty times as thick as the cells are wide take the near field over the whole
    grid (a depth plane of corner values is then larger than a layer's spectrum)."""
    from paper_2112_15562_gb300 import _lib as L

    lib.fake_held_bytes.restype = ct.c_longlong
    lib.cudaSetDevice(0)
    extra = []
    for nz in (2, 60):
        z = (ct.c_double * (nz + 1))(*[k * dz for k in range(nz + 1)])
        g = L.Grid(200, 180, 200, 180, nz, 10.0, 10.0, ct.cast(z, ct.POINTER(ct.c_double)), 0.0, 0, 0)
        before = lib.fake_held_bytes()
        h, info = ct.c_void_p(), L.OpInfo()
        assert lib.gj_bttb_setup_ex(ct.byref(g), 1, None, prec, 0, 0, L.GJ_SETUP_RECOMPUTE_SPECTRA, None, ct.byref(h)) == 0
        assert lib.gj_op_info(h, ct.byref(info)) == 0
        extra.append(lib.fake_held_bytes() - before - info.workspace_bytes - info.spectrum_bytes)
        lib.gj_op_destroy(h)
        assert lib.fake_held_bytes() == before
    plane = 400 * 360 * 8  # corner values of one depth plane over the whole grid
    assert extra[1] - extra[0] <= plane, extra


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("graph", [0, 1])
def test_a_solver_is_destroyed_while_another_thread_captures(lib, graph, batch):
    """Synchronising the device then fails and breaks that capture, so the solver waits for its own
    work alone; its block is not given back before."""
    lib.cudaSetDevice(0)
    h, ops, keep = solver(lib)
    early, broken = lib.fake_early_frees(), lib.fake_broken_captures()
    assert lib.gj_rrcg_iterate(h, 2, graph, None) == 0
    if batch:
        b = ct.c_void_p()
        assert lib.gj_rrcg_batch_create((ct.c_void_p * 1)(h.value), 1, None, ct.byref(b)) == 0
        assert lib.gj_rrcg_batch_step(b, 3, None) == 0
    lib.fake_capture_elsewhere(1)
    try:
        if batch:
            lib.gj_rrcg_batch_destroy(b)
        lib.gj_rrcg_destroy(h)
        assert lib.fake_broken_captures() == broken
        assert lib.fake_early_frees() == early
    finally:
        lib.fake_capture_elsewhere(0)
    for op in ops:
        lib.gj_op_destroy(op)


def test_one_thread_captures_while_another_destroys(lib):
    """A solve's graph is captured (drawn out here to 0.2 s) while another thread takes its solver and
    its operators down, which waits for the device: not during the capture."""
    lib.cudaSetDevice(0)
    (h, ops, keep), (h2, ops2, keep2) = solver(lib), solver(lib)
    broken = lib.fake_broken_captures()
    lib.fake_capture_lasts(200)
    try:
        status = []
        t = threading.Thread(target=lambda: status.append(lib.gj_rrcg_iterate(h, 1, 1, None)))
        t.start()
        while lib.fake_captures() == 0 and t.is_alive():
            time.sleep(0.001)
        lib.gj_rrcg_destroy(h2)
        for op in ops2:
            lib.gj_op_destroy(op)
        t.join()
    finally:
        lib.fake_capture_lasts(0)
    assert status == [0]
    assert lib.fake_broken_captures() == broken
    lib.gj_rrcg_destroy(h)
    for op in ops:
        lib.gj_op_destroy(op)


def test_an_error_is_reported_once(lib):
    """An operator that does not fit the device is refused with GJ_ERR_OOM, and the next call on
    another operator is not told so again."""
    from paper_2112_15562_gb300 import _lib as L

    lib.cudaSetDevice(0)
    h, ops, keep = solver(lib)
    nz = 20000
    z = (ct.c_double * (nz + 1))(*range(nz + 1))
    g = L.Grid(1000, 1000, 1000, 1000, nz, 10.0, 10.0, ct.cast(z, ct.POINTER(ct.c_double)), 0.0, 0, 0)
    big = ct.c_void_p()
    assert lib.gj_bttb_setup(ct.byref(g), 1, None, 0, 2048, 2048, None, ct.byref(big)) == -2 and not big.value
    m, d = (ct.c_double * 32)(), (ct.c_double * 16)()
    assert lib.gj_g_forward(ops[0], ct.addressof(m), ct.addressof(d), None) == 0, lib.gj_last_error()
    lib.gj_rrcg_destroy(h)
    for op in ops:
        lib.gj_op_destroy(op)
