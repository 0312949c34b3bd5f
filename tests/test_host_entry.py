"""What the entry points do around the kernels, on the CPU.

capi.cpp is built with g++ around `tests/host_entry_shim.cpp`: its device
memory is host memory of a settable capacity, its graphs run their branches one
after another, and a solve returns its right-hand side.  So calls that would
race or read memory the library does not hold can be looked at without a GPU.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_2153_gb300", "csrc")
INVALID_ARG, CUDA, OOM = -1, -5, -6


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    out = str(tmp_path_factory.mktemp("entry") / "libentry.so")
    # -Bsymbolic: the library's runtime calls reach the stand-in, whatever else the process has loaded
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", "-I", inc,
                           os.path.join(ROOT, "tests", "host_entry_shim.cpp"), os.path.join(CSRC, "capi.cpp"),
                           "-o", out])
    L = ctypes.CDLL(out)
    L.shim_device.restype = ctypes.c_void_p
    L.shim_device.argtypes = [ctypes.c_int64]
    L.shim_device_free.argtypes = [ctypes.c_void_p]
    L.shim_capacity.argtypes = [ctypes.c_int64]
    L.shim_used.restype = L.shim_peak.restype = ctypes.c_int64
    L.amg_last_error.restype = ctypes.c_char_p
    L.amg_destroy.argtypes = L.amg_batch_destroy.argtypes = [ctypes.c_void_p]
    L.amg_destroy.restype = L.amg_batch_destroy.restype = None
    yield L
    L.shim_capacity(-1)


class Device:
    """A device array of the stand-in runtime; `.a` views it."""

    def __init__(self, lib, values):
        values = np.asarray(values, np.float64)
        self.lib, self.p = lib, lib.shim_device(values.size)
        assert self.p
        self.a = np.ctypeslib.as_array(ctypes.cast(self.p, ctypes.POINTER(ctypes.c_double)), (values.size,))
        self.a[:] = values

    def __del__(self):
        self.lib.shim_device_free(self.p)


def vp(a, offset=0):
    return ctypes.c_void_p((a.p if isinstance(a, Device) else a.ctypes.data) + 8 * offset)


def setup(lib, m, coeff=None):
    h = ctypes.c_void_p()
    rc = lib.amg_setup(2, ctypes.c_int64(m.nv), vp(m.verts), ctypes.c_int64(m.ne), vp(m.elems), vp(m.bflag),
                       None if coeff is None else vp(coeff), None, None, ctypes.byref(h))
    assert rc == 0, lib.amg_last_error()
    return h


def batch_create(lib, handles, nrhs):
    b = ctypes.c_void_p()
    rc = lib.amg_batch_create(len(handles), (ctypes.c_void_p * len(handles))(*[h.value for h in handles]), nrhs,
                              ctypes.c_double(1e-8), None, ctypes.byref(b))
    assert rc == 0, lib.amg_last_error()
    return b


def batch_solve(lib, batch, bs, us):
    n = len(bs)
    its = (ctypes.c_int * n)()
    return lib.amg_batch_solve(batch, (ctypes.c_void_p * n)(*[p.value for p in bs]),
                               (ctypes.c_void_p * n)(*[p.value for p in us]), its, None, None)


# Arrays of a batched call, in units of nv: (bs, us) offsets into one device
# allocation.  Every right-hand side and guess is taken before any solution is
# written, and of two solutions written to one place the later one stays.
OVERLAPS = {
    "u0 on b1": (lambda k: ([0] + [10 + j for j in range(1, k)], [11] + [20 + j for j in range(1, k)])),
    "u0 on half of b1": (lambda k: ([0] + [10 + 2 * j for j in range(1, k)], [12.5] + [30 + j for j in range(1, k)])),
    "last u on b0": (lambda k: ([5 + j for j in range(k)], [20 + j for j in range(k - 1)] + [5])),
    "one u for all": (lambda k: ([j for j in range(k)], [15] * k)),
    "shifted us": (lambda k: ([j for j in range(k)], [15 + 0.5 * j for j in range(k)])),
    "u on its own b": (lambda k: ([j for j in range(k)], [j for j in range(k)])),
    "one b for all": (lambda k: ([3] * k, [10 + j for j in range(k)])),
    "apart": (lambda k: ([j for j in range(k)], [20 + j for j in range(k)])),
}


@pytest.mark.parametrize("name", OVERLAPS)
@pytest.mark.parametrize("nprob,nrhs", [(2, 1), (1, 3), (2, 3), (1, 6)])
def test_batched_arrays_may_overlap(lib, gen, nprob, nrhs, name):
    k = nprob * nrhs
    m = gen.grid2d(5, 1)
    handles = [setup(lib, m) for _ in range(nprob)]
    batch = batch_create(lib, handles, nrhs)
    ob, ou = ([int(o * m.nv) for o in off] for off in OVERLAPS[name](k))
    mem = Device(lib, np.random.default_rng(5).uniform(1, 2, 45 * m.nv))
    want = mem.a.copy()
    sols = [np.where(m.bflag == 0, want[o:o + m.nv], 0) for o in ob]
    for o, u in zip(ou, sols):
        want[o:o + m.nv] = u
    assert batch_solve(lib, batch, [vp(mem, o) for o in ob], [vp(mem, o) for o in ou]) == 0
    assert np.array_equal(mem.a, want)
    lib.amg_batch_destroy(batch)
    for h in handles:
        lib.amg_destroy(h)


GOOD, FAILS = 1.5, 1e200          # the stand-in's coarsest matrix is not positive definite above 1e100


def update(lib, h, m, value, log=False):
    a = np.log(np.full(m.ne, value)) if log else np.full(m.ne, value)
    return (lib.amg_set_log_coefficients if log else lib.amg_update_coefficients)(h, vp(a), None)


@pytest.mark.parametrize("log", [False, True])
def test_a_failed_update_leaves_no_operators_behind(lib, gen, log):
    m = gen.grid2d(5, 1)
    h = setup(lib, m)
    one, many = batch_create(lib, [h], 1), batch_create(lib, [h], 2)
    b, u = np.ones(3 * m.nv), np.zeros(3 * m.nv)
    g, its = np.zeros(m.ne), (ctypes.c_int * 4)()
    prof, val, count = np.zeros(64), ctypes.c_int64(), ctypes.c_int64()
    rtol = ctypes.c_double(1e-8)
    calls = {
        "solve": lambda: lib.amg_solve(h, vp(b), vp(u), rtol, its, None, None),
        "multi": lambda: lib.amg_solve_multi(h, 2, vp(b), vp(u), rtol, its, None, None, None),
        "precond": lambda: lib.amg_precond_apply(h, vp(b), vp(u), None),
        "spmv": lambda: lib.amg_spmv(h, vp(b), vp(u), None),
        "mass": lambda: lib.amg_mass_apply(h, vp(b), vp(u), None),
        "grad": lambda: lib.amg_element_grad(h, vp(b), vp(u), vp(g), None),
        "grad_log": lambda: lib.amg_element_grad_log(h, vp(b), vp(u), vp(g), None),
        "residual": lambda: lib.amg_residual_norm_noalloc(h, vp(b), vp(u), vp(prof), None),
        "profile": lambda: lib.amg_profile(h, vp(b), rtol, vp(prof), its, None),
        "profile_levels": lambda: lib.amg_profile_levels(h, vp(b), rtol, vp(prof), vp(prof), 1, its, None),
        "info": lambda: lib.amg_info(h, 0, 0, ctypes.byref(val)),
        "export": lambda: lib.amg_export(h, 8, 0, None, ctypes.byref(count)),
        "batch_create": lambda: lib.amg_batch_create(1, (ctypes.c_void_p * 1)(h.value), 1, rtol, None, ctypes.byref(ctypes.c_void_p())),
    }
    batches = {"batch": lambda: batch_solve(lib, one, [vp(b)], [vp(u)]),
               "batch of two": lambda: batch_solve(lib, many, [vp(b)] * 2, [vp(u), vp(u, m.nv)])}
    for name, f in {**calls, **batches}.items():
        if name != "batch_create":
            assert f() == 0, (name, lib.amg_last_error())
    assert update(lib, h, m, -1.0) < 0 if not log else True      # refused before anything changes:
    assert calls["solve"]() == 0                                  # the handle keeps its operators
    assert update(lib, h, m, FAILS, log) == CUDA
    solves = lib.shim_solves()
    for name, f in {**calls, **batches}.items():
        assert f() == INVALID_ARG, name
    assert lib.shim_solves() == solves
    assert update(lib, h, m, GOOD, log) == 0
    for name, f in calls.items():
        if name != "batch_create":
            assert f() == 0, (name, lib.amg_last_error())
    for name, f in batches.items():                               # captured before the updates
        assert f() == INVALID_ARG, name
    lib.amg_batch_destroy(one)
    lib.amg_batch_destroy(many)
    lib.amg_destroy(h)


def test_a_failed_update_is_not_taken_for_the_coefficients_held(monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_1410_2153_gb300 import asmg, autograd
    cs = autograd.CoefficientSolver.__new__(autograd.CoefficientSolver)
    cs.solver, cs._set = type("S", (), {"h": None})(), None
    held = []

    def set_(h, c):
        held.append(None)
        if float(c[0]) > 1e100:
            raise asmg.AsmgError(CUDA, "update failed")
        held[-1] = float(c[0])

    monkeypatch.setattr(asmg, "amg_update_coefficients", set_)
    monkeypatch.setattr(asmg, "amg_set_log_coefficients", set_)
    for call in (cs.set_coefficients, cs.set_log_coefficients):
        good = torch.ones(3, dtype=torch.float64)
        call(good)
        with pytest.raises(asmg.AsmgError):
            call(good * 1e200)
        call(good)
        assert held[-1] == 1.0


def test_the_transfer_follows_the_row_order_after_a_failed_update(lib, gen):
    # two colour classes from 2 on: the failed update orders the fine rows as the next good one does
    m = gen.grid2d(5, 1)
    h, fresh = setup(lib, m, np.full(m.ne, GOOD)), setup(lib, m, np.full(m.ne, 3.0))
    assert update(lib, h, m, FAILS) == CUDA
    assert update(lib, h, m, 3.0) == 0
    lib.shim_transfer.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    lib.shim_transfer.restype = ctypes.c_int64
    rows = []
    for x in (h, fresh):
        v = np.full(lib.shim_transfer(x, None), -1.0)
        lib.shim_transfer(x, vp(v))
        rows.append(v)
    assert rows[1].size == 64 and np.array_equal(*rows)
    lib.amg_destroy(h)
    lib.amg_destroy(fresh)


def test_a_mass_product_after_one_that_ran_out_of_memory(lib, gen):
    # the first call builds three arrays: each of their allocations fails once
    m = gen.grid2d(6, 1)
    f, row = np.arange(1.0, m.nv + 1), m.bflag == 0          # whole numbers: exact sums
    want = np.where(row, f * np.bincount(m.elems.ravel(), minlength=m.nv), 0)
    for room in (0, 8 * (m.nv + 1), 8 * (m.nv + 1) + 4 * 3 * m.ne):
        h, b = setup(lib, m), np.zeros(m.nv)
        faults = lib.shim_faults()
        lib.shim_capacity(lib.shim_used() + room)
        assert lib.amg_mass_apply(h, vp(f), vp(b), None) == OOM
        lib.shim_capacity(-1)
        assert lib.amg_mass_apply(h, vp(f), vp(b), None) == 0, lib.amg_last_error()
        assert lib.shim_faults() == faults and np.array_equal(b, want)
        lib.amg_destroy(h)


@pytest.mark.parametrize("where", ["multi", "batch", "batch of two"])
def test_work_state_that_ran_out_of_memory_is_not_used(lib, gen, where):
    # device memory for a part of the work state only, at the first call
    m = gen.grid2d(5, 1)
    h, x, y, its = setup(lib, m), np.ones(2 * m.nv), np.zeros(2 * m.nv), (ctypes.c_int * 4)()
    rtol, batch, n = ctypes.c_double(1e-8), ctypes.c_void_p(), 2 if where == "batch of two" else 1

    def call():
        if where == "multi":
            return lib.amg_solve_multi(h, 2, vp(x), vp(y), rtol, its, None, None, None)
        return lib.amg_batch_create(1, (ctypes.c_void_p * 1)(h.value), n, rtol, None, ctypes.byref(batch))

    faults = lib.shim_faults()
    lib.shim_capacity(lib.shim_used() + 8 * 4 * 32)
    assert call() == OOM
    lib.shim_capacity(-1)
    assert call() == 0, lib.amg_last_error()
    if where != "multi":
        assert batch_solve(lib, batch, [vp(x, j * m.nv) for j in range(n)], [vp(y, j * m.nv) for j in range(n)]) == 0
        lib.amg_batch_destroy(batch)
    assert lib.shim_faults() == faults
    assert np.array_equal(y[:m.nv], m.bflag == 0)
    lib.amg_destroy(h)


@pytest.mark.parametrize("where", ["gradient", "mass", "multi", "batch", "update"])
def test_the_kept_element_stiffness_gives_way(lib, gen, where):
    # device memory for what a call cannot do without, not for the optional element stiffness beside it
    m = gen.grid2d(9, 1)
    x, y, g, its = np.ones(4 * m.nv), np.ones(4 * m.nv), np.zeros(m.ne), (ctypes.c_int * 4)()
    rtol, stiffness = ctypes.c_double(1e-8), 8 * 3 * m.ne

    def call(h, where):
        if where == "gradient":
            return lib.amg_element_grad(h, vp(x), vp(x), vp(g), None)
        if where == "mass":
            return lib.amg_mass_apply(h, vp(x), vp(y), None)
        if where == "multi":
            return lib.amg_solve_multi(h, 4, vp(x), vp(y), rtol, its, None, None, None)
        if where == "batch":
            return lib.amg_batch_create(1, (ctypes.c_void_p * 1)(h.value), 1, rtol, None, ctypes.byref(ctypes.c_void_p()))
        return update(lib, h, m, 3.0)

    bare, h = setup(lib, m), setup(lib, m)
    try:
        if where == "gradient":
            room = max(stiffness, 8 * (2 * m.nv + m.ne))        # enough for the stiffness, were it first
        else:
            assert call(h, "gradient") == 0
            lib.shim_peak()
            before = lib.shim_used()
            assert call(bare, where) == 0
            room = lib.shim_peak() - before - stiffness         # what the call takes, less what h can give back
        lib.shim_capacity(lib.shim_used() + room)
        assert call(h, where) == 0, lib.amg_last_error()
    finally:
        lib.shim_capacity(-1)
    want = g.copy()
    assert call(h, "gradient") == 0 and (where == "gradient" or np.array_equal(g, want)) and g.any()
    lib.amg_destroy(h)
    lib.amg_destroy(bare)
