"""The library's host code against a stand-in for the CUDA runtime
(fake_cudart.cpp): failing allocations, device memory, launches.  No GPU and
no kernel: each script runs in a child process with the stand-in preloaded.
"""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C
import numpy as np
from paper_2008_09441_gb300 import SGError, _lib as L
from paper_2008_09441_gb300.sgpic import Run, Server, sg_estimate_footprint
fake = C.CDLL(None)
for f in ("fake_peak", "fake_in_use"):
    getattr(fake, f).restype = C.c_size_t
fake.fake_launches.restype = C.c_longlong
fake.fake_fail_malloc.argtypes = [C.c_longlong]
launches = lambda part="": fake.fake_launches(part.encode())
rng = np.random.default_rng(1)

def run(d=2, n=6, np_=1000, **kw):
    u, v = rng.random((np_, d)), rng.normal(size=(np_, d))
    return Run((1.0,) * d, n, u, v, np.full(np_, -1.0 / np_), 0.1, **kw)

def status(call, *args):
    try:
        call(*args)
    except SGError as e:
        return e.status
    return L.SG_OK
"""


@pytest.fixture(scope="module")
def stand_in(tmp_path_factory):
    from paper_2008_09441_gb300 import build
    so = tmp_path_factory.mktemp("stand_in") / "fake_cudart.so"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-O1", "-fPIC", "-shared", "-std=c++17", "-I", include, "-o", str(so),
                    os.path.join(HERE, "fake_cudart.cpp")], check=True)

    def script(body):
        r = subprocess.run([sys.executable, "-c", PRELUDE + body], cwd=ROOT, capture_output=True, text=True, timeout=300,
                           env={**os.environ, "LD_PRELOAD": str(so)})
        assert r.returncode == 0, r.stdout + r.stderr
    return script


@pytest.mark.parametrize("d,n,t0,t1", [(2, 6, 1, 3), (3, 4, 1, 2)])
def test_failed_grid_set_leaves_no_launchable_run(stand_in, d, n, t0, t1):
    """No memory for a new tau's arrays: nothing that reads them may launch
    until a grid set is there again."""
    stand_in(f"""
r = run({d}, {n}, tau={t0})
r.step(3)
blob = r.save()
fake.fake_fail_malloc(0)
assert status(r.set_tau, {t1}) == L.SG_ERR_OOM
before = launches()
for call in (lambda: r.step(1), r.step_deposit, r.diagnostics, r.post_diagnostics, r.grid_charges, r.grid_fields,
             r.density, lambda: r.set_solve_variant("passes")):
    assert status(call) == L.SG_ERR_STATE
assert launches() == before
assert r.particles()[0].shape == (1000, {d})
fake.fake_fail_malloc(0)
assert status(r.set_tau, {t1}) == L.SG_ERR_OOM  # the tau that failed is not taken for the current one
r.set_tau({t1})
assert r.grids() and len(r.grids()) == len(run({d}, {n}, tau={t1}).grids())
r.step(2)
r.diagnostics()
fake.fake_fail_malloc(0)
assert status(r.set_tau, {t0}) == L.SG_ERR_OOM
r.load(blob)  # a checkpoint restores the run, whatever its tau
r.step(1)
assert r.diagnostics()["tau"] == {t0}
""")


def test_adaptive_step_without_memory_for_its_tau_can_be_finished(stand_in):
    stand_in("""
r = run(2, 6, tau=L.SG_TAU_ADAPTIVE)
r.set_tau(3)
fake.fake_fail_malloc(0)
assert status(r.step, 1) == L.SG_ERR_OOM  # pushed and deposited, then no room for the selected tau
assert status(r.step, 1) == L.SG_ERR_STATE and status(r.step_fields) == L.SG_ERR_STATE
r.set_tau(2)
r.step_fields()
assert r.diagnostics()["step"] == 1
r.step(2)
assert r.diagnostics()["step"] == 3
""")


def test_failed_estimator_buffers_are_not_taken_for_ready(stand_in):
    stand_in("""
def select_after_failure(nth):
    r = run(3, 4, tau=1)
    base, before = fake.fake_in_use(), launches()
    if nth >= 0:
        fake.fake_fail_malloc(nth)
        if status(r.select_tau) != L.SG_OK:
            assert launches() == before and fake.fake_in_use() == base
    fake.fake_fail_malloc(-1)
    r.select_tau()
    return fake.fake_in_use() - base
whole = select_after_failure(-1)
assert whole > 0
for nth in range(5):
    assert select_after_failure(nth) == whole
""")


def test_failed_admission_launches_no_record(stand_in):
    """The server ends a request whose init failed: nothing reads the arrays
    that the init did not get."""
    stand_in("""
n = 500
for nth in range(2):  # the run's fixed arrays, then its grid set
    s = Server(1 << 30, 2)
    t = s.submit((1.0, 1.0), 5, rng.random((n, 2)), np.zeros((n, 2)), np.full(n, -1.0 / n), 0.1, 2)
    fake.fake_fail_malloc(nth)
    assert status(s.tick) == L.SG_ERR_OOM
    assert s.poll(t)[0] == L.SG_REQ_FAILED and launches("k_diag_record") == 0
""")


@pytest.mark.parametrize("d,prec", [(2, "fp32"), (3, "fp32"), (2, "fp64"), (3, "fp64")])
@pytest.mark.parametrize("sorts", [0, 1])
def test_read_back_takes_no_device_memory(stand_in, d, prec, sorts):
    """Payloads beyond 64 MiB included: a server admits runs by the memory they
    hold between steps, so a read-back may not add to it."""
    np_ = (64 << 20) // ((2 * d + 1) * (4 if prec == "fp32" else 8)) + 259
    stand_in(f"""
d, n = {d}, {np_}
r = run(d, 4, n, precision="{prec}", sort_every=1)
r.step({sorts})  # the current particle set is the second or the first one
a = [np.empty(n, r.dtype) for _ in range(2 * d + 1)]
o = L.sg_particles_out()
o.n, o.w = n, a[2 * d].ctypes.data
for m in range(d):
    o.u[m], o.v[m] = a[m].ctypes.data, a[d + m].ctypes.data
for on_device in (1, 0):
    o.on_device = on_device
    fake.fake_peak(1)
    assert L.lib().sg_pic_get_particles(r.h, C.byref(o)) == L.SG_OK
    assert fake.fake_peak(1) == fake.fake_in_use()
assert launches("k_unpermute_pack") == 1  # the device's own records: in the idle particle set and the keys
""")


def test_every_device_raises_the_shared_memory_limits_it_needs(stand_in):
    """The limit is a property of the kernel on one device: what a first device
    set does not hold on the next."""
    stand_in("""
n, level = 4096, 8
a = [np.zeros(n, np.float32), np.zeros(n, np.float32)]
out = [np.zeros(n, np.uint32) for _ in range(2)] + [np.zeros(1 << (2 * level), np.uint32)]
arr = (C.c_void_p * 3)(a[0].ctypes.data, a[1].ctypes.data, None)
def sort(fn):
    assert fn(L.SG_FP32, 2, level, n, arr, *(C.c_void_p(o.ctypes.data) for o in out), None) == L.SG_OK
for device in (0, 1, 0, 2):
    fake.fake_set_device(device)
    sort(L.lib().sg_cell_sort)
    sort(L.lib().sg_cell_sort_static)
    for kw in (dict(d=2, n=10), dict(d=2, n=11, mode="filter"), dict(d=3, n=6), dict(d=3, n=7, centring="cell"),
               dict(d=2, n=7, precision="fp64"), dict(d=3, n=5, tau=L.SG_TAU_ADAPTIVE)):
        r = run(**kw)
        r.step(7)
        r.close()
    assert fake.fake_missing_opt_in() == 0, device
""")


def test_device_read_back_needs_every_array(stand_in):
    """Host destinations may be left out; a kernel cannot skip a missing device array."""
    stand_in("""
r = run(3, 4)
a = [np.empty(1000, r.dtype) for _ in range(7)]
for missing in range(7):
    o = L.sg_particles_out()
    o.n = 1000
    p = [None if k == missing else x.ctypes.data for k, x in enumerate(a)]
    o.u[0], o.u[1], o.u[2], o.v[0], o.v[1], o.v[2], o.w = p
    o.on_device = 1
    before = launches("k_unpermute")
    assert L.lib().sg_pic_get_particles(r.h, C.byref(o)) == L.SG_ERR_INVALID and launches("k_unpermute") == before
    o.on_device = 0
    assert L.lib().sg_pic_get_particles(r.h, C.byref(o)) == L.SG_OK
""")


@pytest.mark.parametrize("d,ns", [(2, (4, 7, 10)), (3, (4, 5, 6))])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_a_run_fits_its_estimated_footprint(stand_in, d, ns, prec):
    stand_in(f"""
for n in {ns}:
    for tau in (1, 2):
        for np_ in (1000, 100000):
            fake.fake_peak(1)
            before = fake.fake_in_use()
            r = run({d}, n, np_, tau=tau, precision="{prec}")
            r.step(7)
            assert fake.fake_peak(1) - before <= sg_estimate_footprint("{prec}", {d}, n, tau, np_), (n, tau, np_)
            r.close()
""")
