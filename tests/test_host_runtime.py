"""Host side of the library on a CUDA runtime that has no device (fake_cudart.cpp):
buffer sizes, shared-memory limits and failing allocations, without a GPU."""
import os
import subprocess
import sys
import textwrap
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]
LIB = ROOT / "paper_2209_00806_gb300" / "_build" / "libtbpm.so"
HEAD = """
import ctypes as C, os, sys
fake = C.CDLL(sys.argv[1], mode=C.RTLD_GLOBAL)
fake.fake_report.restype = C.c_char_p
fake.fake_reset.argtypes = [C.c_long]
fake.fake_live.restype = fake.fake_failed.restype = fake.fake_pinned.restype = fake.fake_waits.restype = C.c_long
lib = C.CDLL(sys.argv[2])
lib.tbpm_last_error.restype = C.c_char_p
lib.tbpm_last_error.argtypes = [C.c_void_p]
lib.tbpm_destroy.argtypes = [C.c_void_p]
Z = C.c_double(1.5707963267948966)
FP64, FP32, HOST = 0, 1, 0
def dbl(n, v=0.0): return (C.c_double * max(n, 1))(*([v] * n))
def create():
    h = C.c_void_p()
    assert lib.tbpm_create(C.byref(h), 0, None) == 0
    return h
def build(h, n, onsite=True, flags=0, deg=1):
    # `deg` bonds an orbital: (u, u + 1), (u, u + 2), ..., all of one value
    m = n * deg
    i = (C.c_int64 * m)(*[u for d in range(deg) for u in range(n)])
    j = (C.c_int64 * m)(*[(u + d + 1) % n for d in range(deg) for u in range(n)])
    return lib.tbpm_build_hamiltonian(h, C.c_int64(n), dbl(n) if onsite else None, C.c_int64(m), i, j,
                                      dbl(m, 1.0), C.c_double(10.0), 1, None, HOST, flags)
def states(h, n, S): return lib.tbpm_set_phase_states(h, S, dbl(n * S), HOST)
def run(h, S, steps, prec, flags=0):
    return lib.tbpm_propagate(h, Z, steps, prec, dbl(2 * S * (steps + 1)), HOST, flags)
def clean(): assert fake.fake_report() == b"", fake.fake_report()
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    import __graft_entry__
    bn = __graft_entry__._build_module()
    bn.build()
    so = tmp_path_factory.mktemp("fake") / "libfake_cudart.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(bn.CUDA_HOME, "include"), str(Path(__file__).with_name("fake_cudart.cpp")),
                    "-o", str(so)], check=True)
    return so


def run_script(fake, body):
    env = dict(os.environ, LD_PRELOAD=str(fake))
    r = subprocess.run([sys.executable, "-c", HEAD + textwrap.dedent(body), str(fake), str(LIB)],
                       capture_output=True, text=True, env=env, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


# a new number of states with the old number of steps: C and the norms are
# read back whole, by the per-term kernels and by the cluster stepping
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("config", [None, 1])
def test_outputs_fit_the_states(fake, prec, config):
    run_script(fake, f"""
        h = create()
        if {config}: assert lib.tbpm_set_launch_config(h, {prec}, 8, 64, {config}) == 0
        n = 700
        assert build(h, n) == 0
        for S in (1, 16, 2, 5):
            assert states(h, n, S) == 0 and run(h, S, 9, {prec}) == 0, lib.tbpm_last_error(h)
            avg = dbl(2 * 10)
            assert lib.tbpm_correlation(h, avg, HOST) == 0
            clean()
        lib.tbpm_destroy(h)
        assert fake.fake_live() == 0
    """)


# a kernel's shared-memory limit is the process's: a smaller sample in another
# context does not lower what a larger one's launches need (cluster stepping)
@pytest.mark.parametrize("prec,sides", [(0, (8000, 5000)), (1, (16000, 9000))])
def test_shared_memory_limits_are_not_lowered(fake, prec, sides):
    run_script(fake, f"""
        a, b = create(), create()
        for h, n in zip((a, b), {sides}):
            assert build(h, n) == 0 and states(h, n, 4) == 0
            assert run(h, 4, 2, {prec}) == 0, lib.tbpm_last_error(h)
        assert run(a, 4, 2, {prec}) == 0, lib.tbpm_last_error(a)
        clean()
    """)


# long rows of FP32 values: the staged gathers' lists (device memory that stays)
# come only where a group of four or eight states reads them, once the steps
# pay for them
@pytest.mark.parametrize("S,lists", [(1, False), (2, False), (3, False), (16, False), (4, True),
                                     (8, True), (13, True), (20, True)])
def test_lists_are_built_for_the_widths_that_read_them(fake, S, lists):
    run_script(fake, f"""
        h = create()
        assert build(h, 2000, flags=16, deg=17) == 0        # TBPM_BUILD_NO_UNIFORM, 34 entries a row
        assert states(h, 2000, {S}) == 0
        live = []
        for steps in (3, 130, 130):
            assert run(h, {S}, steps, FP32) == 0, lib.tbpm_last_error(h)
            live.append(fake.fake_live())
        clean()
        assert (live[1] > live[0]) == {lists} and live[2] == live[1], live
        lib.tbpm_destroy(h)
        assert fake.fake_live() == 0
    """)


# every allocation of a call fails once: the lists that the default builds on its
# own are optional (the call succeeds without), any other failure is OOM, leaves
# the context usable, and nothing of it stays allocated
@pytest.mark.parametrize("what", ["lists", "asked", "build", "states", "run", "adjoint"])
def test_a_failing_allocation(fake, what):
    run_script(fake, f"""
        what = {what!r}
        n, S, OOM = 2000, 4, 3
        def prepare():
            h = create()
            if what == "asked": assert lib.tbpm_set_launch_config(h, FP32, 8, 64, 4609) == 0
            if what == "build": return h
            assert build(h, n, flags=16, deg=17) == 0
            if what == "states": return h
            assert states(h, n, S) == 0
            if what == "lists": assert run(h, S, 20, FP32) == 0      # 80 states x steps of the 128
            return h
        def call(h):
            if what == "build": return build(h, n, flags=16, deg=17)
            if what == "states": return states(h, n, S)
            if what == "adjoint":
                g, a, b = dbl(2 * S * 4), dbl(17 * n), dbl(n)
                return lib.tbpm_propagate_adjoint(h, Z, 3, g, HOST, 2, a, b, HOST)
            return run(h, S, 20, FP32)
        k = 0
        while True:
            h = prepare()
            fake.fake_reset(k)
            rc = call(h)
            failed = fake.fake_failed()
            fake.fake_reset(-1)
            if what == "lists": assert rc == 0, (k, lib.tbpm_last_error(h))
            else: assert rc == (OOM if failed else 0) or (rc == 0 and what in ("asked", "adjoint")), (k, rc)
            assert call(h) == 0, (k, lib.tbpm_last_error(h))
            clean()
            lib.tbpm_destroy(h)
            clean()
            assert fake.fake_live() == 0, (k, fake.fake_live())
            if not failed: break
            k += 1
        assert k >= 2
    """)


# one-shot contexts pay for no page-locked memory (0.2 ms), whatever the size of C
@pytest.mark.parametrize("steps", [4, 3000])
def test_a_first_run_locks_no_pages(fake, steps):
    run_script(fake, f"""
        h = create()
        assert build(h, 700) == 0 and states(h, 700, 2) == 0 and run(h, 2, {steps}, FP32) == 0
        assert fake.fake_pinned() == 0
        clean()
    """)


# a run waits for the device once, stepped in clusters as term by term
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("config", [None, 1])
def test_a_run_waits_once(fake, prec, config):
    run_script(fake, f"""
        h = create()
        if {config}: assert lib.tbpm_set_launch_config(h, {prec}, 8, 64, {config}) == 0
        assert build(h, 700) == 0 and states(h, 700, 3) == 0 and run(h, 3, 5, {prec}) == 0
        before = fake.fake_waits()
        assert run(h, 3, 5, {prec}) == 0
        assert fake.fake_waits() == before + 1
        clean()
    """)


# a run whose result buffers cannot be had leaves no results of the last one to
# read, but states to go on from
def test_no_results_after_a_failed_run(fake):
    run_script(fake, """
        h = create()
        assert build(h, 700) == 0 and states(h, 700, 2) == 0 and run(h, 2, 5, FP64) == 0
        fake.fake_reset(0)
        assert run(h, 2, 9, FP64) == 3 and fake.fake_failed() == 1
        fake.fake_reset(-1)
        avg, norms = dbl(40), dbl(40)
        assert lib.tbpm_correlation(h, avg, HOST) == 8       # TBPM_E_STATE
        assert lib.tbpm_get_norms(h, norms) == 8
        assert run(h, 2, 9, FP64, 4) == 0                    # TBPM_PROP_RESUME
        assert lib.tbpm_correlation(h, avg, HOST) == 0 and lib.tbpm_get_norms(h, norms) == 0
        clean()
    """)


# the cluster stepping's tables and the fused step's are the same memory
def test_fused_after_cluster_keeps_no_memory(fake):
    run_script(fake, """
        h = create()
        assert build(h, 700) == 0 and states(h, 700, 1) == 0
        assert run(h, 1, 5, FP64) == 0 and run(h, 1, 5, FP64, 8) == 0       # TBPM_PROP_PERSISTENT
        lib.tbpm_destroy(h)
        clean()
        assert fake.fake_live() == 0
    """)


# an allocation that fails while a context's buffers grow: a later, smaller run has
# every buffer that a fresh context has (a null one would be written by a kernel)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("config", [None, 1, 8])
def test_buffers_are_whole_after_a_failed_growth(fake, prec, config):
    run_script(fake, f"""
        n, small, large = 3000, 1, 8
        def context():
            h = create()
            if {config}: assert lib.tbpm_set_launch_config(h, {prec}, 8, 64, {config}) == 0
            assert build(h, n) == 0
            return h
        def go(h, S, steps): return states(h, n, S) or run(h, S, steps, {prec})
        h = context()
        assert go(h, small, 5) == 0
        whole = fake.fake_live()
        lib.tbpm_destroy(h)
        for first in (True, False):             # the growing run is the context's first, or not
            k = 0
            while True:
                h = context()
                if first: assert go(h, small, 5) == 0
                fake.fake_reset(k)
                rc = go(h, large, 5)
                failed = fake.fake_failed()
                fake.fake_reset(-1)
                assert rc == (3 if failed else 0), (k, rc)
                assert go(h, small, 5) == 0 and fake.fake_live() == whole, (first, k, fake.fake_live(), whole)
                clean()
                lib.tbpm_destroy(h)
                assert fake.fake_live() == 0
                if not failed: break
                k += 1
    """)


# a fresh run that fails after it has taken the states back to their start leaves
# nothing to resume
def test_a_failed_fresh_run_cannot_be_resumed(fake):
    run_script(fake, """
        h = create()
        assert build(h, 700) == 0 and states(h, 700, 1) == 0
        assert run(h, 1, 5, FP64, 8) == 0                    # TBPM_PROP_PERSISTENT
        fake.fake_reset(0)                                   # the cluster stepping's state table
        assert run(h, 1, 5, FP64) == 3 and fake.fake_failed() == 1
        fake.fake_reset(-1)
        assert run(h, 1, 5, FP64, 4) == 8                    # TBPM_PROP_RESUME: TBPM_E_STATE
        assert run(h, 1, 5, FP64) == 0 and run(h, 1, 5, FP64, 4) == 0
        clean()
    """)
