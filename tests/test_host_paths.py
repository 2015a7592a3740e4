"""The host code behind the C ABI (csrc/api.cu) against a runtime that keeps books (fake_cuda.cpp): what it enqueues, and what it
leaves behind where a call of the runtime fails. Runs on the CPU."""
import ctypes as C
import os
import subprocess
import sys

import pytest

import paper_2510_02470_b200 as sage

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("host") / "libhost.so")
    csrc = os.path.join(ROOT, "paper_2510_02470_b200", "csrc")
    cmd = ["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", csrc, "-I", os.path.join(CUDA, "include"),
           "-x", "c++", os.path.join(csrc, "api.cu"), os.path.join(HERE, "fake_cuda.cpp"), "-o", out, "-Wl,-z,defs", "-Wl,-Bsymbolic", "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    L = C.CDLL(out)
    for name, (res, args) in sage.SIGNATURES.items():
        if hasattr(L, name):
            getattr(L, name).restype, getattr(L, name).argtypes = res, args
    return L


def _handle(L, D=64, ell=4, P=1, dtype=0):
    h = C.c_void_p()
    assert L.sage_fd_create(C.byref(h), D, ell, dtype, 0) == 0
    if P > 1:
        assert L.sage_fd_set_option(h, 6, P) == 0
    return h


def _appends(L):
    buf = (C.c_longlong * 5000)()
    n = L.fake_appends(buf, 1000)
    return [tuple(buf[5 * i:5 * i + 5]) for i in range(n)]


def _calls(L, name):
    return L.fake_calls(name.encode())


def test_cycles_become_graphs_without_a_capture(lib):
    """The merged form replays its cycles as graphs. A captured stream would be every other thread's business: a synchronisation of
    the device anywhere in the process ends the capture and fails itself."""
    h = _handle(lib, P=2)
    b0, g0 = _calls(lib, "cudaStreamBeginCapture"), _calls(lib, "cudaGraphLaunch")
    assert lib.sage_fd_update(h, 0x1000, 2 * 5 * 40, 64, None) == 0
    assert _calls(lib, "cudaStreamBeginCapture") == b0 and _calls(lib, "cudaGraphLaunch") > g0
    st = sage.SageStats()
    assert lib.sage_fd_stats(h, C.byref(st)) == 0
    launches = st.kernel_launches
    lib.sage_fd_destroy(h)
    # the same rows with direct launches (per-kernel timing on): as many kernels
    h = _handle(lib, P=2)
    lib.sage_fd_set_option(h, 3, 1)
    assert lib.sage_fd_update(h, 0x1000, 2 * 5 * 40, 64, None) == 0
    assert lib.sage_fd_stats(h, C.byref(st)) == 0 and st.kernel_launches == launches
    lib.sage_fd_destroy(h)


def test_a_captured_stream_takes_no_graphs(lib):
    """Updates that the caller captures run launch by launch, also when the sketch has graphs of its cycles by then: a graph cannot be
    launched into a capture."""
    h = _handle(lib, P=2)
    assert lib.sage_fd_update(h, 0x1000, 2 * 5 * 40, 64, None) == 0
    g0, i0 = _calls(lib, "cudaGraphLaunch"), _calls(lib, "cudaGraphInstantiate")
    lib.fake_capturing(1)
    assert lib.sage_fd_update(h, 0x1000, 2 * 5 * 40, 64, None) == 0
    lib.fake_capturing(0)
    assert _calls(lib, "cudaGraphLaunch") == g0 and _calls(lib, "cudaGraphInstantiate") == i0
    lib.sage_fd_destroy(h)


@pytest.mark.parametrize("what", ["cudaGraphCreate", "cudaGraphAddNode_v2", "cudaGraphInstantiate"])
def test_a_cycle_that_cannot_become_a_graph_runs_directly(lib, what):
    h = _handle(lib, P=2)
    lib.fake_fail(what.encode(), 1)
    assert lib.sage_fd_update(h, 0x1000, 2 * 5 * 40, 64, None) == 0
    st = sage.SageStats()
    assert lib.sage_fd_stats(h, C.byref(st)) == 0
    launches = st.kernel_launches
    lib.sage_fd_destroy(h)
    h = _handle(lib, P=2)
    assert lib.sage_fd_update(h, 0x1000, 2 * 5 * 40, 64, None) == 0
    assert lib.sage_fd_stats(h, C.byref(st)) == 0 and st.kernel_launches == launches
    lib.sage_fd_destroy(h)


@pytest.mark.parametrize("what", ["cudaEventRecord", "cudaStreamWaitEvent", "cudaLaunchKernelExC"])
@pytest.mark.parametrize("nth", range(1, 9))
def test_no_row_of_a_failed_update_is_read_later(lib, what, nth):
    """Whichever call of the runtime fails during an update of the merged form, the rows that it held back for a joint append are
    either appended by that call or forgotten: after a reset, an update appends its own rows only."""
    h = _handle(lib, P=4)
    assert lib.sage_fd_update(h, 0x1000, 7, 64, None) == 0
    _appends(lib)
    lib.fake_fail(what.encode(), nth)
    rc = lib.sage_fd_update(h, 0x100000, 18, 64, None)
    lib.fake_fail(what.encode(), 1 << 30)
    first = _appends(lib)
    lib.sage_fd_join(h, None)
    assert lib.sage_fd_reset(h) == 0
    assert lib.sage_fd_update(h, 0x900000, 40, 64, None) == 0
    later = _appends(lib)
    assert later and all(0x900000 <= a[0] < 0x900000 + 40 * 256 and (a[3] == 0 or 0x900000 <= a[2] < 0x900000 + 40 * 256) for a in later), later
    assert sum(a[1] + a[3] for a in later) == 40
    assert rc in (0, 4) and all(0x100000 <= a[0] < 0x100000 + 18 * 256 for a in first)
    lib.sage_fd_destroy(h)


def test_options_that_no_cycle_holds_leave_its_graphs_alone(lib):
    """Only an option that changes a cycle's launches costs the graphs and the wait for the device that goes with it; a call that is
    refused changes nothing."""
    h = _handle(lib, P=2)
    assert lib.sage_fd_update(h, 0x1000, 400, 64, None) == 0
    for key, value, status in ((3, 0, 0), (5, 1, 0), (5, 0, 0), (9, 0, 0), (8, 1, 0), (8, 0, 0), (4, 1, 0), (1, 3, 2), (6, 3, 2), (77, 1, 2)):
        n0, i0 = _calls(lib, "cudaDeviceSynchronize"), _calls(lib, "cudaGraphInstantiate")
        assert lib.sage_fd_set_option(h, key, value) == status
        assert lib.sage_fd_update(h, 0x1000, 100, 64, None) == 0
        assert _calls(lib, "cudaDeviceSynchronize") == n0 and _calls(lib, "cudaGraphInstantiate") == i0, key
    for key, value in ((4, 0), (4, 1)):
        d0 = _calls(lib, "cudaGraphExecDestroy")
        assert lib.sage_fd_set_option(h, key, value) == 0 and _calls(lib, "cudaGraphExecDestroy") > d0
        assert lib.sage_fd_update(h, 0x1000, 400, 64, None) == 0
    assert lib.sage_fd_reset(h) == 0
    d0 = _calls(lib, "cudaGraphExecDestroy")
    assert lib.sage_fd_set_option(h, 1, 3) == 0 and _calls(lib, "cudaGraphExecDestroy") > d0
    lib.sage_fd_destroy(h)


def test_a_checkpoint_with_another_rank_costs_the_graphs(lib):
    a, b = _handle(lib, P=2), _handle(lib, P=2)
    lib.sage_fd_set_option(a, 1, 3)
    assert lib.sage_fd_update(a, 0x1000, 10, 64, None) == 0 and lib.sage_fd_update(b, 0x1000, 400, 64, None) == 0
    need = C.c_size_t()
    lib.sage_fd_export_size(a, C.byref(need))
    blob = C.create_string_buffer(need.value)
    assert lib.sage_fd_export(a, blob, need.value, None) == 0
    d0 = _calls(lib, "cudaGraphExecDestroy")
    assert lib.sage_fd_import(b, blob, need.value, None) == 0 and _calls(lib, "cudaGraphExecDestroy") > d0
    lib.sage_fd_destroy(a)
    lib.sage_fd_destroy(b)


def test_launchers_do_not_throw(lib):
    """Below the entry points of the C ABI nothing that the launchers keep books with may throw where host memory is short. In a
    process of its own, which an exception out of the library would end."""
    code = f"import ctypes; L = ctypes.CDLL({lib._name!r}); print('status', L.fake_allow_smem_without_memory())"
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "status 0", r.stderr[-500:]


def test_a_kernel_compiled_with_other_registers_is_an_error(lib):
    """Kernels that move registers between warps run with the count they were written for only. Another count is an error of its own,
    not the "not supported" for which callers quietly take the CUDA-core kernels."""
    assert lib.fake_allow_smem(64) == 0 and lib.fake_allow_smem(0) == 0
    assert lib.fake_allow_smem(63) == 200            # cudaErrorInvalidKernelImage; cudaErrorNotSupported is 801
