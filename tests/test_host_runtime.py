"""Host paths of the library without a GPU: its object files linked against tests/host_runtime/fake_runtime.cpp, where
kernels do nothing, device memory is host memory and calls fail when asked to."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

import simgen
from paper_1105_2791_gb300 import binding as B
from paper_1105_2791_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host_library(tmp_path_factory):
    build.build()
    out = str(tmp_path_factory.mktemp("host") / "libmodal_host.so")
    cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + os.path.join(cuda, "include"),
                    "-I" + build.CSRC, os.path.join(HERE, "host_runtime", "fake_runtime.cpp")] +
                   sorted(glob.glob(os.path.join(build.BUILD, "*.o"))) + ["-o", out], check=True)
    return out


@pytest.fixture
def lib(host_library, monkeypatch):
    monkeypatch.setattr(B, "_LIB", None)
    monkeypatch.setattr(B, "library_path", lambda: host_library)
    lib = B.load_library()
    for name in ("fake_pending", "fake_live"):
        getattr(lib, name).restype = ctypes.c_longlong
    yield lib
    lib.fake_fail_alloc(0)
    lib.fake_fail_copy(0)


def _plan(prec, L=8, P=3):
    return B.modal_init(L, P, simgen.shifted_legendre_basis(L, P), simgen.cl_model(L), L + 1, 32, prec)


@pytest.mark.parametrize("prec", ["fp32", "fp16x3", "3xtf32"])
def test_state_loads_into_a_plan_without_workspace(lib, prec, tmp_path):
    """A plan that a failed set_chunk left without workspace takes finalised means from a file, holds no temporaries
    afterwards and uses them once it has a workspace again."""
    h = _plan(prec)
    buf = np.zeros(1 << 16)
    B.modal_linear_term(h, buf.ctypes.data, 4, True, stream=0)
    path = str(tmp_path / "state")
    B.modal_save_state(h, path)
    lib.fake_fail_alloc(1)
    with pytest.raises(B.ModalError) as e:
        B.modal_set_chunk(h, 16)
    assert e.value.status == B.MODAL_ENOMEM and B.modal_get_info(h).chunk == 0
    lib.fake_fail_alloc(0)
    B.modal_load_state(h, path)
    info = B.modal_get_info(h)
    assert info.lin_final == 1 and info.n_lin == 4 and lib.fake_live() == 0
    with pytest.raises(B.ModalError) as e:
        B.modal_cubic(h, buf.ctypes.data, 1, True, buf.ctypes.data, stream=0)
    assert e.value.status == B.MODAL_ESTATE
    B.modal_set_chunk(h, 2)
    B.modal_cubic(h, buf.ctypes.data, 1, True, buf.ctypes.data, stream=0)
    B.modal_destroy(h)


@pytest.mark.parametrize("maps", [2, 300])                  # the plan's own workspace; one allocated for the call
@pytest.mark.parametrize("call,copies", [("solve", 3), ("weights", 2)])
def test_failed_solve_leaves_nothing_running(lib, call, copies, maps):
    """Whichever copy of a solve fails, what it queued before has ended when the error is returned: the next call, on any
    stream, may use the same workspace."""
    h = _plan("fp32")
    n = B.modal_get_info(h).n_max
    buf = np.zeros(1 << 16)
    B.modal_cov_accumulate(h, buf.ctypes.data, 3, stream=0)
    for k in range(1, copies + 1):
        lib.fake_fail_copy(k)
        with pytest.raises(B.ModalError) as e:
            if call == "solve":
                B.modal_solve(h, np.ones(n), buf.ctypes.data, maps, stream=0)
            else:
                B.modal_fnl_weights(h, np.ones(n), buf.ctypes.data, stream=0)
        assert e.value.status == B.MODAL_ECUDA
        assert lib.fake_pending() == 0 and lib.fake_live() == 0
    B.modal_destroy(h)
