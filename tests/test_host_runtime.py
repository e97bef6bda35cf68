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
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
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


# the last size of one launch, one past it, 2^31 pixels, and far more than 2^32 in several parts per map
@pytest.mark.parametrize("npix,ctas", [(1 << 20, 128), ((1 << 31) - 16, 152), (1 << 31, 152), (300000 * 8192, 152), (9 << 31, 152), (3 << 29, 2)])
@pytest.mark.parametrize("maps,P", [(1, 3), (3, 2)])
def test_cubic_launches_cover_maps_of_any_size(lib, npix, ctas, maps, P):
    """The tiled copies take 32-bit pixel coordinates: whatever the number of pixels, each pixel range of each map is
    one launch's, at the addresses and with the partial sums of the whole, and no coordinate reaches 2^31."""
    A, W, S, n_max = 1 << 40, 1 << 50, 1 << 56, P * (P + 1) * (P + 2) // 6
    out = (ctypes.c_longlong * 12000)()
    lib.fake_cubic.argtypes = [ctypes.c_longlong] + [ctypes.c_int] * 3 + [ctypes.c_longlong] * 3 + [ctypes.c_void_p, ctypes.c_int]
    n = lib.fake_cubic(npix, P, maps, ctas, A, W, S, out, len(out))
    assert 1 <= n <= 1000
    whole = (-(-npix // ctas) + 127) // 128 * 128           # pixels of a range
    seen = set()
    for k in range(n):
        base, cols, rows, pitch, wbase, wcols, partial, px, ppc, nctas, nunits, grid = out[12 * k:12 * k + 12]
        assert ppc == whole and pitch == 4 * npix and cols == wcols == px and rows == P * (nunits // nctas)
        assert px + ppc < 1 << 31 and nunits % nctas == 0 and grid == (nunits + 1) // 2
        for u in range(nunits):
            slot = (partial - S) // 8 // n_max + u
            b, r = divmod(slot, ctas)
            at = u // nctas * P * npix * 4 + u % nctas * ppc * 4   # where the launch reads unit u, from its maps
            if r * whole < npix:
                assert base + at == A + (b * P * npix + r * whole) * 4
                assert wbase + u % nctas * ppc * 4 == W + r * whole * 4
                assert min(px, (u % nctas + 1) * ppc) - u % nctas * ppc == min(npix, (r + 1) * whole) - r * whole
            assert slot not in seen
            seen.add(slot)
    assert seen == set(range(maps * ctas))
