"""An allocation that finds the device full gives the parked buffers back and tries once more: it
then succeeds where they were what was missing, and fails with FIRAL_ERR_NOMEM where they were not.
Needs a GPU."""
import ctypes
import gc

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

GIB = 1 << 30


@pytest.fixture
def lib():
    from paper_2409_07392_gb300 import _lib as L, build
    build.build()
    lib = L.load()
    gc.collect()
    lib.firal_cache_trim()
    torch.cuda.empty_cache()
    yield lib
    gc.collect()
    torch.cuda.empty_cache()
    lib.firal_cache_trim()


def pool(n, d):
    return torch.ones(n, d, device="cuda"), torch.full((n, 2), 0.5, device="cuda")


def test_parked_buffers_make_room(lib):
    from paper_2409_07392_gb300 import api
    H = api.Handle()
    X, h = pool(4 << 20, 128)
    api.Problem(H, X, h, precision="fp32").close()   # parks x's 2 GiB
    assert lib.firal_cache_bytes() >= 2 * GIB
    del X, h
    X, h = pool(6 << 20, 128)                        # x takes 3 GiB: no parked block is as large
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 2 * GIB, dtype=torch.uint8, device="cuda")
    prob = api.Problem(H, X, h, precision="fp32")    # fits in 2 GiB and the parked 2
    z = torch.full((X.shape[0],), 1e-3, device="cuda")
    g = -torch.ones_like(z)
    z = prob.md_step(z, g, 5.0)                      # no launch check reports the failed attempt
    assert abs(float(z.double().sum()) - 5.0) < 1e-3
    prob.close()
    del fill


def test_no_room_at_all(lib):
    from paper_2409_07392_gb300 import _lib as L, api
    H = api.Handle()
    X, h = pool(1 << 20, 32)
    api.Problem(H, X, h, precision="fp32").close()
    assert lib.firal_cache_bytes() > 0
    # 550 GB of x: refused before any row is read
    big = L.FiralPool(X.data_ptr(), h.data_ptr(), 1 << 30, 128, 2, 1, 1)
    out = ctypes.c_void_p()
    code = lib.firal_problem_create(H.ptr, ctypes.byref(big), None, api.PRECISIONS["fp32"],
                                    ctypes.byref(out))
    assert code != 0 and not out
    buf = ctypes.create_string_buffer(512)
    lib.firal_last_error(H.ptr, buf, 512)
    assert b"cudaMalloc" in buf.value and b"out of memory" in buf.value, buf.value
    assert lib.firal_cache_bytes() == 0              # the parked blocks went back first
    prob = api.Problem(H, X, h, precision="fp32")
    z = torch.full((X.shape[0],), 1e-3, device="cuda")
    z = prob.md_step(z, -torch.ones_like(z), 5.0)
    assert abs(float(z.double().sum()) - 5.0) < 1e-3
    prob.close()
