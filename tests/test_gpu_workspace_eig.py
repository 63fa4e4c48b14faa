"""The FP64 setup eigensolver runs in a workspace that holds as many partial Gram products as 64-wide tiles and runs of 4096
dofs need, fewer than it asks for, and finds the same pairs; a smaller workspace is refused."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _chunks(tile, run, least, p, n, sms):
    tiles = (-(-p // tile)) ** 2
    nk = max(-(-4 * sms // tiles), least)
    return max(min(nk, max(n // run, 1)), 1)


@pytest.mark.parametrize("dims,k", [((4, 4, 4, 8), 20), ((8, 8, 8, 8), 64)])
def test_fp64_eigensolver_in_the_smaller_workspace(dims, k):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat = dtr.make_lattice(dims)
    g = dtr.make_gauge(lat, 0.7, 3)
    P = dtr.eig_params(k, store="f64", degree=32, max_iter=40, tol=1e-4)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = (k + max(k // 8, 16) + 15) // 16 * 16
    full = dtr._lib.dtr_eig_workspace_bytes(lat._h, ctypes.byref(P))
    more = _chunks(16, 256, 8, p, lat.N, sms) - _chunks(64, 4096, 1, p, lat.N, sms)
    assert more > 0
    nbytes = full - more * p * p * 16
    w = torch.empty(full, dtype=torch.uint8, device="cuda")

    def solve(size):
        res, st, h = np.zeros(k), dtr.EigStats(), ctypes.c_void_p()
        rc = dtr._lib.dtr_eig_deflation(g._h, -0.6, ctypes.byref(P), dtr._ptr(w), size, res.ctypes.data_as(ctypes.c_void_p),
                                        ctypes.byref(st), ctypes.byref(h), dtr._stream())
        return rc, (dtr.Deflation(lat, None, None, handle=h, k=k).lambdas() if rc == dtr.DTR_OK else None)
    assert solve(nbytes - 256)[0] == dtr.DTR_ENOMEM
    rc, want = solve(full)
    assert rc == dtr.DTR_OK
    rc, got = solve(nbytes)
    assert rc == dtr.DTR_OK, dtr._lib.dtr_last_error()
    # residuals of 1e-4 |lambda| bound each value's error by 1e-4 |lambda|
    assert np.abs(np.sort(got) - np.sort(want)).max() <= 2e-4 * np.abs(want).max()
