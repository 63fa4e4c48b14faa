"""The timing of the deflation contraction in a workspace that is not zero (it reads an error word that only the tensor-core
contraction sets), with and without the share of the digits (1024 + 64 k b bytes, b columns)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f64", "f32", "bf16"])
def test_timing_in_a_used_workspace(store):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat, k, b = dtr.make_lattice((4, 4, 4, 8)), 32, 8
    rng = np.random.default_rng(k)
    V = rng.standard_normal((lat.N, k)) + 1j * rng.standard_normal((lat.N, k))
    D = dtr.defl_create(lat, V, rng.uniform(0.3, 1.5, k), prec=store)
    nbytes = dtr._lib.dtr_time_deflate_workspace_bytes(D._h, b)
    w = torch.full((nbytes,), 255, dtype=torch.uint8, device="cuda")
    ms = ctypes.c_double()
    for size in (nbytes, nbytes - (1024 + 64 * k * b + 255) // 256 * 256):
        rc = dtr._lib.dtr_time_deflate(D._h, b, 2, dtr._ptr(w), size, ctypes.byref(ms), dtr._stream())
        assert rc == dtr.DTR_OK, dtr._lib.dtr_last_error()
        assert ms.value > 0
