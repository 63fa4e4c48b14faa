"""A projection and an estimate run in a workspace without the share of the tensor-core digits (1024 +
64 k b bytes, b columns), by FP64 sums; a smaller workspace is refused."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dtr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr as _dtr
    return _dtr


def _share(k, b):
    return (1024 + 64 * k * b + 255) // 256 * 256


def _space(dtr, dims, k, store):
    lat = dtr.make_lattice(dims)
    rng = np.random.default_rng(k)
    V = (rng.standard_normal((lat.N, k)) + 1j * rng.standard_normal((lat.N, k))) / np.sqrt(2 * lat.N)
    return lat, dtr.defl_create(lat, V, rng.uniform(0.3, 1.5, k), prec=store)


@pytest.mark.parametrize("store", ["f64", "f32", "bf16"])
def test_projection_in_the_smaller_workspace(dtr, store):
    import torch
    k, nrhs = 40, 16
    lat, D = _space(dtr, (8, 8, 4, 4), k, store)
    z = torch.randn(nrhs, lat.N, dtype=torch.complex128, device="cuda")
    want = dtr.deflate_project(D, z, want_coeff=True, want_x0=True)
    got = [torch.zeros_like(t) for t in want]
    nbytes = dtr._lib.dtr_deflate_workspace_bytes(D._h, nrhs) - _share(k, nrhs)
    w = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

    def project(size):
        return dtr._lib.dtr_deflate_project(D._h, dtr._ptr(z), nrhs, *(dtr._ptr(t) for t in got), dtr._ptr(w), size,
                                            dtr._stream())
    assert project(nbytes - 256) == dtr.DTR_ENOMEM
    assert project(nbytes) == dtr.DTR_OK, dtr._lib.dtr_last_error()
    for a, b in zip(got, want):   # both within n 2^-53 of sums of moduli, which are below sqrt(n) of the values' norm
        assert float((a - b).norm() / b.norm()) <= 1e-12


@pytest.mark.parametrize("lanes", [1, 2])
def test_estimate_in_the_smaller_workspace(dtr, lanes):
    import torch
    dims, k, block = (4, 4, 4, 8), 33, 8
    lat, D = _space(dtr, dims, k, "f32")
    g = dtr.make_gauge(lat, 0.5, 3)
    p = dtr.trace_params(seed=5, n_z0=32, block=block, lanes=lanes, solve=dtr.solve_params(solver="mixed_f32"))
    ws = dtr.TraceWorkspace(g, D, p)
    want = dtr.trace_estimate(g, -0.4, D, p, workspace=ws)
    ws.nbytes -= lanes * _share(k, block)
    ws.buf = torch.empty(ws.nbytes, dtype=torch.uint8, device="cuda")
    got = dtr.trace_estimate(g, -0.4, D, p, workspace=ws)
    assert np.abs(got["samples"] - want["samples"]).max() <= 1e-11 * np.abs(want["samples"]).max()
