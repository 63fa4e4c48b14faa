"""A mixed solve or estimate of single columns runs in the workspace of the whole-lattice solver (an FP64 vector and
seven FP32 ones beyond the fixed part), although the red-black solver, which pads the column to a pair, takes more and
the size query says so; a smaller workspace is refused."""
import ctypes

import numpy as np
import pytest

from paper_1603_05988_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dtr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1603_05988_gb300 import dtr as m
    return m


def _al(n):
    return (n + 255) // 256 * 256


def _extra(V):
    """What 12 padded half-lattice vectors take beyond an FP64 and seven FP32 vectors."""
    return 12 * _al(V // 2 * 12 * 2 * 8) - _al(12 * V * 16) - 7 * _al(12 * V * 8)


@pytest.mark.parametrize("solver", ["mixed_f32", "mixed_f16", "mixed_bf16"])
@pytest.mark.parametrize("graph", [True, False])
def test_single_column_solve_in_the_smaller_workspace(dtr, solver, graph):
    import torch
    dims, m0 = (4, 6, 4, 8), -0.6
    lat = dtr.make_lattice(dims)
    g = dtr.gauge_from_host(lat, synth.random_su3_links(dims, 0.7, 21))
    p = dtr.solve_params(tol=1e-10, solver=solver, graph=graph)
    z = torch.randn(1, lat.N, dtype=torch.complex128, device="cuda")
    y = torch.zeros_like(z)
    full = dtr._lib.dtr_solve_workspace_bytes(lat._h, 1, ctypes.byref(p))
    nbytes = full - _extra(lat.V)
    assert nbytes < full
    w = torch.empty(nbytes, dtype=torch.uint8, device="cuda")

    def solve(size):
        return dtr._lib.dtr_solve_batch(g._h, m0, dtr._ptr(z), dtr._ptr(y), 1, ctypes.byref(p), dtr._ptr(w), size, None,
                                        dtr._stream())
    assert solve(nbytes - 512) == dtr.DTR_ENOMEM
    assert solve(nbytes) == dtr.DTR_OK, dtr._lib.dtr_last_error()
    assert float((z - dtr.dslash(g, m0, y)).norm() / z.norm()) <= 1.001e-10


@pytest.mark.parametrize("lanes", [1, 2])
def test_single_column_estimate_in_the_smaller_workspace(dtr, lanes):
    import torch
    dims, m0 = (4, 4, 4, 4), -0.4
    lat = dtr.make_lattice(dims)
    g = dtr.gauge_from_host(lat, synth.random_su3_links(dims, 0.5, 3))
    p = dtr.trace_params(seed=5, n_z0=4, block=1, lanes=lanes, solve=dtr.solve_params(solver="mixed_f32"))
    ws = dtr.TraceWorkspace(g, None, p)
    want = dtr.trace_estimate(g, m0, None, p, workspace=ws)
    ws.nbytes -= lanes * _extra(lat.V)
    ws.buf = torch.empty(ws.nbytes, dtype=torch.uint8, device="cuda")
    got = dtr.trace_estimate(g, m0, None, p, workspace=ws)
    assert got["all_converged"]
    # both meet 1e-10, so z^H y differs by at most 2e-10 ||z||^2 / sigma_min, ||z||^2 = N
    assert np.abs(got["samples"] - want["samples"]).max() <= 2e-10 * lat.N * 10
