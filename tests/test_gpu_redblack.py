"""Mixed solves on the red-black Schur complement at the shapes where its indexing can go wrong: the smallest
lattice, extents of 2 (both neighbours are one site), uneven extents, one column (padded to a pair), block widths
that are no power of two and the widest block, and a negative diagonal.  The residual is recomputed by the oracle
in FP64 on the whole lattice, so a wrong neighbour, link or odd-site reconstruction shows as a residual of order
one; the bound is the solver's own tolerance."""
import numpy as np
import pytest

from oracle import wilson
from paper_1603_05988_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dtr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1603_05988_gb300 import dtr as m
    return m


@pytest.mark.parametrize("solver", ["mixed_f32", "mixed_f16", "mixed_bf16"])
@pytest.mark.parametrize("dims,nrhs,m0", [((2, 2, 2, 2), 1, -0.4), ((2, 6, 4, 10), 3, -0.6), ((6, 2, 2, 4), 64, -0.4),
                                          ((12, 10, 6, 14), 7, -0.75), ((4, 4, 4, 4), 33, 1.0),
                                          ((10, 4, 2, 6), 2, -8.6)])
def test_redblack_solve_meets_tolerance(dtr, solver, dims, nrhs, m0):
    import torch
    U = synth.random_su3_links(dims, 0.7, 21)
    lat = dtr.make_lattice(dims)
    g = dtr.gauge_from_host(lat, U)
    rng = np.random.default_rng(4)
    Z = rng.standard_normal((nrhs, lat.N)) + 1j * rng.standard_normal((nrhs, lat.N))
    if nrhs > 2:
        Z[1] *= 1e-3      # columns of other scales, and one without any red (even) site
        x = np.arange(lat.V)
        par = (x % dims[0] + x // dims[0] % dims[1] + x // (dims[0] * dims[1]) % dims[2]
               + x // (dims[0] * dims[1] * dims[2])) & 1
        Z[2] *= np.repeat(par, 12)
    y, st = dtr.solve_batch(g, m0, torch.from_numpy(Z).cuda(), params=dtr.solve_params(tol=1e-10, solver=solver))
    Y = y.cpu().numpy().T
    res = np.linalg.norm(Z.T - wilson.apply(U, dims, m0, Y), axis=0) / np.linalg.norm(Z, axis=1)
    assert all(s["converged"] for s in st)
    assert res.max() <= 1.001e-10, res.max()
