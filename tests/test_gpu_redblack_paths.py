"""Paths of the solvers beside the mixed red-black one from a zero guess: the plain FP64 red-black solver at the shapes
where its indexing can go wrong (the smallest lattice, extents of 2, uneven extents, one column, widths that are no power
of two, a negative diagonal); start vectors that are not zero, one column of them zero, one already the solution, one far
off; and the whole-lattice solvers, which take over where the diagonal is too small for the red-black ones
(|4 + m0| < 1/2, near the free field on 2^4, where a Krylov method still converges).  The oracle recomputes the residual on
the whole lattice; the bound is the solver's own tolerance."""
import numpy as np
import pytest

from oracle import wilson
from paper_1603_05988_gb300 import synth

pytestmark = pytest.mark.gpu

SOLVERS = ["f64", "mixed_f32", "mixed_f16", "mixed_bf16"]


@pytest.fixture(scope="module")
def dtr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1603_05988_gb300 import dtr as m
    return m


def _random(rng, n, N):
    return rng.standard_normal((n, N)) + 1j * rng.standard_normal((n, N))


def _check(dtr, dims, eps, m0, Z, y0, **params):
    import torch
    U = synth.random_su3_links(dims, eps, 21)
    g = dtr.gauge_from_host(dtr.make_lattice(dims), U)
    start = None if y0 is None else torch.from_numpy(y0).cuda()
    y, st = dtr.solve_batch(g, m0, torch.from_numpy(Z).cuda(), y0=start, params=dtr.solve_params(tol=1e-10, **params))
    res = np.linalg.norm(Z.T - wilson.apply(U, dims, m0, y.cpu().numpy().T), axis=0) / np.linalg.norm(Z, axis=1)
    assert all(s["converged"] for s in st)
    assert res.max() <= 1.001e-10, res.max()
    return st


@pytest.mark.parametrize("dims,nrhs,m0", [((2, 2, 2, 2), 1, -0.4), ((2, 6, 4, 10), 3, -0.6), ((6, 2, 2, 4), 64, -0.4),
                                          ((12, 10, 6, 14), 7, -0.75), ((4, 4, 4, 4), 33, 1.0),
                                          ((10, 4, 2, 6), 2, -8.6)])
def test_fp64_redblack_shapes(dtr, dims, nrhs, m0):
    rng = np.random.default_rng(4)
    V = int(np.prod(dims))
    Z = _random(rng, nrhs, 12 * V)
    if nrhs > 2:
        x = np.arange(V)
        par = (x % dims[0] + x // dims[0] % dims[1] + x // (dims[0] * dims[1]) % dims[2]
               + x // (dims[0] * dims[1] * dims[2])) & 1
        Z[1] *= 1e-3
        Z[2] *= np.repeat(par, 12)
    _check(dtr, dims, 0.7, m0, Z, None, solver="f64")


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("solver", SOLVERS)
@pytest.mark.parametrize("dims,nrhs", [((2, 6, 4, 10), 5), ((4, 4, 4, 4), 1), ((6, 4, 4, 2), 33)])
def test_nonzero_start_vectors(dtr, solver, graph, dims, nrhs):
    import torch
    rng = np.random.default_rng(nrhs)
    N, m0 = 12 * int(np.prod(dims)), -0.6
    Z = _random(rng, nrhs, N)
    y0 = 0.3 * _random(rng, nrhs, N)
    if nrhs > 3:
        g = dtr.gauge_from_host(dtr.make_lattice(dims), synth.random_su3_links(dims, 0.7, 21))
        tight = dtr.solve_params(tol=1e-12, solver="f64")
        y0[0] = 0.0
        y0[1] = dtr.solve_batch(g, m0, torch.from_numpy(Z[1:2].copy()).cuda(), params=tight)[0].cpu().numpy()
        y0[3] *= 1e4
    st = _check(dtr, dims, 0.7, m0, Z, y0, solver=solver, graph=graph)
    if nrhs > 3:
        assert st[1]["iterations"] == 0 and st[0]["iterations"] > 0


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("solver", SOLVERS)
@pytest.mark.parametrize("nrhs,m0", [(1, -3.55), (5, -4.4)])
def test_small_diagonal_takes_the_whole_lattice(dtr, solver, graph, nrhs, m0):
    Z = _random(np.random.default_rng(8), nrhs, 192)
    _check(dtr, (2, 2, 2, 2), 0.02, m0, Z, None, solver=solver, graph=graph)
    _check(dtr, (2, 2, 2, 2), 0.02, m0, Z, 0.3 * Z, solver=solver, graph=graph)
