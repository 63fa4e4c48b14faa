"""Deflation projection of graded blocks: deflation vectors and right-hand sides that are small, entry by entry, where the
other is large (decaying from opposite ends of the lattice; in random order within every site), point sources, and
deflated solutions where all vectors are small.  Fixed-point digits relative to a column's largest entry lose such products,
FP64 sums do not.

Bounds: a sum of n real products carries 2 n roundings, each at most 2^-53 of the sum of moduli S and of independent
sign, so 3 sqrt(2 n) 2^-53 S for C (n = 12 V); for x0 the 2 k + 2 roundings add up, at most 2^-53 S each.  A point
source has one nonzero product, a stored entry times one: exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dtr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr as _dtr
    return _dtr


def _ld(a):
    return np.asarray(a, np.longdouble)


def _mm(A, B):
    ar, ai, br, bi = _ld(A.real), _ld(A.imag), _ld(B.real), _ld(B.imag)
    return ar.T @ br - ai.T @ bi, ar.T @ bi + ai.T @ br


@pytest.mark.parametrize("store", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("dims,k,nrhs,kind,decades",
                         [((8, 8, 4, 4), 40, 17, "opposite", 10), ((8, 8, 4, 4), 33, 16, "opposite", 16),
                          ((8, 8, 4, 4), 40, 17, "shuffled", 10), ((16, 8, 8, 12), 65, 17, "opposite", 10),
                          ((8, 8, 4, 4), 40, 12, "point", 12), ((2, 2, 2, 6), 5, 3, "opposite", 12)])
def test_projection_of_graded_blocks(dtr, store, dims, k, nrhs, kind, decades):
    import torch
    lat = dtr.make_lattice(dims)
    n = lat.N
    rng = np.random.default_rng(k + decades)
    t = rng.random(n) if kind == "shuffled" else np.arange(n) / n
    V = (rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))) * 10.0 ** (-decades * t[:, None])
    lam = rng.uniform(0.3, 1.5, k) * rng.choice((-1, 1), k)
    if kind == "point":
        at = n - 1 - rng.choice(n // 2, nrhs, replace=False)   # where V is small
        Z = np.zeros((nrhs, n), complex)
        Z[np.arange(nrhs), at] = 1.0
    else:
        Z = (rng.standard_normal((nrhs, n)) + 1j * rng.standard_normal((nrhs, n))) * 10.0 ** (-decades * (1 - t[None, :]))
    D = dtr.defl_create(lat, V, lam, prec=store)
    Vs, _ = D.to_host()
    d, C, x0 = dtr.deflate_project(D, torch.from_numpy(Z).cuda(), want_coeff=True, want_x0=True)
    C, x0 = C.cpu().numpy().T, x0.cpu().numpy().T
    g5 = np.tile(np.array([1.0] * 6 + [-1.0] * 6), n // 12)
    if kind == "point":
        assert np.array_equal(C[:, :nrhs], np.conj(Vs[at]).T)
        assert np.array_equal(C[:, nrhs:], np.conj(Vs[at]).T * g5[at][None, :])
    else:
        B = np.concatenate([Z.T, g5[:, None] * Z.T], axis=1)
        m, j = rng.choice(k, 5, replace=False), np.arange(0, 2 * nrhs, 4)   # a sample: long doubles are slow
        re, im = _mm(np.conj(Vs[:, m]), B[:, j])
        err = np.hypot((C[np.ix_(m, j)].real - re).astype(float), (C[np.ix_(m, j)].imag - im).astype(float))
        S = np.abs(Vs[:, m]).T @ np.abs(B[:, j])
        ratio = err / (2.0 ** -53 * S)
        assert ratio.max() <= 3 * np.sqrt(2 * n), (ratio.max(), 3 * np.sqrt(2 * n))
    i, j = np.arange(0, n, 5), np.arange(0, nrhs, 4)
    W = C[:, nrhs + j] * (1.0 / lam)[:, None]
    xr, xi = _mm(Vs[i].T, W)
    err = np.hypot((x0[np.ix_(i, j)].real - xr).astype(float), (x0[np.ix_(i, j)].imag - xi).astype(float))
    S = np.abs(Vs[i]) @ np.abs(W)
    ratio = err / (2.0 ** -53 * np.where(S > 0, S, 1))
    assert ratio.max() <= 2 * (2 * k + 2), ratio.max()
