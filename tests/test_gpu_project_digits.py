"""Deflation projection of general FP64 blocks by exact integer digits on the tensor cores, against extended-precision
sums, at the edges of its tiles (32 vectors, 16 columns, 8 sites) and of its number range: columns of very different
scales, a zero column, probing noise (one digit), entries that the integers cannot hold (not finite, or a column below
2^-800), which the FP64 kernel takes, and sizes on the FP64 side of the rules.

Bounds, for entries below 2^ev and 2^ez: an entry is rounded by at most 2^-55 of its column's power of two, and the
dropped digit pairs are below 2^-59 of the product of the two powers; with a power of two at most twice the column's
largest entry and two real products to each part, n terms are off by at most n 2^-51 max|v| max|z|."""
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
    """A^T B of complex arrays in extended precision (A: n x p, B: n x q) -> p x q, as (re, im)."""
    ar, ai, br, bi = _ld(A.real), _ld(A.imag), _ld(B.real), _ld(B.imag)
    return ar.T @ br - ai.T @ bi, ar.T @ bi + ai.T @ br


@pytest.mark.parametrize("store", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("dims,k,nrhs,kind", [((2, 2, 2, 2), 1, 1, "normal"), ((4, 2, 2, 6), 31, 3, "scales"),
                                              ((8, 4, 4, 4), 33, 17, "z4"), ((4, 4, 4, 8), 65, 64, "normal"),
                                              ((8, 8, 4, 4), 32, 16, "scales"), ((8, 8, 4, 4), 31, 16, "tiny"),
                                              ((8, 4, 4, 8), 40, 12, "nan")])
def test_projection_digits(dtr, store, dims, k, nrhs, kind):
    import torch
    lat = dtr.make_lattice(dims)
    rng = np.random.default_rng(k)
    V = (rng.standard_normal((lat.N, k)) + 1j * rng.standard_normal((lat.N, k))) / np.sqrt(2 * lat.N)
    V *= 2.0 ** rng.integers(-8, 8, k)
    V *= 10.0 ** rng.uniform(-3, 0, (lat.N, 1))   # entries of one column over several orders
    lam = rng.uniform(0.3, 1.5, k) * rng.choice((-1, 1), k)
    if kind == "z4":
        Z = np.array([1, 1j, -1, -1j])[rng.integers(0, 4, (nrhs, lat.N))]
    else:
        Z = rng.standard_normal((nrhs, lat.N)) + 1j * rng.standard_normal((nrhs, lat.N))
    if kind == "scales":
        Z *= 10.0 ** np.linspace(-200, 150, nrhs)[:, None]
        Z[1] = 0.0
    if kind == "tiny":
        Z[2] *= 1e-260
    if kind == "nan":
        Z[3, 7] = np.nan
        Z[0, 5] = np.inf
    D = dtr.defl_create(lat, V, lam, prec=store)
    Vs, _ = D.to_host()
    d, C, x0 = dtr.deflate_project(D, torch.from_numpy(np.ascontiguousarray(Z)).cuda(), want_coeff=True, want_x0=True)
    C, x0 = C.cpu().numpy().T, x0.cpu().numpy().T          # k x 2 nrhs, N x nrhs
    g5 = np.tile(np.array([1.0] * 6 + [-1.0] * 6), lat.N // 12)
    bad = ~np.isfinite(Z).all(axis=1)
    assert not np.isfinite(C[:, :nrhs][:, bad]).all() if bad.any() else True
    ok = np.flatnonzero(~bad)
    Zt = Z[ok].T
    B = np.concatenate([Zt, g5[:, None] * Zt], axis=1)
    re, im = _mm(np.conj(Vs), B)
    cols = np.concatenate([ok, nrhs + ok])
    vmax, zmax = np.abs(Vs).max(axis=0), np.abs(B).max(axis=0)
    bound = lat.N * 2.0 ** -51 * vmax[:, None] * zmax[None, :] * 2
    err = np.hypot((C.real[:, cols] - re).astype(float), (C.imag[:, cols] - im).astype(float))
    assert np.all(err <= bound), (err / np.where(bound > 0, bound, 1)).max()
    W = C[:, nrhs + ok] / lam[:, None]                      # the weights that the library expands
    xr, xi = _mm(Vs.T, W)
    wmax = (np.abs(W) * vmax[:, None]).max(axis=0)
    err = np.hypot((x0.real[:, ok] - xr).astype(float), (x0.imag[:, ok] - xi).astype(float))
    assert np.all(err <= (k + 4) * 2.0 ** -50 * wmax[None, :]), (err.max(axis=0) / np.where(wmax > 0, wmax, 1))
