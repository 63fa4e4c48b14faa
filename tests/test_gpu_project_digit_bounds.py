"""Deflation projection of plain blocks (Gaussian and Z4) to the accuracy that the integer digits are meant to have, tight
enough that a missing or misplaced digit plane shows: without the products of the lowest weight kept the errors are ten
times larger.

Bounds, six standard deviations.  An entry below 2^e is rounded to a multiple of 2^(e - 54): 2^-55 / sqrt(3) RMS of 2^e,
against the moduli it is multiplied with.  The digit pairs dropped, five of the next lower weight with digits of RMS 74, in
units of 256^4 2^-108, come to 2^-62.  The FP64 sums of at most V / 16 chunks (C) round by at most 2^-53 / sqrt(3) RMS of a
running sum, in mean square over the chunks half of the last: 2^-53 / sqrt(3) sqrt(V / 32) of it, and of two sums (the
halves of the spins) of variance sum |v|^2 |z|^2 / 4 in each part; a value itself by 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _ld(a):
    return np.asarray(a, np.longdouble)


def _mm(A, B):
    ar, ai, br, bi = _ld(A.real), _ld(A.imag), _ld(B.real), _ld(B.imag)
    return ar.T @ br - ai.T @ bi, ar.T @ bi + ai.T @ br


def _pow2(a):
    """2^e above the largest real or imaginary part of every column."""
    return 2.0 ** np.frexp(np.maximum(np.abs(a.real), np.abs(a.imag)).max(axis=0))[1]


@pytest.mark.parametrize("store", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("dims,k,nrhs,kind", [((8, 8, 4, 4), 64, 16, "normal"), ((8, 8, 8, 6), 33, 17, "normal"),
                                              ((8, 8, 4, 4), 40, 12, "z4"), ((12, 10, 6, 14), 96, 16, "normal")])
def test_projection_is_as_accurate_as_its_digits(store, dims, k, nrhs, kind):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat = dtr.make_lattice(dims)
    n = lat.N
    rng = np.random.default_rng(k)
    V = (rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))) / np.sqrt(2 * n)
    lam = rng.uniform(0.3, 1.5, k) * rng.choice((-1, 1), k)
    if kind == "z4":
        Z = np.array([1, 1j, -1, -1j])[rng.integers(0, 4, (nrhs, n))]
    else:
        Z = rng.standard_normal((nrhs, n)) + 1j * rng.standard_normal((nrhs, n))
    D = dtr.defl_create(lat, V, lam, prec=store)
    Vs, _ = D.to_host()
    _, C, x0 = dtr.deflate_project(D, torch.from_numpy(Z).cuda(), want_coeff=True, want_x0=True)
    C, x0 = C.cpu().numpy().T, x0.cpu().numpy().T
    g5 = np.tile(np.array([1.0] * 6 + [-1.0] * 6), n // 12)
    B = np.concatenate([Z.T, g5[:, None] * Z.T], axis=1)
    pv, pz = _pow2(Vs), _pow2(B)
    m, j = rng.choice(k, 12, replace=False), rng.choice(2 * nrhs, 10, replace=False)   # a sample of C: long doubles are slow
    re, im = _mm(np.conj(Vs[:, m]), B[:, j])
    Vm, Bj, Cmj = Vs[:, m], B[:, j], C[np.ix_(m, j)]
    v2, z2 = (np.abs(Vm) ** 2).sum(axis=0), (np.abs(Bj) ** 2).sum(axis=0)
    rnd = 2.0 ** -55 / np.sqrt(3) * np.sqrt(pv[m, None] ** 2 * z2[None, :] + v2[:, None] * pz[None, j] ** 2)
    drop = 2.0 ** -62 * np.sqrt(2 * n) * pv[m, None] * pz[None, j]
    run = 2.0 ** -53 / np.sqrt(3) * np.sqrt(lat.V / 32) * np.sqrt((np.abs(Vm) ** 2).T @ (np.abs(Bj) ** 2) / 2)
    bound = 6 * np.sqrt(rnd ** 2 + drop ** 2 + run ** 2) + 2.0 ** -52 * np.abs(Cmj)
    for got, want in ((Cmj.real, re), (Cmj.imag, im)):
        ratio = np.abs((got - want).astype(float)) / bound
        assert ratio.max() <= 1, ratio.max()
    W = C[:, nrhs:] * (1.0 / lam)[:, None]                   # the weights that the library expands
    i, j = rng.choice(n, 3000, replace=False), rng.choice(nrhs, 3, replace=False)
    W, Vi, x0 = W[:, j], Vs[i], x0[np.ix_(i, j)]
    xr, xi = _mm(Vi.T, W)
    pw = _pow2(W * pv[:, None])                              # of W times the vectors' powers of two
    w2 = (np.abs(W * pv[:, None]) ** 2).sum(axis=0)
    r2 = (np.abs(Vi / pv[None, :]) ** 2).sum(axis=1)
    rnd = 2.0 ** -55 / np.sqrt(3) * np.sqrt(w2[None, :] + r2[:, None] * pw[None, :] ** 2)
    bound = 6 * np.sqrt(rnd ** 2 + (2.0 ** -62 * np.sqrt(2 * k) * pw[None, :]) ** 2) + 2.0 ** -52 * np.abs(x0)
    for got, want in ((x0.real, xr), (x0.imag, xi)):
        ratio = np.abs((got - want).astype(float)) / bound
        assert ratio.max() <= 1, ratio.max()
