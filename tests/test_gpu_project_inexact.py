"""Deflated solutions of FP32 and BF16 spaces whose entries have more bits than their column's integers hold: one broad
vector beside vectors that decay by 14 decades, so that over most of the lattice the solution is the broad vector's
contribution and the integers of all others have lost bits, which 16 entries of an otherwise sufficient size must not hide.

Bound: 2 k roundings of FP64 sums, each at most 2^-53 of the sum of moduli S, of RMS 1 / sqrt(3) of that and of independent
sign: 3 sqrt(2 k / 3) 2^-53 times the norm of S over 16 entries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("dims,k,nrhs", [((8, 8, 8, 8), 40, 16), ((8, 8, 4, 8), 33, 17)])
def test_entries_that_lose_bits(store, dims, k, nrhs):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1603_05988_gb300 import dtr
    lat = dtr.make_lattice(dims)
    n = lat.N
    rng = np.random.default_rng(k)
    t = np.arange(n)[:, None] / n
    V = rng.standard_normal((n, k)) + 1j * rng.standard_normal((n, k))
    V[:, :1] *= 8.0 ** -t
    V[:, 1:] *= 10.0 ** (-14 * t)
    lam = rng.uniform(0.8, 1.2, k)
    Z = np.array([1, 1j, -1, -1j])[rng.integers(0, 4, (nrhs, n))]
    D = dtr.defl_create(lat, V, lam, prec=store)
    Vs, _ = D.to_host()
    _, C, x0 = dtr.deflate_project(D, torch.from_numpy(Z).cuda(), want_coeff=True, want_x0=True)
    j = np.arange(0, nrhs, 5)
    W = C.cpu().numpy().T[:, nrhs + j] * (1.0 / lam)[:, None]
    i = (np.arange(0, n // 16, 7)[:, None] * 16 + np.arange(16)).ravel()
    ld = lambda a: np.asarray(a, np.longdouble)  # noqa: E731
    vr, vi, wr, wi = ld(Vs[i].real), ld(Vs[i].imag), ld(W.real), ld(W.imag)
    got = x0.cpu().numpy().T[np.ix_(i, j)]
    err = np.hypot((got.real - (vr @ wr - vi @ wi)).astype(float), (got.imag - (vr @ wi + vi @ wr)).astype(float))
    S = np.abs(Vs[i]) @ np.abs(W)
    norm = lambda a: np.sqrt((a.reshape(-1, 16, len(j)) ** 2).sum(axis=1))  # noqa: E731
    ratio = norm(err) / (2.0 ** -53 * norm(S))
    assert ratio.max() <= 3 * np.sqrt(2 * k / 3), (ratio.max(), 3 * np.sqrt(2 * k / 3))
