"""The work that users of the library have it do, as cases that can be timed and compared.

Every case goes through the binding's public calls (paper_1603_05988_gb300.dtr) on inputs of the kind the
library is built for: random SU(3) links U = exp(i eps H) at the workloads' (eps, m0) = (0.5, -0.4),
(0.7, -0.6), (0.8, -0.75), (0.8, -0.78), Z4 noise right-hand sides, solves to the default tolerance 1e-10.

  listed()            the cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs and handles a program holds before the call
  run(state)          one pass: the call and its outputs
  work(case)          bytes and flops the pass cannot do without
  exact(case, seed)   the outputs in 64 bits by plain torch and numpy

Kinds: "dslash" (the operator alone), "project" (deflation projection), "solve" (A y = z for a block), "trace"
(the whole estimator), "net" (a training step of the learned preconditioner), "eig" (the setup eigensolver).
"""
import math

import numpy as np
import torch

from paper_1603_05988_gb300 import dtr

# (eps, m0) of the library's workloads, by lattice size from the smallest up
FIELDS = ((0.5, -0.4), (0.7, -0.6), (0.8, -0.75), (0.8, -0.78))
FLOPS_DSLASH = 1368.0  # per site and right-hand side
# operator applications that a Krylov method needs for the ten digits of a solve on these fields (condition
# numbers 7 to 11, red-black ordering used)
APPLICATIONS = 24


def listed():
    return [
        # the smallest call: one stencil on one field, FP64; a correctness check or a user's own iteration
        dict(name="dslash_f64_4x4x4x4", kind="dslash", lx=4, ly=4, lz=4, lt=4, nrhs=1, prec="f64", dagger=False,
             eps=0.5, m0=-0.4),
        # the stencil on a block of fields in single precision, A^H as a user's normal equations need it
        dict(name="dslash_f32_16x16x16x32_r16", kind="dslash", lx=16, ly=16, lz=16, lt=32, nrhs=16, prec="f32",
             dagger=True, eps=0.8, m0=-0.75),
        # the half-storage stencil on one field of the headline lattice
        dict(name="dslash_bf16_32x32x32x64", kind="dslash", lx=32, ly=32, lz=32, lt=64, nrhs=1, prec="bf16",
             dagger=False, eps=0.8, m0=-0.78),
        # deflation projection of a block, with the deflated solution as a start vector
        dict(name="project_f32_16x16x16x32_k64", kind="project", lx=16, ly=16, lz=16, lt=32, nrhs=16, k=64,
             store="f32", x0=True),
        # a small block of solves: the 8^4 workload's block, latency-bound
        dict(name="solve_f32_8x8x8x8_r16", kind="solve", lx=8, ly=8, lz=8, lt=8, nrhs=16, solver="mixed_f32",
             eps=0.7, m0=-0.6),
        # an uneven lattice and a block that is no power of two
        dict(name="solve_f32_12x10x6x14_r7", kind="solve", lx=12, ly=10, lz=6, lt=14, nrhs=7, solver="mixed_f32",
             eps=0.8, m0=-0.75),
        # the headline: a block of 16 at 32^3 x 64 with half-storage inner solves
        dict(name="solve_f16_32x32x32x64_r16", kind="solve", lx=32, ly=32, lz=32, lt=64, nrhs=16,
             solver="mixed_f16", eps=0.8, m0=-0.78),
        # the plain FP64 solver, which users take as their reference
        dict(name="solve_f64_16x16x16x16_r8", kind="solve", lx=16, ly=16, lz=16, lt=16, nrhs=8, solver="f64",
             eps=0.8, m0=-0.75),
        # the 8^4 estimator: many short runs of 16 probing vectors, eight blocks in flight
        dict(name="trace_8x8x8x8_hp16x32_k100", kind="trace", lx=8, ly=8, lz=8, lt=8, ncolors=16, nvec=16, runs=32,
             block=16, lanes=8, k=100, store="f64", solver="mixed_f32", eps=0.7, m0=-0.6),
        # one stretch of a 512-colour run on the 16^3 x 32 lattice, deflation space in BF16
        dict(name="trace_16x16x16x32_hp512_k64", kind="trace", lx=16, ly=16, lz=16, lt=32, ncolors=512, nvec=64,
             runs=1, block=32, lanes=1, k=64, store="bf16", solver="mixed_f32", eps=0.8, m0=-0.75),
        # one Adam step of the learned preconditioner on (residual, error) pairs
        dict(name="net_train_16x16x16x32_b4", kind="net", lx=16, ly=16, lz=16, lt=32, nrhs=4, act=1, eps=0.8,
             m0=-0.75),
        # the deflation space of the 8^4 workload, to the usual loose residual
        dict(name="eig_f64_8x8x8x8_k64", kind="eig", lx=8, ly=8, lz=8, lt=8, k=64, eps=0.7, m0=-0.6),
    ]


def _spread(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _extents(rng, most, step=2):
    """Four extents, multiples of step, the last up to twice as long as the others may be."""
    out = [max(4, step, step * round(_spread(rng, 4, m) / step)) for m in (most, most, most, 2 * most)]
    return dict(lx=out[0], ly=out[1], lz=out[2], lt=out[3])


def draw(rng):
    kind = rng.choice(("dslash", "project", "solve", "solve", "solve", "trace", "trace", "net", "eig"))
    eps, m0 = rng.choice(FIELDS)
    if kind == "dslash":
        prec = rng.choice(("f64", "f32", "bf16", "f16", "df32"))
        c = dict(_extents(rng, 32), kind=kind, prec=prec, dagger=prec in ("f64", "f32") and rng.random() < 0.5,
                 eps=eps, m0=m0)
        c["nrhs"] = _spread(rng, 1, max(1, min(32, (1 << 22) // _volume(c))))
    elif kind == "project":
        c = dict(_extents(rng, 16), kind=kind, k=_spread(rng, 8, 96), store=rng.choice(("f64", "f32", "bf16")),
                 nrhs=_spread(rng, 1, 16), x0=rng.random() < 0.5)
    elif kind == "solve":
        solver = rng.choice(("mixed_f32", "mixed_f32", "mixed_f16", "mixed_f16", "mixed_bf16", "f64"))
        c = dict(_extents(rng, 12 if solver == "f64" else 24), kind=kind, solver=solver, eps=eps, m0=m0)
        c["nrhs"] = _spread(rng, 1, max(1, min(32, (1 << 18 if solver == "f64" else 1 << 22) // _volume(c))))
    elif kind == "trace":
        ncolors = rng.choice((1, 16, 32, 256))
        period = {1: 2, 16: 2, 32: 4, 256: 4}[ncolors]
        c = dict(_extents(rng, 8, period), kind=kind, ncolors=ncolors, nvec=min(ncolors, rng.choice((8, 16))),
                 k=_spread(rng, 8, 96), store=rng.choice(("f64", "f32", "bf16")), lanes=rng.choice((1, 2, 4)),
                 block=rng.choice((4, 8, 16)), solver=rng.choice(("mixed_f32", "mixed_f16")), eps=eps, m0=m0)
        c["runs"] = _spread(rng, 8, 32) if ncolors == 1 else _spread(rng, 1, 4)
    elif kind == "net":
        c = dict(_extents(rng, 16), kind=kind, nrhs=rng.randint(1, 4), act=rng.choice((0, 1)), eps=eps, m0=m0)
    else:
        c = dict(_extents(rng, 6), kind=kind, k=_spread(rng, 8, 48), eps=0.7, m0=-0.6)
    return c


def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _volume(c):
    return c["lx"] * c["ly"] * c["lz"] * c["lt"]


# ------------------------------------------------------------------ inputs
def _tile(extent, most):
    """The longest period up to `most` that divides the extent."""
    return next(d for d in range(min(extent, most), 0, -1) if extent % d == 0)


def _links(c):
    """(V, 4, 3, 3) complex128 on the GPU: U = exp(i eps H), H Gaussian, Hermitian and traceless. A lattice beyond
    16^3 x 32 repeats a smaller field periodically, as the library's own large benchmarks do. One field for each
    lattice and eps: a program estimates on one configuration of its ensemble with many noise vectors."""
    g = torch.Generator(device="cuda").manual_seed(1000)
    base = [_tile(d, m) for d, m in zip(_dims(c), (16, 16, 16, 32))]
    n = 4 * math.prod(base)
    re = torch.randn(n, 3, 3, generator=g, device="cuda", dtype=torch.float64)
    im = torch.randn(n, 3, 3, generator=g, device="cuda", dtype=torch.float64)
    h = torch.complex(re, im)
    h = 0.5 * (h + h.mH)
    tr = h.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3.0
    h = h - tr[:, None, None] * torch.eye(3, device="cuda", dtype=h.dtype)
    x = 1j * c["eps"] * h / 256.0   # exp by scaling and squaring of the series
    u = torch.eye(3, device="cuda", dtype=h.dtype).expand_as(x).clone()
    for q in range(10, 0, -1):
        u = torch.eye(3, device="cuda", dtype=h.dtype) + _mm3(x, u) / q
    for _ in range(8):
        u = _mm3(u, u)
    u = u.reshape(base[3], base[2], base[1], base[0], 36)
    reps = [d // b for d, b in zip(_dims(c), base)]
    return u.repeat(reps[3], reps[2], reps[1], reps[0], 1).reshape(-1, 4, 3, 3)


_GAUGES = {}  # the handles of the configurations at work, kept as a program keeps its own


def _gauge(c, lat):
    key = _dims(c) + (c["eps"],)
    if key not in _GAUGES:
        _GAUGES[key] = dtr.gauge_from_host(lat, _links(c).cpu().numpy())
    return _GAUGES[key]


def _mm3(a, b):
    """Product of many 3 x 3 matrices."""
    return (a[:, :, :1] * b[:, :1, :] + a[:, :, 1:2] * b[:, 1:2, :]) + a[:, :, 2:] * b[:, 2:, :]


def _z4(rows, n, seed):
    """Rows of Z4 noise, (rows, n) complex128."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 29)
    out = torch.empty(rows, n, dtype=torch.complex128, device="cuda")
    val = torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device="cuda")
    for row in out:
        row.copy_(val[torch.randint(0, 4, (n,), generator=g, device="cuda")])
    return out


def _normal(rows, n, seed):
    """Rows of complex Gaussian entries, (rows, n) complex128."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 31)
    return torch.view_as_complex(torch.randn(rows, n, 2, generator=g, device="cuda", dtype=torch.float64))


def _space(c, seed):
    """Deflation vectors as rows (k, N), unit length up to rounding to the storage type, and their eigenvalues:
    signed, between 0.3 and 1.5 as on these fields."""
    n = 12 * _volume(c)
    v = _normal(c["k"], n, seed) / math.sqrt(2.0 * n)
    to = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[c["store"]]
    v = torch.view_as_complex(torch.view_as_real(v).to(to).to(torch.float64))
    r = np.random.default_rng(seed + 5)
    return v, (0.3 + 1.2 * np.sort(r.random(c["k"]))) * r.choice((-1.0, 1.0), c["k"])


def _weights(seed):
    """Network weights near a damped identity, representable in BF16."""
    r = np.random.default_rng(seed + 7)
    w = (0.02 * r.standard_normal((4, 81, 24, 24))).astype(np.float32)
    w[:, 40] += np.eye(24, dtype=np.float32) * np.array([0.3, 1, 1, 1], np.float32)[:, None, None]
    return torch.from_numpy(w).to(torch.bfloat16).to(torch.float32).numpy()


def _pairs(c, seed):
    """(residual, error) pairs of unit scale: error = residual / 4 plus a correction, the size of A^-1 r here."""
    n = 12 * _volume(c)
    return _normal(c["nrhs"], n, seed), 0.25 * _normal(c["nrhs"], n, seed) + 0.05 * _normal(c["nrhs"], n, seed + 1)


def prepare(case, seed):
    c = case
    lat = dtr.make_lattice(_dims(c))
    s = dict(case=c, seed=seed, lat=lat)
    if "eps" in c and c["kind"] != "net":
        s["gauge"] = _gauge(c, lat)
    if c["kind"] in ("project", "trace"):
        v, lam = _space(c, seed)
        s["defl"] = dtr.defl_create(lat, v.cpu().numpy().T, lam, c["store"])
    if c["kind"] == "dslash":
        s["x"] = _normal(c["nrhs"], lat.N, seed)
    elif c["kind"] in ("project", "solve"):
        s["z"] = _z4(c["nrhs"], lat.N, seed)
    elif c["kind"] == "net":
        s["net"] = dtr.Net(lat, act=c["act"], weights=_weights(seed))
        s["r"], s["e"] = _pairs(c, seed)
    if c["kind"] == "solve":
        s["params"] = dtr.solve_params(solver=c["solver"])
    elif c["kind"] == "trace":
        s["params"] = dtr.trace_params(seed=seed, z0_first=1, n_z0=c["runs"], ncolors=c["ncolors"], nvec=c["nvec"],
                                       block=c["block"], lanes=c["lanes"],
                                       solve=dtr.solve_params(solver=c["solver"]))
        s["work"] = dtr.TraceWorkspace(s["gauge"], s["defl"], s["params"])
    elif c["kind"] == "eig":
        s["params"] = dtr.eig_params(c["k"], store="f64", degree=32, seed=seed)
    return s


# --------------------------------------------------------------------- run
def run(s):
    c = s["case"]
    if c["kind"] == "dslash":
        return dtr.dslash(s["gauge"], c["m0"], s["x"], dagger=c["dagger"], prec=c["prec"])
    if c["kind"] == "project":
        return list(dtr.deflate_project(s["defl"], s["z"], want_coeff=True, want_x0=c["x0"]))
    if c["kind"] == "solve":
        return dtr.solve_batch(s["gauge"], c["m0"], s["z"], params=s["params"])[0]
    if c["kind"] == "trace":
        out = dtr.trace_estimate(s["gauge"], c["m0"], s["defl"], s["params"], workspace=s["work"])
        return dict(samples=out["samples"], trace=np.array([out["trace"]]), T_D=np.array([out["T_D"]]))
    if c["kind"] == "net":
        loss, grad = s["net"].train_step(s["r"], s["e"], want_grad=True)
        return dict(loss=loss, grad=grad)
    defl = dtr.eig_deflation(s["gauge"], c["m0"], s["params"])[0]
    return dict(lam=defl.lambdas(), T_D=np.array([defl.T_D()]))


def work(case):
    c = case
    v = _volume(c)
    n = 12 * v
    links = 4 * 9 * 16 * v
    if c["kind"] == "dslash":
        return dict(bytes=2 * n * c["nrhs"] * 16 + links, flops=FLOPS_DSLASH * v * c["nrhs"])
    if c["kind"] == "project":
        width = {"f64": 16, "f32": 8, "bf16": 4}[c["store"]]
        fields = 2 if c["x0"] else 1
        return dict(bytes=n * c["k"] * width + fields * n * c["nrhs"] * 16,
                    flops=8.0 * n * c["k"] * c["nrhs"] * (2 + (1 if c["x0"] else 0)))
    if c["kind"] == "solve":
        return dict(bytes=2 * n * c["nrhs"] * 16 + links, flops=APPLICATIONS * FLOPS_DSLASH * v * c["nrhs"])
    if c["kind"] == "trace":
        width = {"f64": 16, "f32": 8, "bf16": 4}[c["store"]]
        solves = c["runs"] * c["nvec"]
        return dict(bytes=links + n * c["k"] * width,
                    flops=APPLICATIONS * FLOPS_DSLASH * v * solves + 8.0 * n * c["k"] * 2 * c["runs"])
    if c["kind"] == "net":  # four layers: forward, input gradient of the last three, weight gradient
        return dict(bytes=2 * n * c["nrhs"] * 16 + 2 * 4 * 4 * 81 * 24 * 24,
                    flops=2.0 * 81 * 24 * 24 * v * c["nrhs"] * (4 + 3 + 4))
    # degree 32, two stencils per degree and column, at least two filters and one extraction
    return dict(bytes=links + n * c["k"] * 16,
                flops=2 * c["k"] * v * 2 * 32 * FLOPS_DSLASH + 3 * 8.0 * n * c["k"] * c["k"])


# ------------------------------------------------------------------- exact
def _gammas():
    """gamma_x, gamma_y, gamma_z, gamma_t in the chiral basis."""
    s = torch.zeros(4, 2, 2, dtype=torch.complex128)
    s[0] = torch.tensor([[0, 1], [1, 0]])
    s[1] = torch.tensor([[0, -1j], [1j, 0]])
    s[2] = torch.tensor([[1, 0], [0, -1]])
    g = torch.zeros(4, 4, 4, dtype=torch.complex128)
    for k in range(3):
        g[k, :2, 2:] = -1j * s[k]
        g[k, 2:, :2] = 1j * s[k]
    g[3, :2, 2:] = g[3, 2:, :2] = torch.eye(2)
    return g.cuda()


class _Operator:
    """A (or A^H) on rows (nrhs, N), complex128, straight from its definition."""

    def __init__(self, c, links):
        self.c, self.u = c, links
        self.gam, self.one = _gammas(), torch.eye(4, dtype=torch.complex128, device="cuda")

    def _shift(self, f, mu, step):
        x, y, z, t = _dims(self.c)
        return torch.roll(f.reshape(t, z, y, x, -1), -step, 3 - mu).reshape(f.shape)

    def __call__(self, x, dagger=False):
        g5 = torch.tensor([1, 1, -1, -1], device="cuda")[:, None]
        f = x.reshape(x.shape[0], -1, 4, 3).permute(1, 3, 2, 0).contiguous()  # (V, colour, spin, rhs)
        if dagger:
            f = f * g5
        out = (4.0 + self.c["m0"]) * f
        for mu in range(4):
            u = self.u[:, mu]
            hop = self._colour(u, self._shift(f, mu, 1))
            out -= 0.5 * torch.einsum("ij,vcjr->vcir", self.one - self.gam[mu], hop)
            hop = self._shift(self._colour(u.mH, f), mu, -1)
            out -= 0.5 * torch.einsum("ij,vcjr->vcir", self.one + self.gam[mu], hop)
        if dagger:
            out = out * g5
        return out.permute(3, 0, 2, 1).reshape(x.shape)

    @staticmethod
    def _colour(u, f):
        return torch.matmul(u, f.reshape(f.shape[0], 3, -1)).reshape(f.shape)

    def solve(self, z, tol=1e-13, most=400):
        """BiCGStab, all rows at once; None if it does not get there."""
        x, r = torch.zeros_like(z), z.clone()
        rhat, p = r.clone(), r.clone()
        dot = lambda a, b: (a.conj() * b).sum(1, keepdim=True)  # noqa: E731
        rho, norm = dot(rhat, r), dot(z, z).real
        for _ in range(most):
            v = self(p)
            alpha = rho / dot(rhat, v)
            s = r - alpha * v
            t = self(s)
            omega = dot(t, s) / dot(t, t)
            x = x + alpha * p + omega * s
            r = s - omega * t
            if bool((dot(r, r).real <= tol * tol * norm).all()):
                break
            new = dot(rhat, r)
            p = r + (new / rho) * (alpha / omega) * (p - omega * v)
            rho = new
        r = z - self(x)
        return x if bool((dot(r, r).real <= 1e-22 * norm).all()) else None


def _gamma5(c):
    return torch.tensor([1.0] * 6 + [-1.0] * 6, device="cuda").repeat(_volume(c))


def _z0(seed, run, n):
    """The Z4 noise of one run from its definition: 2-bit codes of the Philox4x64-10 stream with key (seed, 0) and
    counters (dof // 128, run, 0, 0). numpy's generator steps its counter before it draws."""
    words = np.random.Philox(key=seed, counter=(run << 64) - 1).random_raw(4 * ((n + 127) // 128))
    codes = (words[:, None] >> (2 * np.arange(32, dtype=np.uint64))) & np.uint64(3)
    return np.array([1, 1j, -1, -1j])[codes.reshape(-1)[:n].astype(np.int64)]


def _colours(c):
    """Hierarchical-probing colour of every site."""
    lx, ly, lz, lt = _dims(c)
    t, z, y, x = (a.reshape(-1) for a in np.meshgrid(*(np.arange(m) for m in (lt, lz, ly, lx)), indexing="ij"))
    colour, n, level = np.zeros(x.shape, np.int64), 1, 0
    if c["ncolors"] > 1:
        colour, n = (x + y + z + t) & 1, 2
    while n < c["ncolors"]:
        colour = colour + n * (((y >> level) & 1) + 2 * ((z >> level) & 1) + 4 * ((t >> level) & 1))
        n *= 8
        if n >= c["ncolors"]:
            break
        level += 1
        colour = colour + n * (((x >> level) + (y >> level) + (z >> level) + (t >> level)) & 1)
        n *= 2
    return colour


def _probing(c, seed, run):
    """The run's probing vectors, rows (nvec, N)."""
    z0 = _z0(seed, run, 12 * _volume(c))
    both = _colours(c)[None, :] & np.arange(c["nvec"])[:, None]
    odd = np.zeros(both.shape, np.int64)
    while both.any():
        odd ^= both & 1
        both >>= 1
    return torch.from_numpy(np.repeat(1 - 2 * odd, 12, axis=1) * z0[None, :]).cuda()


def _deflated(c, v, lam, z):
    """(d, C, x0) of rows z: C = V^H [z, g5 z], d = sum_m conj(C) C5 / lambda, x0 = V Lambda^-1 V^H g5 z."""
    cz, c5 = v.conj() @ z.T, v.conj() @ (z * _gamma5(c)).T
    w = c5 / torch.from_numpy(lam).cuda()[:, None]
    return (cz.conj() * w).sum(0), torch.cat([cz, c5], 1).T.contiguous(), (v.T @ w).T.contiguous()


def _exact_net(c, seed):
    """Loss and weight gradient of the network by automatic differentiation."""
    r, e = _pairs(c, seed)
    w = torch.from_numpy(_weights(seed)).cuda().double().requires_grad_()
    lx, ly, lz, lt = _dims(c)
    grad, total = torch.zeros_like(w), 0.0
    for j in range(c["nrhs"]):
        f = torch.view_as_real(r[j]).reshape(lt, lz, ly, lx, 24)
        for layer in range(4):
            out = 0.0
            for o in range(81):
                step = [-(o // 27 - 1), -(o // 9 % 3 - 1), -(o // 3 % 3 - 1), -(o % 3 - 1)]
                out = out + torch.roll(f, step, (0, 1, 2, 3)) @ w[layer, o].T
            f = torch.nn.functional.leaky_relu(out, 0.25) if c["act"] and layer < 3 else out
        want = torch.view_as_real(e[j]).reshape(f.shape)
        loss = (f - want).square().sum() / want.square().sum()
        grad += torch.autograd.grad(loss, w)[0]
        total += float(loss.detach())
    return dict(loss=total, grad=grad)


def exact(case, seed):
    c = case
    v = _volume(c)
    if c["kind"] == "net":
        return _exact_net(c, seed)
    if c["kind"] == "eig":
        return None  # the pairs stop at a loose residual, so they are not the operator's own eigenvalues
    if c["kind"] == "project":
        vec, lam = _space(c, seed)
        d, coeff, x0 = _deflated(c, vec, lam, _z4(c["nrhs"], 12 * v, seed))
        return [d, coeff, x0 if c["x0"] else None]
    a = _Operator(c, _links(c))
    if c["kind"] == "dslash":
        x = _normal(c["nrhs"], 12 * v, seed)
        return torch.cat([a(row, c["dagger"]) for row in x.split(8)])
    if c["kind"] == "solve":
        if v * c["nrhs"] > 1 << 22:
            return None  # the plain torch solve would take minutes
        return a.solve(_z4(c["nrhs"], 12 * v, seed))
    if v * c["runs"] * c["nvec"] > 1 << 24:
        return None
    vec, lam = _space(c, seed)
    samples = []
    for run_ in range(1, 1 + c["runs"]):
        z = _probing(c, seed, run_)
        d = _deflated(c, vec, lam, z)[0]
        parts = [a.solve(row) for row in z.split(16)]
        if any(p is None for p in parts):
            return None
        samples.append(((z.conj() * torch.cat(parts)).sum(1) - d).cpu().numpy())
    t_d = ((vec.conj() * vec * _gamma5(c)).sum(1).real.cpu().numpy() / lam).sum()
    samples = np.array(samples)
    return dict(samples=samples, trace=np.array([t_d + samples.mean()]), T_D=np.array([t_d + 0j]))
