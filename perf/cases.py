"""The work that a user of this solver has it do, as measurable cases.

``listed()`` names twelve cases and ``draw(rng)`` gives further ones of the
same ranges.  A case goes through the package's public entry points:

* ``apply``   -- the fermion matrix on a block of spinor fields (``apply_H``;
  ``apply_H_mixed`` for the float-float operator), what a caller's
  own Krylov or residual code does with a lattice;
* ``cg``      -- ``shifted_cg``: every quadrature-point system of a window,
  the solutions wanted (the shift-vector update form);
* ``moments`` -- ``moments`` / ``moments_noalloc`` of solutions in hand;
* ``ssmom``   -- ``ssqcd_ss_moments`` into device memory: the whole filtered
  subspace of a window (seed recurrence, stored residuals, combination);
* ``solve``   -- ``ss_solve`` / ``ss_solve_windows`` to the eigenvalues;
* ``serve``   -- a batch of solves through the request scheduler.

Lattices, couplings and windows are those of the tests and the benchmark
(4^4 Haar links, 8^4, 12^4 and 16^3 x 32 smooth links) or ragged ones around
them.  Links and sources are drawn from the seed: the smooth fields' low
clusters move by far less than the window's margin from one draw to the next.

The solves return the eigenvalues that converged (residual <= 1e-8, the bound
the library itself counts by).  Eigenvectors of a twelvefold, nearly
degenerate cluster, the residuals at their rounding level and iteration
counts are not functions of the input to the last digits, so they are not
returned; the vectors of the same path are compared in the ``ssmom`` cases
(in FP64: after a thousand steps of the indefinite seed recurrence
float-float vectors agree to seven or eight digits only).  The FP32 operators
reach no eigenpair at that bound, and which of their variants runs is a
matter of timing, so no case stands for them.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1004_0292_gb300 as ss

PRECISIONS = {"fp64": ss.FP64, "df": ss.DF, "dfshift": ss.FP64_DFSHIFT}
CONVERGED = 1e-8


def listed():
    return [
        # one field on the smallest lattice: latency and launches
        dict(name="apply-4x4x4x4", kind="apply", X=4, Y=4, Z=4, T=4, links="haar", eps=0.0, kappa=0.13, nrhs=1,
             precision="fp64"),
        # odd extents, a volume that fills no block evenly, an odd number of fields
        dict(name="apply-7x9x5x11", kind="apply", X=7, Y=9, Z=5, T=11, links="haar", eps=0.0, kappa=0.13, nrhs=3,
             precision="fp64"),
        # the benchmark's lattice with its eight sources
        dict(name="apply-16x16x16x32", kind="apply", X=16, Y=16, Z=16, T=32, links="smooth", eps=0.5, kappa=0.135,
             nrhs=8, precision="fp64"),
        # the float-float operator on the same lattice
        dict(name="apply-df-16x16x16x32", kind="apply", X=16, Y=16, Z=16, T=32, links="smooth", eps=0.5, kappa=0.135,
             nrhs=4, precision="df"),
        # four fields on the middle lattice
        dict(name="apply-12x12x12x12", kind="apply", X=12, Y=12, Z=12, T=12, links="smooth", eps=0.4, kappa=0.13,
             nrhs=4, precision="fp64"),
        # every solution of the 8^4 window, in FP64
        dict(name="cg-8x8x8x8", kind="cg", X=8, Y=8, Z=8, T=8, links="smooth", eps=0.3, kappa=0.125, L=4, N=32,
             beta=0.6, precision="fp64", iters=770),
        # the same call on a ragged lattice with float-float shift vectors, fewer points
        dict(name="cg-dfshift-6x10x8x12", kind="cg", X=6, Y=10, Z=8, T=12, links="smooth", eps=0.3, kappa=0.125, L=2,
             N=16, beta=0.6, precision="dfshift", iters=700),
        # moments of one source's solutions on the benchmark's lattice
        dict(name="moments-16x16x16x32", kind="moments", X=16, Y=16, Z=16, T=32, L=1, N=32, M=16, noalloc=False),
        # one source of the benchmark's lattice from links to moments: its seed recurrence and combination
        dict(name="ssmom-16x16x16x32", kind="ssmom", X=16, Y=16, Z=16, T=32, links="smooth", eps=0.5, kappa=0.135,
             L=1, N=32, M=16, beta=0.6, precision="fp64", iters=1700),
        # eigenvalues of the 12^4 window, four sources, FP64
        dict(name="solve-12x12x12x12", kind="solve", X=12, Y=12, Z=12, T=12, links="smooth", eps=0.4, kappa=0.13, L=4,
             N=32, M=8, beta=0.3, precision="fp64", windows=1, block=0, iters=1300),
        # float-float on 8^4: a window on each side of the gap, sources in blocks side by side
        dict(name="solve-df-8x8x8x8", kind="solve", X=8, Y=8, Z=8, T=8, links="smooth", eps=0.3, kappa=0.125, L=4,
             N=32, M=8, beta=0.3, precision="df", windows=2, block=2, iters=850),
        # a batch of uneven requests on two resident 8^4 lattices, all submitted at once
        dict(name="serve-8x8x8x8", kind="serve", X=8, Y=8, Z=8, T=8, links="smooth", eps=0.3, kappa=0.125, L=4, N=32,
             M=8, beta=0.3, requests=6, iters=850),
    ]


def _spread(rng, lo, hi):
    """A whole number from lo to hi, even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "cg", "moments", "ssmom", "solve"])
    if kind in ("apply", "moments"):
        while True:
            d = [_spread(rng, 2, 16), _spread(rng, 2, 16), _spread(rng, 2, 16), _spread(rng, 2, 32)]
            V = d[0] * d[1] * d[2] * d[3]
            if V >= 64:
                break
        c = dict(kind=kind, X=d[0], Y=d[1], Z=d[2], T=d[3])
        if kind == "moments":
            most = max(1, min(8, 4200000 // (32 * V)))
            return dict(c, L=rng.randint(1, most), N=2 * rng.randint(2, 16), M=rng.randint(2, 16),
                        noalloc=rng.random() < 0.5)
        return dict(c, links=rng.choice(["haar", "smooth"]), eps=round(rng.uniform(0.2, 0.6), 3),
                    kappa=round(rng.uniform(0.1, 0.14), 4), nrhs=_spread(rng, 1, 8),
                    precision=rng.choice(["fp64", "fp64", "df"]))
    if kind == "solve":
        return dict(kind=kind, X=8, Y=8, Z=8, T=8, links="smooth", eps=0.3, kappa=0.125, L=rng.randint(3, 6),
                    N=2 * rng.randint(14, 18), M=rng.randint(6, 9), beta=0.3, precision=rng.choice(["fp64", "df"]),
                    windows=rng.randint(1, 2), block=rng.choice([0, 1, 2]), iters=850)
    d = [rng.randint(4, 10) for _ in range(3)] + [rng.randint(4, 14)]
    c = dict(kind=kind, X=d[0], Y=d[1], Z=d[2], T=d[3], links="smooth", eps=round(rng.uniform(0.25, 0.4), 3),
             kappa=round(rng.uniform(0.115, 0.125), 4), L=rng.randint(1, 4), N=2 * rng.randint(4, 16),
             beta=round(rng.uniform(0.4, 0.9), 2), iters=800)
    if kind == "cg":
        return dict(c, precision=rng.choice(["fp64", "fp64", "dfshift"]))
    # the low cluster depends on the links, kappa and T alone: any spatial extents have it in the window
    return dict(c, X=rng.randint(6, 10), Y=rng.randint(6, 10), Z=rng.randint(6, 10), T=8, eps=0.3, kappa=0.125,
                M=rng.randint(4, 12), precision="fp64")


# ---- inputs ------------------------------------------------------------------------------
def _dims(c):
    return c["X"], c["Y"], c["Z"], c["T"]


def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + what)


def _gauss(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.complex128)


def _links(c, seed, what=1):
    """SU(3) links (4, V, 3, 3): Haar, or exp(i eps G) with Gaussian traceless Hermitian G."""
    V = math.prod(_dims(c))
    g = _gen(seed, what)
    if c["links"] == "haar":
        a, b = _gauss(g, 4 * V, 3), _gauss(g, 4 * V, 3)
        a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
        b = b - a * (a.conj() * b).sum(-1, keepdim=True)
        b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
        u = torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2)
    else:
        x = _gauss(g, 4 * V, 3, 3)
        h = 0.5 * (x + x.mH)
        h = h - torch.eye(3, device="cuda") * (h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3)[:, None, None]
        u = torch.linalg.matrix_exp(1j * c["eps"] * h)
    return u.reshape(4, V, 3, 3).contiguous()


def _interval(c):
    """The accepted interval: the lowest positive cluster of the smooth fields of the tests."""
    if c["X"] == 12:
        return 0.085, 0.091
    if c["X"] == 16:
        return 0.0769, 0.1081
    return 0.105, 0.120


def _nprime(c):
    return c["N"] // 2 + (c["N"] // 2) % 2


def _nodes(c):
    a, b = _interval(c)
    n, p = c["N"], _nprime(c)
    gamma, rho = 0.5 * (a + b), 0.5 * (b - a) * (n / 2 - 1) / (p / 2 - 1)
    x = np.repeat(-1 + 2 * np.arange(n // 2) / (n / 2 - 1), 2)
    zeta = x + 1j * c.get("beta", 0.3) * np.where(np.arange(n) % 2 == 0, 1.0, -1.0)
    return gamma, rho, zeta


def _weights(zeta):
    """w_j = -P(0) / P'(zeta_j), P the polynomial with the nodes as its zeros."""
    d = zeta[:, None] - zeta[None, :]
    np.fill_diagonal(d, 1.0)
    return -np.prod(-zeta) / np.prod(d, axis=1)


def _requests(c):
    """Uneven requests of the batch: number of sources and points of each."""
    return [(c["L"] - k % 2, c["N"] - 4 * (k % 3), k % 2) for k in range(c["requests"])]


def prepare(case, seed):
    c, V, kind = case, math.prod(_dims(case)), case["kind"]
    st = dict(case=c, stream=torch.cuda.Stream())
    if kind == "moments":
        _, _, zeta = _nodes(dict(c, beta=0.3))
        st["zeta"], st["w"] = zeta, _weights(zeta)
        # solutions (z - A)^-1 v of a Gaussian v: random, growing towards the nodes by the axis
        y = _gauss(_gen(seed, 2), c["L"], c["N"], V, 4, 3)
        st["y"] = y.mul_(torch.as_tensor(1.0 / (0.3 + np.abs(zeta)), device="cuda")[None, :, None, None, None])
        st["lat"] = ss.create_lattice(_dims(c), 0.125, -1, stream=st["stream"])
        torch.cuda.synchronize()
        return st
    u = _links(c, seed)
    kinds = ["fp64", "df"] if kind == "serve" else [c["precision"]]
    st["lats"] = []
    torch.cuda.synchronize()
    for p in kinds:
        lat = ss.create_lattice(_dims(c), c["kappa"], -1, precision=PRECISIONS[p], stream=st["stream"])
        ss.upload_gauge(lat, u)
        st["lats"].append(lat)
    st["lat"] = st["lats"][0]
    fields = c["nrhs"] if kind == "apply" else c["L"]
    st["v"] = _gauss(_gen(seed, 2), fields, V, 4, 3)
    if kind == "cg":
        gamma, rho, zeta = _nodes(c)
        st["z"] = gamma + rho * zeta
    torch.cuda.synchronize()
    return st


# ---- one pass ----------------------------------------------------------------------------
def _converged(res):
    ev, _, resid, _ = ss.ss_eigpairs(res, want_vectors=False)
    return ev[resid <= CONVERGED]


def run(st):
    c, kind = st["case"], st["case"]["kind"]
    if kind == "apply":
        if c["precision"] == "fp64":
            return ss.apply_H(st["lat"], st["v"])
        return ss.apply_H_mixed(st["lat"], st["v"])
    if kind == "cg":
        status, y, _, _, _ = ss.shifted_cg(st["lat"], st["z"], st["v"], precision=PRECISIONS[c["precision"]])
        if status != ss.OK:
            raise RuntimeError("shifted CG ended with status %d" % status)
        return y
    if kind == "moments":
        if c["noalloc"]:
            return ss.moments_noalloc(st["w"], st["zeta"], st["y"], c["M"])
        return ss.moments(st["lat"], st["w"], st["zeta"], st["y"], c["M"])
    if kind == "ssmom":
        lat, lib = st["lat"], ss.lib()
        out = torch.empty((c["L"], c["M"], lat.V, 4, 3), dtype=torch.complex128, device="cuda")
        o = ss.Opts()
        lib.ssqcd_default_opts(ctypes.byref(o))
        o.beta, o.nprime = c["beta"], _nprime(c)
        o.sources, o.sources_on_device = st["v"].data_ptr(), 1
        # one source's stored residuals of the large lattice, as the benchmark holds two of them
        o.basis_max_bytes = 80e9
        iv, stats = (ctypes.c_double * 2)(*_interval(c)), ss.Stats()
        code = lib.ssqcd_ss_moments(lat.handle, iv, c["N"], c["M"], c["L"], ctypes.byref(o), out.data_ptr(), 1,
                                    ctypes.byref(stats))
        if code != ss.OK:
            raise RuntimeError("ss_moments ended with status %d" % code)
        return out
    a, b = _interval(c)
    if kind == "solve":
        if c["windows"] == 2:
            res = ss.ss_solve_windows(st["lat"], [(-b, -a), (a, b)], c["N"], c["M"], st["v"], beta=c["beta"],
                                      nprime=_nprime(c), source_block=c["block"], block_streams=2)
        else:
            res = ss.ss_solve(st["lat"], (a, b), c["N"], c["M"], st["v"], beta=c["beta"], nprime=_nprime(c),
                              source_block=c["block"])
        if res.status != ss.OK:
            raise RuntimeError(res.error)
        return _converged(res)
    server = ss.Server(60 * 10**9)
    ids = []
    for L, N, which in _requests(c):
        ids.append(server.submit(st["lats"][which], (a, b), N, c["M"], st["v"][:L].contiguous(), beta=c["beta"],
                                 nprime=_nprime(dict(c, N=N))))
    done = 0
    while done < len(ids):
        done += server.progress(wait=True)
    out = [_converged(server.take(i)) for i in ids]
    server.close()
    return out


# ---- what a pass cannot do without ----------------------------------------------------------
def work(case):
    c, V, kind = case, math.prod(_dims(case)), case["kind"]
    field, links, hop = 192 * V, 576 * V, 1368 * V
    if kind == "apply":
        return dict(bytes=links + 2 * c["nrhs"] * field, flops=c["nrhs"] * hop)
    if kind == "moments":
        return dict(bytes=c["L"] * (c["N"] + c["M"]) * field, flops=8 * 12 * V * c["L"] * c["N"] * c["M"])
    if kind == "cg":  # the solutions and the updates of y and p-hat
        return dict(bytes=links + c["L"] * (1 + c["N"]) * field,
                    flops=c["iters"] * c["L"] * (hop + 12 * V * (20 + 16 * c["N"])))
    if kind == "serve":
        runs = [(L, 1) for L, _, _ in _requests(c)]
    else:
        runs = [(c["L"], c.get("windows", 1))]
    flops = sum(c["iters"] * L * (hop + 12 * V * (20 + 4 * c["M"] * W)) for L, W in runs)
    if kind == "ssmom":
        return dict(bytes=links + c["L"] * (1 + c["M"]) * field, flops=flops)
    return dict(bytes=links + c["L"] * field, flops=flops)


# ---- the same in plain torch, 64 bits ---------------------------------------------------------
_B = [[[0, 1j], [1j, 0]], [[0, -1], [1, 0]], [[1j, 0], [0, -1j]], [[1, 0], [0, 1]]]


def _operator(u, kappa, dims):
    """A psi = gamma5 (psi - kappa D psi) on (L, V, 4, 3), antiperiodic in t."""
    X, Y, Z, T = dims
    grid = u.reshape(4, T, Z, Y, X, 3, 3)
    ones = torch.eye(4, device="cuda", dtype=torch.complex128)
    g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], device="cuda", dtype=torch.float64)
    gam = []
    for b in _B:
        g = torch.zeros(4, 4, device="cuda", dtype=torch.complex128)
        g[:2, 2:] = torch.tensor(b, device="cuda", dtype=torch.complex128)
        g[2:, :2] = g[:2, 2:].mH
        gam.append(g)

    def matmul(m, f):  # per site 3x3 on the colour index
        return torch.einsum("tzyxab,ltzyxsb->ltzyxsa", m, f)

    def apply(psi):
        f = psi.reshape(-1, T, Z, Y, X, 4, 3)
        d = torch.zeros_like(f)
        for mu in range(4):
            ax = 4 - mu
            fwd = torch.roll(f, -1, dims=ax)
            if mu == 3:
                fwd[:, T - 1] *= -1
            d += torch.einsum("ij,ltzyxja->ltzyxia", ones - gam[mu], matmul(grid[mu], fwd))
            bwd = torch.roll(matmul(grid[mu].mH, f), 1, dims=ax)
            if mu == 3:
                bwd[:, 0] *= -1
            d += torch.einsum("ij,ltzyxja->ltzyxia", ones + gam[mu], bwd)
        return ((f - kappa * d) * g5[:, None]).reshape(psi.shape)

    return apply


def _solutions(A, v, z, most=6000):
    """y (L, N, ...) of (z_j - A) y_j = v_l by the multi-shift CG recurrences, past the solver's own stop."""
    L, N = v.shape[0], len(z)
    zz = torch.as_tensor(z, device="cuda").reshape(1, N)
    dot = lambda a, b: (a.conj() * b).reshape(L, -1).sum(-1).real
    up = lambda s: s.reshape(L, 1, 1, 1)
    vn = dot(v, v).sqrt()
    r, p = v / up(vn), v / up(vn)
    y = torch.zeros(L, N, *v.shape[1:], device="cuda", dtype=torch.complex128)
    pj = v[:, None].repeat(1, N, 1, 1, 1)
    xi = vn.reshape(L, 1).to(torch.complex128).repeat(1, N)  # times the unit residual r
    ratio = torch.ones(L, N, device="cuda", dtype=torch.complex128)
    al0, be0 = torch.ones(L, device="cuda", dtype=torch.float64), torch.zeros(L, device="cuda", dtype=torch.float64)
    for k in range(most):
        q = -A(p)
        al = 1.0 / dot(p, q)
        r = r - up(al) * q
        rr = dot(r, r)
        a, b = al0[:, None] + 0j, (al * be0)[:, None] + 0j
        ratio = a / (b * (1 - ratio) + a * (1 + zz * al[:, None]))
        y += (al[:, None] * ratio).reshape(L, N, 1, 1, 1) * pj
        xi = xi * ratio * rr.sqrt()[:, None]
        s = 1.0 / rr.sqrt()
        r = r * up(s)
        p = r + up(rr * s) * p
        pj.mul_((ratio * ratio * rr[:, None]).reshape(L, N, 1, 1, 1)).add_(xi.reshape(L, N, 1, 1, 1) * r[:, None])
        al0, be0 = al, rr
        if k % 20 == 19 and float((xi.abs() / vn[:, None]).max()) < 1e-15:
            break
    return y


def _sums(y, zeta, M):
    w = _weights(zeta)
    coef = torch.as_tensor(w[:, None] * zeta[:, None] ** np.arange(M), device="cuda")
    return torch.einsum("jm,ljvsc->lmvsc", coef, y)


def _eigenvalues(A, s, a, b):
    """Rayleigh-Ritz on the span of the moments s (L, M, ...): the converged Ritz values in [a, b]."""
    S = s.reshape(s.shape[0] * s.shape[1], -1)
    S = S / torch.linalg.vector_norm(S, dim=-1, keepdim=True)
    Q = torch.linalg.qr(torch.linalg.qr(S.mT)[0])[0]
    AQ = A(Q.mT.reshape(-1, *s.shape[2:])).reshape(Q.shape[1], -1).mT
    H = Q.mH @ AQ
    lam, W = torch.linalg.eigh(0.5 * (H + H.mH))
    res = torch.linalg.vector_norm(AQ @ W - (Q @ W) * lam, dim=0)
    return lam[(lam >= a) & (lam <= b) & (res <= CONVERGED)].cpu().numpy()


def exact(case, seed):
    c, dims, kind = case, _dims(case), case["kind"]
    V = math.prod(dims)
    if kind == "moments":
        st = prepare(c, seed)
        return _sums(st["y"], st["zeta"], c["M"])
    if kind == "apply":
        v = _gauss(_gen(seed, 2), c["nrhs"], V, 4, 3)
        return _operator(_links(c, seed), c["kappa"], dims)(v)
    if V * c["N"] * c["L"] > 4096 * 300:  # the 12^4 and 16^3 x 32 recurrences take over twenty seconds here
        return None
    A = _operator(_links(c, seed), c["kappa"], dims)
    v = _gauss(_gen(seed, 2), c["L"], V, 4, 3)
    a, b = _interval(c)

    def sums(L, N, sign=1):
        gamma, rho, zeta = _nodes(dict(c, N=N))
        return _sums(_solutions(A, v[:L], sign * gamma + rho * zeta), zeta, c["M"])

    if kind == "cg":
        gamma, rho, zeta = _nodes(c)
        return _solutions(A, v, gamma + rho * zeta)
    if kind == "ssmom":
        return sums(c["L"], c["N"])
    if kind == "solve":
        parts = [_eigenvalues(A, sums(c["L"], c["N"]), a, b)]
        if c["windows"] == 2:
            parts.insert(0, _eigenvalues(A, sums(c["L"], c["N"], -1), -b, -a))
        return np.concatenate(parts)
    # every request of the batch asks for the same window of the same links
    ev = _eigenvalues(A, sums(c["L"], c["N"]), a, b)
    return [ev for _ in _requests(c)]
