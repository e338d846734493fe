"""The library's workloads as timed cases: what one call of each entry point costs a program.

`listed()` holds the cases, `draw(rng)` more of the same ranges, `prepare` makes a
case's inputs and plan on the GPU, `run` is one pass through the public calls,
`work` counts what a pass cannot do without and `exact` is its result in float64
from plain torch, by the discrete operators' own definition.

Orbitals are sums of three s- or p-type Gaussian primitives (exponents
U[0.5, 2] bohr^-2) on random atom centres, orthonormalised, on grids of the
spacings and sizes of `workloads/`: grid axes of 16 to 128 points in multiples of
eight (tensor-core plans), 1 to 256 orbitals.
"""
import math

import numpy as np
import torch

import paper_2406_16998_gb300 as kx

D, P = kx.KX_DIRICHLET, kx.KX_PERIODIC
U, S = kx.KX_UNSCREENED, kx.KX_SCREENED
OMEGA = 0.11
EXACT_FLOPS = 8e12  # float64 work above which `exact` would take too long


def _case(name, op, n, h, bc, kind, n_orb, **more):
    c = {"op": op, "n1": n[0], "n2": n[1], "n3": n[2], "h": h, "bc": bc, "kind": kind, "n_orb": n_orb,
         "precision": kx.KX_F16X3, "occ": False, "l_max": -1, "k1": 1, "k2": 1, "k3": 1, "n_vec": 0}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a molecule of four orbitals on a 32^3 box, where launches and latency count
        _case("vx_32_4", "vx", (32, 32, 32), 0.5, "DDD", U, 4),
        # the same system in float64, the accuracy reference a user checks a new system against
        _case("vx_fp64_32_4", "vx", (32, 32, 32), 0.5, "DDD", U, 4, precision=kx.KX_FP64),
        # a few Poisson solves between SCF steps on a ragged box with mixed boundaries
        _case("solve_56x40x48_6", "solve", (56, 40, 48), 0.3, "PPD", U, 6),
        # an isolated molecule of ordinary size: the SCF's exchange apply at 96^3
        _case("vx_96_64", "vx", (96, 96, 96), 0.25, "DDD", U, 64),
        # the largest: 256 orbitals of a 64-water periodic cell, screened kernel
        _case("vx_periodic_80_256", "vx", (80, 80, 80), 0.293375, "PPP", S, 256),
        # a large box with few orbitals (planes too large for the fused middle products)
        _case("vx_120_16", "vx", (120, 112, 120), 0.25, "DDD", S, 16),
        # differentiation: E_x and its gradient through autograd, fractional occupations
        _case("grad_64x64x96_64", "grad", (64, 64, 96), 0.3, "PPP", S, 64, occ=True),
        # an isolated system with multipole boundary values of order 2
        _case("vx_multipole_72_40", "vx", (72, 72, 72), 0.3, "DDD", U, 40, l_max=2),
        # Brillouin-zone sampling of a slab (vacuum along the third axis)
        _case("kpoints_slab_64_16", "kpoints", (64, 64, 64), 0.3, "PPD", U, 16, k1=2, k2=2),
        # Brillouin-zone sampling of a bulk cell with unequal axes, fractional occupations
        _case("kpoints_bulk_48x40x56_6", "kpoints", (48, 40, 56), 0.3, "PPP", S, 6, k1=2, k2=2, occ=True),
        # the compressed operator: built once per outer iteration, applied to the bands
        _case("ace_96_64", "ace", (96, 96, 96), 0.25, "DDD", U, 64, n_vec=64),
        # the DFT variant on a periodic cell
        _case("vx_fft_80_48", "vx", (80, 80, 80), 0.293375, "PPP", S, 48, precision=kx.KX_FFT32),
    ]


def _pairs(c):
    return c["n_orb"] * (c["n_orb"] + 1) // 2


def _solves(c):
    if c["op"] == "solve":
        return c["n_orb"]
    if c["op"] == "kpoints":
        nk = c["k1"] * c["k2"] * c["k3"]
        return nk * (nk + 1) // 2 * c["n_orb"] ** 2
    return _pairs(c)


def _cost(c):
    """Rough relative cost of a pass: grid values solved for (k-point solves are complex, float64 is slow)."""
    N = c["n1"] * c["n2"] * c["n3"]
    if c["op"] == "ace":
        return 0.3 * N * (c["n_orb"] + c["n_vec"])
    return _solves(c) * N * {"kpoints": 3.0, "grad": 1.5}.get(c["op"], 1.0) * (100 if c["precision"] == kx.KX_FP64 else 1)


_SMOOTH = [16, 20, 24, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 90, 96, 100]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind of call, then sizes over its whole range."""
    top = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["vx", "vx", "vx", "solve", "grad", "multipole", "kpoints", "kpoints", "ace", "fft", "fp64"])
        n = [8 * rng.randint(2, 16) for _ in range(3)]
        bc = rng.choice(["DDD", "PPP", "PPD", "PDD", "DPD"])
        h = round(rng.uniform(0.2, 0.5), 3)
        more = {"occ": rng.random() < 0.4}
        if op == "fft":
            n, bc = [rng.choice(_SMOOTH) for _ in range(3)], "PPP"
            if n[1] * (n[0] + 1) > 12800 or n[0] * n[1] * n[2] % 4:  # a plane per CTA, float4 grid vectors
                continue
            c = _case("", "vx", n, h, bc, S, _log_int(rng, 2, 64), precision=kx.KX_FFT32, **more)
        elif op == "fp64":
            n = [rng.randint(12, 48) for _ in range(3)]
            c = _case("", "vx", n, h, bc, S, _log_int(rng, 1, 12), precision=kx.KX_FP64, **more)
        elif op == "multipole":
            n = [min(m, 96) for m in n]
            c = _case("", "vx", n, h, "DDD", U, _log_int(rng, 2, 64), l_max=rng.choice([1, 2]), **more)
        elif op == "kpoints":
            n = [min(m, 96) for m in n]
            bc = rng.choice(["PPP", "PPD", "PDD"])
            k = [rng.choice([1, 2]) if b == "P" else 1 for b in bc]
            c = _case("", "kpoints", n, h, bc, S if bc == "PPP" else rng.choice([U, S]), _log_int(rng, 1, 24),
                      k1=k[0], k2=k[1], k3=k[2], **more)
        elif op == "ace":
            c = _case("", "ace", n, h, bc, S, _log_int(rng, 4, 128), n_vec=_log_int(rng, 1, 160))
        elif op == "solve":
            c = _case("", "solve", n, h, bc, S if bc == "PPP" else rng.choice([U, S]), _log_int(rng, 1, 64))
        else:
            c = _case("", op, n, h, bc, S if bc == "PPP" else rng.choice([U, S]), _log_int(rng, 2, 160), **more)
        N = n[0] * n[1] * n[2]
        vectors = (c["n_orb"] + c["n_vec"]) * c["k1"] * c["k2"] * c["k3"]
        # at least 5 bohr^3 of box per vector (linearly independent orbitals)
        if _cost(c) <= top / 2 and N * vectors <= 80 ** 3 * 256 and N * h ** 3 >= 5 * max(c["n_orb"], c["n_vec"]):
            return c


# ---------------------------------------------------------------- inputs
def _bc(c):
    return [D if b == "D" else P for b in c["bc"]]


def _n(c):
    return [c["n1"], c["n2"], c["n3"]]


def _orbitals(c, rng, count, dev):
    """`count` orthonormal real vectors (count, N) in the case's box."""
    n, h, bc = _n(c), c["h"], _bc(c)
    L = [(n[a] + 1) * h if bc[a] == D else n[a] * h for a in range(3)]
    lo = np.array([0.25 * L[a] if bc[a] == D else 0.0 for a in range(3)])
    hi = np.array([0.75 * L[a] if bc[a] == D else L[a] for a in range(3)])
    n_c = max(3, (3 * count + 3) // 4)
    centres = rng.uniform(lo, hi, (n_c, 3))
    at, kind, ax = (rng.integers(0, k, (count, 3)) for k in (n_c, 2, 3))
    alpha, coef = rng.uniform(0.5, 2.0, (count, 3)), rng.standard_normal((count, 3))
    g = []
    for a in range(3):
        x = (np.arange(n[a]) + (1.0 if bc[a] == D else 0.0)) * h
        d = x - centres[at, a][..., None]
        if bc[a] == P:
            d = (d + 0.5 * L[a]) % L[a] - 0.5 * L[a]
        e = np.exp(-alpha[..., None] * d * d)
        e = np.where(((kind == 1) & (ax == a))[..., None], e * d, e)
        g.append(torch.from_numpy(e if a else e * coef[..., None]).to(dev))
    psi = torch.zeros((count, n[2], n[1], n[0]), dtype=torch.float64, device=dev)
    for p in range(3):
        yx = g[1][:, p, :, None] * g[0][:, p, None, :]
        psi.addcmul_(g[2][:, p, :, None, None].expand(-1, -1, n[1], n[0]),
                     yx[:, None].expand(-1, n[2], -1, -1))
    psi = psi.view(count, -1)
    G = (h ** 3 * (psi @ psi.T)).cpu().numpy()
    W = np.linalg.inv(np.linalg.cholesky(G + 1e-10 * np.trace(G) / count * np.eye(count)))
    return torch.from_numpy(W).to(dev) @ psi


def _theta(c):
    ks = [c["k1"], c["k2"], c["k3"]]
    th = [[2 * math.pi * i / ks[0], 2 * math.pi * j / ks[1], 2 * math.pi * k / ks[2]]
          for k in range(ks[2]) for j in range(ks[1]) for i in range(ks[0])]
    return th, [1.0 / len(th)] * len(th)


def _inputs(c, seed):
    """The case's tensors on the GPU, from the seed alone."""
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    N = c["n1"] * c["n2"] * c["n3"]
    s = {}
    if c["op"] == "kpoints":
        th, wk = _theta(c)
        n = _n(c)
        psi = torch.empty((len(th), c["n_orb"], N), dtype=torch.complex128, device=dev)
        for k, t in enumerate(th):
            re, im = (_orbitals(c, rng, c["n_orb"], dev) for _ in range(2))
            ph = [torch.arange(n[a], dtype=torch.float64, device=dev) * (t[a] / n[a]) for a in range(3)]
            ang = (ph[2][:, None, None] + ph[1][None, :, None] + ph[0][None, None, :]).reshape(-1)
            psi[k] = torch.polar(torch.full_like(ang, math.sqrt(0.5)), ang) * torch.complex(re, im)
        s["psi"] = psi
        shape = (len(th), c["n_orb"])
    else:
        s["psi"] = _orbitals(c, rng, c["n_orb"], dev)
        shape = (c["n_orb"],)
        if c["op"] == "solve":  # charge densities: products of orbitals, of either sign
            s["psi"] = s["psi"] * s["psi"].roll(1, 0)
        if c["op"] == "ace":
            # a local (Slater-like) exchange potential stands in for Vx: negative definite, smooth
            v = torch.pow((s["psi"] ** 2).sum(0), 1.0 / 3.0) + 0.05
            s["vx"] = -v * s["psi"]
            s["phi"] = _orbitals(c, rng, c["n_vec"], dev)
    s["occ"] = torch.from_numpy(rng.uniform(0.3, 1.0, shape)).to(dev) if c["occ"] else None
    return s


def prepare(case, seed):
    c = dict(case)
    s = _inputs(c, seed)
    s["op"] = c["op"]
    s["plan"] = kx.Plan(_n(c), [c["h"]] * 3, _bc(c), c["kind"], OMEGA, precision=c["precision"])
    if c["l_max"] >= 0:
        s["plan"].set_multipole(c["l_max"])
    if c["op"] == "kpoints":
        s["theta"], s["wk"] = _theta(c)
    if c["op"] == "grad":
        s["psi"].requires_grad_(True)
    return s


def run(s):
    op, plan = s["op"], s["plan"]
    if op == "solve":
        return kx.kx_apply_fL(plan, s["psi"])
    if op == "kpoints":
        return kx.kx_vx_kpoints(plan, s["theta"], s["wk"], s["psi"], s["occ"])
    if op == "ace":
        xi, M = kx.kx_ace(plan, s["psi"], s["vx"])
        return xi, M, kx.kx_ace_apply(plan, xi, s["phi"])
    if op == "grad":
        e = kx.exchange_energy(s["psi"], plan, s["occ"])
        (g,) = torch.autograd.grad(e, s["psi"])
        return e.detach(), g
    return kx.kx_vx_apply(plan, s["psi"], s["occ"])


# ---------------------------------------------------------------- work
def _solve_flops(c):
    """One f(L) b: a fast transform and back per periodic axis, a dense one per Dirichlet axis."""
    n = _n(c)
    N = n[0] * n[1] * n[2]
    cplx = c["op"] == "kpoints"
    fl = 0.0
    for a in range(3):
        if c["bc"][a] == "P":
            fl += 2 * 2.5 * N * math.log2(n[a]) * (2 if cplx else 1)
        else:
            fl += 4.0 * N * n[a] * (2 if cplx else 1)
    return fl


def work(case):
    c = dict(case)
    N = c["n1"] * c["n2"] * c["n3"]
    n_orb, n_vec = c["n_orb"], c["n_vec"]
    if c["op"] == "ace":  # psi, vx, phi in; xi, M, V phi out
        return {"bytes": 8.0 * N * (3 * n_orb + 2 * n_vec) + 8.0 * n_orb ** 2,
                "flops": 2.0 * N * n_orb * (2 * n_orb + 2 * n_vec)}
    nk = c["k1"] * c["k2"] * c["k3"]
    vectors = n_orb * nk * (2 if c["op"] == "kpoints" else 1)
    flops = _solves(c) * (_solve_flops(c) + 6.0 * N)
    if c["op"] == "grad":  # E_x alone first: the forward half
        flops *= 1.5
    return {"bytes": 2 * 8.0 * N * vectors, "flops": flops}


# ---------------------------------------------------------------- float64 result
def _fd_weights(order):
    m = order // 2
    w = [-2.0 * sum(1.0 / (p * p) for p in range(1, m + 1))]
    fm = math.factorial(m)
    return w + [2.0 * (-1) ** (p + 1) * fm * fm / (p * p * math.factorial(m - p) * math.factorial(m + p))
                for p in range(1, m + 1)]


class _Exact:
    """f(L) in complex or real float64: Fourier modes on periodic axes, eigenvectors on Dirichlet axes."""

    def __init__(self, c, theta=(0.0, 0.0, 0.0)):
        self.n, self.bc, h = _n(c), _bc(c), c["h"]
        dev = torch.device("cuda")
        w = _fd_weights(12)
        self.V, self.phase, lam = [], [], []
        for a in range(3):
            n = self.n[a]
            if self.bc[a] == P:
                kap = (2 * math.pi * np.arange(n) + theta[a]) / n
                lam.append((w[0] + 2 * sum(w[p] * np.cos(p * kap) for p in range(1, 7))) / h ** 2)
                self.V.append(None)
                ph = np.exp(1j * theta[a] * np.arange(n) / n) if theta[a] else None
                self.phase.append(None if ph is None else torch.from_numpy(ph).to(dev))
            else:
                i = np.arange(n)
                d = np.abs(i[:, None] - i[None, :])
                l, V = np.linalg.eigh(np.where(d <= 6, np.array(w + [0.0] * n)[np.minimum(d, 7)], 0.0) / h ** 2)
                lam.append(l)
                self.V.append(torch.from_numpy(V).to(dev))
                self.phase.append(None)
        mu = -(lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :])
        if c["kind"] == U:
            f = 4 * math.pi / mu
        else:
            small = np.abs(mu) < 1e-12
            m1 = np.where(small, 1.0, mu)
            f = np.where(small, math.pi / OMEGA ** 2, -4 * math.pi * np.expm1(-m1 / (4 * OMEGA ** 2)) / m1)
        self.f = torch.from_numpy(f).to(dev)

    def __call__(self, b):
        """b: (R, N) real or complex; returns the same."""
        real = not b.is_complex()
        t = b.view(-1, self.n[2], self.n[1], self.n[0])
        shape = [(1, 1, 1, -1), (1, 1, -1, 1), (1, -1, 1, 1)]
        dense = [a for a in range(3) if self.bc[a] != P]
        four = [3 - a for a in range(3) if self.bc[a] == P]
        for a in dense:
            t = self._mode(t, a, self.V[a])
        for a in range(3):
            if self.phase[a] is not None:
                t = t * self.phase[a].conj().view(shape[a])
        if four and real:  # Hermitian half along the last Fourier axis
            k = torch.fft.rfftn(t, dim=four)
            f = self.f.narrow(four[-1] - 1, 0, k.shape[four[-1]])
            t = torch.fft.irfftn(k * f, s=[t.shape[d] for d in four], dim=four)
        elif four:
            t = torch.fft.ifftn(torch.fft.fftn(t, dim=four) * self.f, dim=four)
        else:
            t = t * self.f
        for a in range(3):
            if self.phase[a] is not None:
                t = t * self.phase[a].view(shape[a])
        for a in dense:
            t = self._mode(t, a, self.V[a].T)
        return t.reshape(b.shape)

    @staticmethod
    def _mode(t, a, M):
        """Contract grid axis a of t (R, n3, n2, n1) with the rows of M."""
        if t.is_complex():
            return torch.complex(_Exact._mode(t.real, a, M), _Exact._mode(t.imag, a, M))
        if a == 0:
            return t @ M
        if a == 1:
            return M.T @ t
        r, n3, n2, n1 = t.shape
        return (M.T @ t.reshape(r, n3, n2 * n1)).view(r, n3, n2, n1)


def _multipole_terms(c, dV):
    """Rank-K form of the boundary values: phi = f(L)(b + sum_k q_k g_k), q_k = dV <R_k, b>, in Cartesian
    moments up to l_max <= 2 about the box centre."""
    n, h = _n(c), c["h"]
    w = _fd_weights(12)
    x = [(np.arange(-6, n[a] + 6) + 1.0) * h - (n[a] + 1) * h / 2 for a in range(3)]
    one = lambda X, Y, Z, r: np.ones_like(r)
    polys = [(one, lambda X, Y, Z, r: 1 / r)]
    if c["l_max"] >= 1:
        for a in range(3):
            polys.append((lambda X, Y, Z, r, a=a: (X, Y, Z)[a] + 0 * r,
                          lambda X, Y, Z, r, a=a: (X, Y, Z)[a] / r ** 3))
    if c["l_max"] >= 2:
        for a in range(3):
            for b in range(3):
                polys.append((lambda X, Y, Z, r, a=a, b=b: 3 * (X, Y, Z)[a] * (X, Y, Z)[b] - (a == b) * r * r,
                              lambda X, Y, Z, r, a=a, b=b: 0.5 * (X, Y, Z)[a] * (X, Y, Z)[b] / r ** 5))
    inner = [x[a][6:-6] for a in range(3)]

    def at(fn, xs):
        X, Y, Z = xs[0][None, None, :], xs[1][None, :, None], xs[2][:, None, None]
        return fn(X, Y, Z, np.sqrt(X * X + Y * Y + Z * Z))

    dev = torch.device("cuda")
    R, G = [], []
    for reg, irr in polys:
        R.append(torch.from_numpy(np.ascontiguousarray(at(reg, inner)).reshape(-1)).to(dev))
        g = np.zeros((n[2], n[1], n[0]))
        for a in range(3):
            g_a = np.moveaxis(g, 2 - a, 0)
            for j in list(range(-6, 0)) + list(range(n[a], n[a] + 6)):
                xs = list(inner)
                xs[a] = x[a][j + 6:j + 7]
                layer = np.moveaxis(at(irr, xs), 2 - a, 0)[0]
                for i in range(max(0, j - 6), min(n[a], j + 7)):
                    g_a[i] += w[abs(i - j)] / h ** 2 * layer / (4 * math.pi)
        G.append(torch.from_numpy(g.reshape(-1)).to(dev))
    return dV * torch.stack(R), torch.stack(G)


def exact(case, seed):
    c = dict(case)
    n, N = _n(c), c["n1"] * c["n2"] * c["n3"]
    dense = sum(n[a] for a in range(3) if c["bc"][a] == "D")
    cplx = 2.0 if c["op"] == "kpoints" else 1.0
    if c["op"] != "ace" and _solves(c) * N * cplx * (4.0 * dense + 200.0) > EXACT_FLOPS:
        return None
    s = _inputs(c, seed)
    psi, dV = s["psi"], c["h"] ** 3
    if c["op"] == "solve":
        return _Exact(c)(psi)
    if c["op"] == "ace":
        M = dV * (psi @ s["vx"].T)
        R = torch.linalg.cholesky((-0.5 * (M + M.T)).cpu()).T.contiguous()
        xi = torch.linalg.inv(R).T.to(psi.device) @ s["vx"]
        return xi, M, -((dV * (s["phi"] @ xi.T)) @ xi)
    if c["op"] == "kpoints":
        th, wk = _theta(c)
        occ = s["occ"] if s["occ"] is not None else torch.ones(psi.shape[:2], dtype=torch.float64, device=psi.device)
        out = torch.zeros_like(psi)
        for k in range(len(th)):
            for q in range(len(th)):
                fl = _Exact(c, [th[k][a] - th[q][a] for a in range(3)])
                for v in range(c["n_orb"]):
                    phi = fl(psi[q].conj() * psi[k, v])
                    out[k, v] -= wk[q] * ((occ[q, :, None] * psi[q]) * phi).sum(0)
        e = sum(0.5 * dV * wk[k] * (occ[k][:, None] * (psi[k].conj() * out[k]).real).sum() for k in range(len(th)))
        return out, e.reshape(1)
    fl = _Exact(c)
    g = s["occ"] if s["occ"] is not None else torch.ones(c["n_orb"], dtype=torch.float64, device=psi.device)
    mp = _multipole_terms(c, dV) if c["l_max"] >= 0 else None
    out = torch.zeros_like(psi)
    e = torch.zeros(1, dtype=torch.float64, device=psi.device)
    for i in range(c["n_orb"]):
        for j0 in range(i, c["n_orb"], 64):
            js = slice(j0, min(j0 + 64, c["n_orb"]))
            rho = psi[i] * psi[js]
            phi = fl(rho if mp is None else rho + (rho @ mp[0].T) @ mp[1])
            gp = g[js, None] * phi
            out[i] -= (psi[js] * gp).sum(0)
            lo = 1 if j0 == i else 0  # the diagonal pair counts once
            out[js][lo:] -= g[i] * psi[i] * phi[lo:]
            t = (rho * gp).sum(1)
            e -= 0.5 * dV * g[i] * (2 * t.sum() - (t[0] if j0 == i else 0.0))
    if c["op"] == "grad":
        return e[0], 2 * dV * g[:, None] * out
    return out, e
