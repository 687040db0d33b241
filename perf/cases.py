"""Performance cases of the slab library: what its users have it do, at the sizes they do it.

The library's work is the Chebyshev-filtered eigensolver (apply_H, cheb_filter, rayleigh_ritz),
the Poisson solve with a bias, and their variants (batched bias sweep, Bloch wave vector, Gauss
quadrature potential, nonlocal projectors, gradients).  Meshes, vector counts and degrees are
those of the repository's workloads (6x6x16 cells p = 3, 16x16x48 p = 5 with 512 vectors,
12x12x40 p = 4, 8x8xH sweeps) and of its tests (ragged cell and vector counts, p = 2 to 6,
Neumann faces); every input comes from the seed alone.

`exact` restates each path in 64 bits with plain torch: assembled one-dimensional element
matrices applied along the axes, projectors as a dense matrix, and the Poisson problem solved
in the eigenbasis of the one-dimensional matrices.
"""
import math

import numpy as np
import torch

import paper_2504_00998_gb300 as fe
from paper_2504_00998_gb300 import autograd as fe_autograd
from workloads import HARTREE_PER_VOLT, Bias

DEV = torch.device("cuda", 0)
F64 = torch.float64
CELL = 2.0           # cell size (bohr) along every axis, as in the repository's workloads
NL_SIGMA, NL_CUT = 0.8, 2.6
LARGEST = 16 * 16 * 48 * 125 * 512 * 30   # cells x p^3 x vectors x degree of the largest case


# ---- the cases ------------------------------------------------------------------------------
def _case(name, kind, cells, p, nvec=0, degree=0, **more):
    return dict({"name": name, "kind": kind, "nx": cells[0], "ny": cells[1], "nz": cells[2], "p": p,
                 "nvec": nvec, "degree": degree}, **more)


def listed():
    return [
        # one H X inside a user's own small loop: launch and latency count
        _case("apply-small", "apply", (6, 6, 16), 3, 32, 1),
        # the plain double slab: one filter + Rayleigh-Ritz cycle
        _case("cycle-f64", "cycle", (6, 6, 16), 3, 32, 10),
        # an SCF filter call on a medium slab (block about the size of L2)
        _case("filter-p4", "filter", (12, 12, 40), 4, 64, 20),
        # the mixed-precision filter at full size
        _case("filter-large", "filter", (16, 16, 48), 5, 512, 30),
        # odd cell counts, an odd number of vectors in padded rows, one Neumann face
        _case("filter-ragged", "filter", (9, 7, 21), 6, 101, 12, neumann_top=True),
        # a bias sweep: independent slabs of uneven height filtered together
        _case("sweep", "sweep", (8, 8, 40), 4, 128, 20, slabs=24, nz_min=8),
        # one k-point of a Brillouin-zone sampling: complex blocks
        _case("kpoint", "filter", (16, 16, 16), 5, 128, 12, kx=0.1, ky=0.05),
        # the potential integrated by Gauss quadrature
        _case("quadrature", "filter", (16, 16, 16), 5, 256, 8, quad=True),
        # nonlocal pseudopotential projectors on every atom
        _case("nonlocal", "filter", (8, 8, 24), 5, 128, 15, nonlocal_=True),
        # the electrostatics of an SCF step: constant field, zero-Neumann
        _case("poisson-cef", "poisson", (16, 16, 48), 5, bias="cef"),
        # the same with the potential fixed on two planes
        _case("poisson-cpd", "poisson", (12, 12, 40), 4, bias="cpd"),
        # H X under autograd: forward, dL/dX and dL/dV
        _case("gradient", "gradient", (10, 10, 20), 3, 96, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["apply", "cycle", "filter", "filter", "filter", "ragged", "sweep", "kpoint",
                           "quad", "nonlocal", "poisson", "poisson", "gradient"])
        cells = (rng.randint(5, 20), rng.randint(5, 20), rng.randint(7, 48))
        p = rng.choice([2, 3, 4, 4, 5, 5, 6])
        nvec, degree = 4 * _log_int(rng, 4, 128), _log_int(rng, 6, 40)
        more = {}
        if kind in ("apply", "gradient"):
            c = _case("", kind, cells, p, nvec, 1)
        elif kind == "cycle":
            cells, p, nvec, degree = (rng.randint(5, 10), rng.randint(5, 10), rng.randint(8, 20)), rng.choice(
                [3, 4]), 2 * rng.randint(8, 32), rng.randint(8, 14)
            c = _case("", kind, cells, p, nvec, degree)
        elif kind == "sweep":
            c = _case("", kind, (rng.randint(5, 10), rng.randint(5, 10), rng.randint(16, 40)), rng.choice([3, 4, 5]),
                      4 * _log_int(rng, 8, 32), rng.randint(8, 24), slabs=rng.randint(4, 24), nz_min=8)
        elif kind == "poisson":
            bias = rng.choice(["cef", "cef", "cpd", "lcpd"])
            c = _case("", kind, cells, p, bias=bias)
        else:
            if kind == "ragged":
                nvec, more = nvec + rng.randint(1, 3), {"neumann_top": rng.random() < 0.5}
            elif kind == "kpoint":
                more = {"kx": round(rng.uniform(-0.2, 0.2), 3), "ky": round(rng.uniform(0.01, 0.2), 3)}
                nvec = max(8, nvec // 2 // 2 * 2)
            elif kind == "quad":
                more = {"quad": True}
            elif kind == "nonlocal":
                more = {"nonlocal_": True}
                cells = (rng.randint(5, 10), rng.randint(5, 10), rng.randint(10, 24))
            c = _case("", "filter", cells, p, nvec, degree, **more)
        del c["name"]
        # the quadrature and complex variants cost about twice the plain operator
        weight = 2 if kind in ("quad", "kpoint", "nonlocal", "sweep", "cycle") else 1
        cost = c["nx"] * c["ny"] * c["nz"] * p ** 3 * max(1, c["nvec"]) * max(1, c["degree"]) * c.get("slabs", 1)
        if weight * cost <= LARGEST / 2:
            return c


# ---- the one-dimensional rules -----------------------------------------------------------------
def _rules(p):
    """GLL nodes and weights, element matrices (stiffness, mass, gradient), Gauss points and
    weights, and the interpolation from the GLL nodes to the Gauss points."""
    leg = np.polynomial.legendre
    c = np.zeros(p + 1)
    c[p] = 1.0
    x = np.concatenate([[-1.0], np.sort(np.real(leg.legroots(leg.legder(c)))), [1.0]]) if p > 1 else np.array([-1.0, 1.0])
    for _ in range(3):   # Newton on (1 - x^2) P_p'(x) for the interior nodes
        d1, d2 = leg.legval(x[1:-1], leg.legder(c)), leg.legval(x[1:-1], leg.legder(c, 2)) if p > 1 else 1.0
        x[1:-1] -= d1 / d2
    w = 2.0 / (p * (p + 1) * leg.legval(x, c) ** 2)
    gx, gw = leg.leggauss(p + 1)

    def lagrange(t):
        L, D = np.ones((len(t), p + 1)), np.zeros((len(t), p + 1))
        for i in range(p + 1):
            for j in range(p + 1):
                if j != i:
                    f = (t - x[j]) / (x[i] - x[j])
                    D[:, i] = D[:, i] * f + L[:, i] / (x[i] - x[j])
                    L[:, i] = L[:, i] * f
        return L, D

    B, D = lagrange(gx)
    K = D.T @ (gw[:, None] * D)
    M = B.T @ (gw[:, None] * B)
    G = B.T @ (gw[:, None] * D)
    return x, w, K, M, G, gx, gw, B


class Grid:
    """The slab's tensor-product nodes; fields are [NZ, NY, NX, ...] over all z planes."""

    def __init__(self, cells, p):
        self.cells, self.p = cells, p
        self.x, self.w, self.K, self.M, self.G, self.gx, self.gw, self.B = _rules(p)
        self.n = (cells[0] * p, cells[1] * p, cells[2] * p + 1)
        self.L = tuple(CELL * c for c in cells)

    def t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=F64, device=DEV)

    def axis(self, d):
        """Node coordinates along axis d (0 x, 1 y, 2 z)."""
        one = (np.arange(self.cells[d])[:, None] + (self.x[None, :-1] + 1) / 2) * CELL
        return self.t(np.append(one.ravel(), self.L[2]) if d == 2 else one.ravel())

    def gauss_axis(self, d):
        return self.t(((np.arange(self.cells[d])[:, None] + (self.gx[None, :] + 1) / 2) * CELL).ravel())

    def mass1(self, d):
        m = np.tile(np.append(2 * self.w[0], self.w[1:-1]), self.cells[d])
        if d == 2:
            m = np.append(m, self.w[0])
            m[0] = self.w[0]
        return self.t(m * CELL / 2)

    def mass(self):
        return self.mass1(2)[:, None, None] * self.mass1(1)[None, :, None] * self.mass1(0)[None, None, :]

    def copies(self, d):
        """The global index of every cell's nodes along axis d."""
        i = (np.arange(self.cells[d])[:, None] * self.p + np.arange(self.p + 1)[None, :]).ravel()
        return torch.as_tensor(i % self.n[d], device=DEV)

    def blocks(self, A, U, dim):
        """The matrix A applied to every cell's copies along dimension dim."""
        A = self.t(A).to(U.dtype)
        s = U.shape
        lead, tail = int(np.prod(s[:dim], dtype=np.int64)), int(np.prod(s[dim + 1:], dtype=np.int64))
        V = torch.matmul(A, U.reshape(lead * (s[dim] // A.shape[1]), A.shape[1], tail))
        return V.reshape(s)

    def spread(self, U, d):
        return U.index_select(2 - d, self.copies(d))

    def gather(self, U, d):
        shape = list(U.shape)
        shape[2 - d] = self.n[d]
        return torch.zeros(shape, dtype=U.dtype, device=DEV).index_add_(2 - d, self.copies(d), U)

    def along(self, A, U, d):
        """The assembled one-dimensional operator of the element matrix A along axis d."""
        return self.gather(self.blocks(A, self.spread(U, d), 2 - d), d)

    def stiffness(self, U):
        """K U: the assembled stiffness (cubic cells of side CELL)."""
        a = CELL / 2
        my, ky = self.along(self.M, U, 1), self.along(self.K, U, 1)
        flat = self.along(self.K, my, 0) + self.along(self.M, ky, 0)
        return a * (self.along(self.M, flat, 2) + self.along(self.K, self.along(self.M, my, 0), 2))

    def gradient(self, U, kx, ky):
        """(kx Gx + ky Gy) U."""
        a = CELL * CELL / 4
        gx = self.along(self.G, self.along(self.M, U, 1), 0)
        gy = self.along(self.M, self.along(self.G, U, 1), 0)
        return a * self.along(self.M, kx * gx + ky * gy, 2)

    def quadrature(self, U, W):
        """The consistent potential matrix applied to U; W = w |J| V at the Gauss points."""
        for d in range(3):
            U = self.blocks(self.B, self.spread(U, d), 2 - d)
        U = U * W
        for d in range(3):
            U = self.gather(self.blocks(self.B.T, U, 2 - d), d)
        return U


def _grid(case, nz=None):
    return Grid((case["nx"], case["ny"], nz or case["nz"]), case["p"])


# ---- atoms and fields ------------------------------------------------------------------------
def _atoms(grid, rng):
    """A jittered stack of layers centred in the box: positions and charges."""
    nx, ny = (max(1, int(round(v / 4.0))) for v in grid.L[:2])
    layers = int(np.clip((grid.L[2] - 10.0) // 5.0, 1, 4))
    R = []
    for k in range(layers):
        off = 0.5 * (k % 2)
        z = grid.L[2] / 2 + (k - (layers - 1) / 2) * 2.5
        R += [((i + 0.5 + off) * grid.L[0] / nx, (j + 0.5 + off) * grid.L[1] / ny, z) for j in range(ny) for i in range(nx)]
    R = np.asarray(R) + rng.uniform(-0.2, 0.2, (len(R), 3))
    R[:, 0] %= grid.L[0]
    R[:, 1] %= grid.L[1]
    return R, np.full(len(R), 3.0)


def _radii(grid, axes, a, reach):
    """(slice of planes, squared distances [images][z, y, x]) of the nodes within `reach` of an
    atom in z; every periodic image that comes nearer than `reach` in x and y."""
    z = (axes[2] - a[2]).cpu().numpy()
    near = np.nonzero(np.abs(z) <= reach)[0]
    if not len(near):
        return None, []
    sl = slice(int(near[0]), int(near[-1]) + 1)

    def images(d):
        u = axes[d] - a[d]
        if grid.L[d] < 2 * reach:
            return [u + s * grid.L[d] for s in (-1, 0, 1)]
        return [u - grid.L[d] * torch.round(u / grid.L[d])]

    dz = (axes[2][sl] - a[2])[:, None, None] ** 2
    return sl, [dz + v[None, :, None] ** 2 + u[None, None, :] ** 2 for u in images(0) for v in images(1)]


def _gauss(r2, sigma):
    return torch.exp(-r2 / (2 * sigma * sigma)) / ((2 * math.pi) ** 1.5 * sigma ** 3)


def _screened(grid, axes, R, Z, sigma=0.5, rc=1.0):
    """V_loc - V_sm of the atoms: -Z erf(r / rc) / r + Z erf(r / (sqrt2 sigma)) / r."""
    out = torch.zeros([len(a) for a in (axes[2], axes[1], axes[0])], dtype=F64, device=DEV)
    s = math.sqrt(2) * sigma
    for a, q in zip(R, Z):
        sl, rs = _radii(grid, axes, a, 7.0)
        for r2 in rs:
            r = torch.sqrt(r2).clamp_min(1e-12)
            out[sl] += q * (torch.erf(r / s) - torch.erf(r / rc)) / r
    return out


def _density(grid, axes, R, Z, sigma, norm=None):
    """sum_a Z_a g_sigma; with `norm` (the lumped mass) each atom's part has the integral Z_a."""
    out = torch.zeros([len(a) for a in (axes[2], axes[1], axes[0])], dtype=F64, device=DEV)
    for a, q in zip(R, Z):
        sl, rs = _radii(grid, axes, a, 9.0 * sigma)
        g = sum(_gauss(r2, sigma) for r2 in rs)
        out[sl] += q * g / ((norm[sl] * g).sum() if norm is not None else 1.0)
    return out


def _sawtooth(z, E, Lz):
    """Slope -E on [0.1 Lz, 0.9 Lz], straight back to zero at both faces."""
    mid, end = -E * (z - Lz / 2), 0.4 * E * Lz
    return torch.where(z < 0.1 * Lz, end * z / (0.1 * Lz), torch.where(z > 0.9 * Lz, -end * (Lz - z) / (0.1 * Lz), mid))


def _potential(grid, axes, R, Z, rng):
    """A slab's V_eff: the atoms' wells, a smooth electrostatic part and the field."""
    V = _screened(grid, axes, R, Z)
    u = 2 * math.pi * axes[2] / grid.L[2]
    V += (-0.25 * (1 - torch.cos(u)) - _sawtooth(axes[2], -0.005, grid.L[2]))[:, None, None]
    c = rng.uniform(-0.1, 0.1, 4)
    for d, (k, q) in enumerate(((c[0], c[1]), (c[2], c[3]))):
        v = 2 * math.pi * axes[d] / grid.L[d]
        w = k * torch.cos(v) + q * torch.sin(v)
        V += w[None, None, :] if d == 0 else w[None, :, None]
    return V


# ---- operator inputs --------------------------------------------------------------------------
class Slab:
    """One Hamiltonian: grid, stored planes, potential, and what the variants need."""

    def __init__(self, case, seed, nz=None):
        rng = np.random.default_rng(seed)
        self.grid = g = _grid(case, nz)
        self.planes = slice(1, g.n[2] if case.get("neumann_top") else g.n[2] - 1)
        self.R, self.Z = _atoms(g, rng)
        self.quad, self.k = bool(case.get("quad")), (case.get("kx", 0.0), case.get("ky", 0.0))
        axes = [g.gauss_axis(d) if self.quad else g.axis(d) for d in range(3)]
        V = _potential(g, axes, self.R, self.Z, rng)
        self.root = torch.sqrt(g.mass())[self.planes]
        if self.quad:
            n, (cx, cy, cz) = case["p"] + 1, g.cells
            w = g.t(np.tile(g.gw, max(g.cells)))
            self.W = V * (CELL / 2) ** 3 * w[: cz * n, None, None] * w[None, : cy * n, None] * w[None, None, : cx * n]
            self.V = V.reshape(cz, n, cy, n, cx, n).permute(0, 2, 4, 1, 3, 5).reshape(cx * cy * cz, n ** 3).contiguous()
        else:
            self.V = V[self.planes].reshape(-1).contiguous()
        self.D = None
        if case.get("nonlocal_"):
            self.D = np.stack([rng.uniform(0.5, 1.5, len(self.R))] + 3 * [rng.uniform(-0.4, -0.1, len(self.R))], axis=1)
        self.n = self.root.numel()
        self.a, self.b, self.a0 = 0.0, 0.0, 0.0

    def apply(self, X):
        """Ht X for a block [n, m] (64 bits)."""
        g, m = self.grid, X.shape[1]
        U = torch.zeros((g.n[2], g.n[1], g.n[0], m), dtype=X.dtype, device=DEV)
        U[self.planes] = X.reshape(*self.root.shape, m) / self.root[..., None]
        Y = 0.5 * g.stiffness(U)
        if self.k != (0.0, 0.0):
            Y = Y - 1j * g.gradient(U, *self.k)
        if self.quad:
            Y = Y + g.quadrature(U, self.W[..., None])
        Y = (Y[self.planes] / self.root[..., None]).reshape(self.n, m)
        if not self.quad:
            Y = Y + self.V[:, None] * X
        if self.k != (0.0, 0.0):
            Y = Y + 0.5 * (self.k[0] ** 2 + self.k[1] ** 2) * X
        if self.D is not None:
            P = self.projectors()
            Y = Y + P @ (torch.as_tensor(self.D, device=DEV).reshape(-1, 1) * (P.T @ X))
        return Y

    def projectors(self):
        """M^1/2 p at the nodes: four columns (s, x, y, z) an atom."""
        if not hasattr(self, "_P"):
            g = self.grid
            axes = [g.axis(d) for d in range(3)]
            P = torch.zeros((len(self.R), 4, *self.root.shape), dtype=F64, device=DEV)
            for i, a in enumerate(self.R):
                d = [axes[k] - a[k] for k in range(3)]
                d = [d[k] - g.L[k] * torch.round(d[k] / g.L[k]) for k in range(2)] + [d[2][self.planes]]
                r2 = d[2][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[0][None, None, :] ** 2
                v = torch.where(r2 <= NL_CUT ** 2, torch.exp(-r2 / (2 * NL_SIGMA ** 2)), torch.zeros_like(r2)) * self.root
                P[i, 0], P[i, 1] = v, v * (d[0] / NL_SIGMA)[None, None, :]
                P[i, 2], P[i, 3] = v * (d[1] / NL_SIGMA)[None, :, None], v * (d[2] / NL_SIGMA)[:, None, None]
            self._P = P.reshape(4 * len(self.R), -1).T.contiguous()
        return self._P

    def bounds(self, seed, steps=16):
        """Lanczos bounds of the spectrum and the cut of the filter."""
        gen = torch.Generator(device=DEV).manual_seed(seed)
        v = torch.randn((self.n, 1), generator=gen, device=DEV, dtype=F64)
        if self.k != (0.0, 0.0):
            v = v.to(torch.complex128)
        v, old, al, be = v / v.norm(), torch.zeros_like(v), [], []
        for j in range(steps):
            f = self.apply(v) - (be[-1] * old if be else 0.0)
            al.append(torch.sum(v.conj() * f).real)
            f = f - al[-1] * v
            be.append(f.norm())
            old, v = v, f / be[-1]
        al, be = torch.stack(al).cpu().numpy(), torch.stack(be).cpu().numpy()
        ev = np.linalg.eigvalsh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
        self.a0, self.b = float(ev[0]), float(ev[-1] + be[-1])
        self.a = self.a0 + 0.03 * (self.b - self.a0)
        return self

    def mesh(self, case):
        m = fe.Mesh(self.grid.L, self.grid.cells, case["p"], (True, not case.get("neumann_top", False)))
        if self.k != (0.0, 0.0):
            m.set_kpoint(*self.k)
        if self.D is not None:
            m.set_nonlocal(self.R, np.full(len(self.R), NL_SIGMA), self.D, NL_CUT)
        if self.quad:
            m.set_potential_quad(self.V)
        else:
            m.set_potential(self.V)
        return m

    def filter(self, X, degree):
        """The scaled Chebyshev filter of the block X (64 bits)."""
        e, c = (self.b - self.a) / 2, (self.b + self.a) / 2
        s = e / (self.a0 - c)
        tau = 2 / s
        Y = (s / e) * (self.apply(X) - c * X)
        for _ in range(degree - 1):
            sn = 1 / (tau - s)
            X, Y = Y, (2 * sn / e) * (self.apply(Y) - c * Y) - s * sn * X
            s = sn
        return Y


def _block(n, nvec, seed, dtype):
    """N(0, 1) vectors; rows padded to 16 bytes where the count is odd."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    per = max(1, 16 // torch.empty(0, dtype=dtype).element_size())
    X = torch.zeros((n, -(-nvec // per) * per), dtype=dtype, device=DEV)[:, :nvec]
    for i in range(0, n, 1 << 18):
        X[i:i + (1 << 18)] = torch.randn((min(1 << 18, n - i), nvec), generator=gen, device=DEV, dtype=dtype)
    return X


def _sweep_heights(case):
    """The slabs' heights are part of the case, not of the inputs: the same for every seed."""
    rng = np.random.default_rng(1004)
    return [int(h) for h in rng.integers(case["nz_min"], case["nz"] + 1, case["slabs"])]


def _inputs(case, seed):
    """Slabs and blocks of an operator case, from the seed alone."""
    kind = case["kind"]
    if kind == "sweep":
        slabs = [Slab(case, seed + 101 * i, nz).bounds(seed + i) for i, nz in enumerate(_sweep_heights(case))]
        return slabs, [_block(s.n, case["nvec"], seed + 17 * i, torch.float32) for i, s in enumerate(slabs)]
    s = Slab(case, seed)
    if kind in ("filter", "cycle"):
        s.bounds(seed + 1)
    if kind == "cycle":
        # an SCF iteration filters the orthonormal block of the one before
        return [s], [torch.linalg.qr(_block(s.n, case["nvec"], seed + 2, F64))[0].contiguous()]
    dtype = torch.complex64 if s.k != (0.0, 0.0) else torch.float32
    X = [_block(s.n, case["nvec"], seed + 2, dtype)]
    if kind == "gradient":
        X.append(_block(s.n, case["nvec"], seed + 3, dtype))
    return [s], X


# ---- electrostatics inputs -----------------------------------------------------------------------
def _bias(case, grid):
    Lx, Ly, Lz = grid.L
    if case["bias"] == "cef":
        return Bias("cef", field=0.005)
    patch = ((0.25 * Lx, 0.25 * Ly), (0.5 * Lx, 0.5 * Ly)) if case["bias"] == "lcpd" else None
    return Bias("cpd", dV=0.5 * HARTREE_PER_VOLT, zA=2.0, zB=Lz - 2.0, patch=patch)


def _charges(case, seed):
    """Atoms and an electron density polarised against them, as a self-consistent one is."""
    rng = np.random.default_rng(seed)
    g = _grid(case)
    R, Z = _atoms(g, rng)
    axes = [g.axis(d) for d in range(3)]
    rho = _density(g, axes, R + rng.uniform(-0.1, 0.1, R.shape), Z, 1.0)
    rho *= Z.sum() / (rho * g.mass()).sum()
    return g, R, Z, rho


def _reference_poisson(case, seed):
    """phi and V_bare in 64 bits: the problem is diagonal in the generalised eigenbasis of the
    one-dimensional matrices (over the free planes along z)."""
    g, R, Z, rho = _charges(case, seed)
    bias, axes, mass = _bias(case, g), [g.axis(d) for d in range(3)], g.mass()
    vlms = _screened(g, axes, R, Z)
    f = 4 * math.pi * mass * (rho - _density(g, axes, R, Z, 0.5, norm=mass))
    z = axes[2]
    free = torch.ones(g.n[2], dtype=torch.bool, device=DEV)
    phi = torch.zeros_like(f)
    if bias.kind == "cef":
        f = f - mass * (f.sum() / mass.sum())
    else:
        lo, hi = z <= bias.zA + 1e-9, z >= bias.zB - 1e-9
        free = ~(lo | hi)
        phi[lo], phi[hi] = -vlms[lo], bias.dV - vlms[hi]
    lam, vec = [], []
    for d in range(3):
        eye = torch.eye(g.n[d], dtype=F64, device=DEV).reshape([g.n[d] if 2 - i == d else 1 for i in range(3)] + [g.n[d]])
        K, M = (g.along(A, eye, d).reshape(g.n[d], g.n[d]) for A in (g.K, g.M))
        if d == 2:
            K, M = K[free][:, free], M[free][:, free]
        C = torch.linalg.inv(torch.linalg.cholesky(M))
        w, q = torch.linalg.eigh(C @ K @ C.T)
        lam.append(w)
        vec.append(C.T @ q)
    den = CELL / 2 * (lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :])
    if bias.kind == "cef":
        den[0, 0, 0] = math.inf
    for _ in range(2):   # the second pass takes up the first one's rounding
        r = (f - g.stiffness(phi[..., None])[..., 0])[free]
        t = torch.einsum("zyx,zc,yb,xa->cba", r, *vec[::-1]) / den
        phi[free] += torch.einsum("cba,zc,yb,xa->zyx", t, *vec[::-1])
        if bias.kind == "cef":
            phi -= (mass * phi).sum() / mass.sum()
    vbare = phi + vlms
    if bias.kind == "cef":
        vbare = vbare + _sawtooth(z, bias.field, g.L[2])[:, None, None]
    return {"phi": phi.reshape(-1), "vbare": vbare[1:-1].reshape(-1)}


# ---- the measured calls -------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        g, R, Z, rho = _charges(case, seed)
        m = fe.Mesh(g.L, g.cells, case["p"])
        m.set_atoms(R, Z)
        return {"kind": kind, "mesh": m, "bias": _bias(case, g), "rho": rho.reshape(-1).contiguous()}
    slabs, X = _inputs(case, seed)
    meshes = [s.mesh(case) for s in slabs]
    st = {"kind": kind, "degree": case["degree"], "X0": X, "a": [s.a for s in slabs], "b": [s.b for s in slabs],
          "a0": [s.a0 for s in slabs]}
    if kind == "sweep":
        st["batch"] = fe.Batch(meshes)
    else:
        st["mesh"] = meshes[0]
    if kind in ("filter", "sweep", "cycle"):
        st["X"] = [torch.empty_strided(x.shape, x.stride(), dtype=x.dtype, device=DEV) for x in X]
    if kind == "apply":
        st["Y"] = torch.empty_like(X[0])
    if kind == "gradient":
        st["V"] = slabs[0].V.requires_grad_(True)
        X[0].requires_grad_(True)
    return st


def run(st):
    kind = st["kind"]
    if kind == "poisson":
        phi, vbare, _ = st["mesh"].poisson_solve(st["bias"], rho=st["rho"], rtol=1e-12)
        return {"phi": phi, "vbare": vbare}
    if kind == "apply":
        return st["mesh"].apply_H(st["X0"][0], st["Y"], prec=fe.FE_F32)
    if kind == "gradient":
        X, gY = st["X0"]
        Y = fe_autograd.apply_H(st["mesh"], X, st["V"], prec=fe.FE_F32)
        gX, gV = torch.autograd.grad(Y, [X, st["V"]], gY)
        return {"Y": Y.detach(), "gX": gX, "gV": gV}
    # the filter works in place: the user keeps the block it starts from
    torch._foreach_copy_(st["X"], st["X0"])
    if kind == "sweep":
        return st["batch"].cheb_filter(st["X"], st["degree"], st["a"], st["b"], st["a0"], prec=fe.FE_F32)
    X, prec = st["X"][0], fe.FE_F64 if kind == "cycle" else fe.FE_F32
    st["mesh"].cheb_filter(X, st["degree"], st["a"][0], st["b"][0], st["a0"][0], prec=prec)
    if kind == "cycle":
        return {"eig": st["mesh"].rayleigh_ritz(X, prec=prec), "X": X}
    return X


def work(case):
    """Bytes: every operator application reads the block and the previous iterate and writes
    the next one (a block does not fit on the chip); the potential once an application.
    Flops: the sum-factorised cell products, 12 (p + 1)^4 a cell and vector."""
    p, kind = case["p"], case["kind"]
    heights = _sweep_heights(case) if kind == "sweep" else [case["nz"]]
    cells = sum(case["nx"] * case["ny"] * h for h in heights)
    nodes = sum(case["nx"] * case["ny"] * p * p * (h * p - 1) for h in heights)
    cell = 12 * (p + 1) ** 4
    if kind == "poisson":
        # density in, phi and V_bare out; at least one residual of the double operator
        return {"bytes": 8 * 3 * nodes, "flops": cell * cells}
    lanes = case["nvec"] * (2 if "kx" in case else 1)
    size = 8 if kind == "cycle" else 4
    steps = case["degree"] if kind != "gradient" else 2
    per = 3 if kind in ("filter", "sweep", "cycle") else 2
    flops = cell * cells * lanes * steps
    if case.get("quad"):
        flops *= 2
    nbytes = size * nodes * lanes * per * steps + 8 * nodes * steps
    if kind == "cycle":
        flops += cell * cells * lanes + 6 * nodes * lanes * lanes
        nbytes += 3 * size * nodes * lanes
    if kind == "gradient":
        nbytes += 2 * size * nodes * lanes
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        # (a patch of fixed potential has no separable form)
        return None if case["bias"] == "lcpd" else _reference_poisson(case, seed)
    slabs, X = _inputs(case, seed)

    def wide(x):
        return x.to(torch.complex128 if x.is_complex() else F64)

    def chunked(s, x, f):
        # 0.4 GB of double columns at a time
        step = max(1, int(4e8 / 8 / s.n))
        return torch.cat([f(wide(x[:, i:i + step])) for i in range(0, x.shape[1], step)], dim=1)

    if kind == "apply":
        return chunked(slabs[0], X[0], slabs[0].apply)
    if kind == "gradient":
        s, (x, gy) = slabs[0], X
        return {"Y": chunked(s, x, s.apply), "gX": chunked(s, gy, s.apply), "gV": (wide(x) * wide(gy)).sum(1)}
    out = [chunked(s, x, lambda c, s=s: s.filter(c, case["degree"])) for s, x in zip(slabs, X)]
    if kind == "cycle":
        q = torch.linalg.qr(out[0])[0]
        # (the vectors' signs are free)
        return {"eig": torch.linalg.eigvalsh(q.T @ slabs[0].apply(q)), "X": None}
    return out if kind == "sweep" else out[0]
