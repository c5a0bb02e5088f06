"""The work that a user of this framework has it do, as cases to be timed.

Every case is one call of the public interface on a seeded synthetic density of
the kind the package's own workloads use (inputs.py): a rare-gas dimer, a
binding curve, a rare-gas monolayer on an orthogonal and on a hexagonal cell, a
rare-gas chain, a molecule and a metal slab with an adsorbed flake.  Atoms are
displaced a little by the seed, and the periodic densities carry seeded noise,
as theirs do.

The pair sums at precision "fp32" resolve single precision: the library states
1e-6 relative for the energy and 1e-5 of max|v| for the potential, although its
interface hands both back in 64-bit containers.  The programs here keep those
results as single-precision numbers, as a caller that asked for fp32 does; what
the fp64 path and the grid-level calls return stays in 64 bits.
"""
import functools
import math

import numpy as np
import torch

import paper_0810_2273_gb300 as V
from paper_0810_2273_gb300 import inputs

DEV = "cuda:0"

# operations per ordered pair interaction: 71 and 123 per unordered pair for E and
# for E + v (table branch: geometry, cell split, B-spline weights, 4 x 4 stencil,
# accumulation)
OPS_E, OPS_V = 35.5, 61.5


def _case(name, call, system, dims, precision="fp32", gradient="fd"):
    return {"name": name, "call": call, "system": system, "n0": dims[0], "n1": dims[1], "n2": dims[2],
            "precision": precision, "gradient": gradient}


def listed():
    return [
        # one energy of a small open dimer: the smallest call, launches and latency count
        _case("dimer_energy_fp32", "energy", "dimer", (24, 18, 18)),
        # the same question in double precision, on a ragged grid
        _case("dimer_energy_fp64", "energy", "dimer", (31, 23, 19), "fp64"),
        # a binding curve: 16 dimers and 2 single atoms of uneven size in one batch
        _case("binding_curve_fp32", "batched", "curve", (32, 24, 24)),
        # a molecule's energy as a term of a differentiable loss: forward and backward
        _case("molecule_autograd_fp32", "autograd", "molecule", (64, 64, 64)),
        # a monolayer's energy and potential, the headline size
        _case("monolayer_potential_fp32", "potential", "monolayer", (48, 84, 120)),
        # ... and on the coarse grid of a first look
        _case("monolayer_coarse_fp32", "potential", "monolayer", (24, 42, 60)),
        # ... and in double precision, to check the former against
        _case("monolayer_coarse_fp64", "potential", "monolayer", (24, 42, 60), "fp64"),
        # the energy on a skewed (hexagonal) cell
        _case("hexagonal_energy_fp32", "energy", "hex", (48, 48, 120)),
        # a dense metal slab with an adsorbate: large q0, many pairs at large D
        _case("slab_potential_fp32", "potential", "slab", (64, 56, 100)),
        # a chain, periodic along one axis, ragged grid, band-limited (FFT) gradient
        _case("chain_potential_fp32", "potential", "chain", (23, 71, 67), "fp32", "spectral"),
        # the semilocal energies of eq. 3 on a fine grid
        _case("semilocal_molecule", "semilocal", "molecule", (128, 112, 200), "fp64"),
        # the far field past the cutoff and its potential
        _case("far_tail_monolayer", "far_tail", "monolayer", (48, 84, 120), "fp64"),
    ]


# per kind of call: (call, system, precision, gradient, base grid, smallest and largest
# number of grid points relative to it); the pair sums grow with its square
_RANGES = [
    ("energy", "dimer", "fp32", "fd", (24, 18, 18), 0.25, 20.0),
    ("energy", "dimer", "fp64", "fd", (24, 18, 18), 0.25, 4.0),
    ("batched", "curve", "fp32", "fd", (32, 24, 24), 0.1, 1.5),
    ("autograd", "molecule", "fp32", "fd", (64, 64, 64), 0.02, 1.2),
    ("potential", "monolayer", "fp32", "fd", (48, 84, 120), 0.02, 0.9),
    ("energy", "monolayer", "fp32", "fd", (48, 84, 120), 0.02, 1.0),
    ("potential", "monolayer", "fp64", "fd", (24, 42, 60), 0.1, 1.1),
    ("energy", "hex", "fp32", "fd", (48, 48, 120), 0.03, 1.2),
    ("potential", "hex", "fp32", "fd", (48, 48, 120), 0.03, 1.1),
    ("potential", "slab", "fp32", "fd", (64, 56, 100), 0.05, 1.2),
    ("potential", "chain", "fp32", "spectral", (23, 71, 67), 0.1, 1.5),
    ("semilocal", "molecule", "fp64", "fd", (128, 112, 200), 0.02, 1.0),
    ("far_tail", "monolayer", "fp64", "fd", (48, 84, 120), 0.05, 1.0),
]


def draw(rng):
    call, system, precision, gradient, base, lo, hi = rng.choice(_RANGES)
    s = math.exp(rng.uniform(math.log(lo), math.log(hi))) ** (1.0 / 3.0)
    top = int(hi * base[0] * base[1] * base[2])
    while True:
        dims = [max(7, int(round(b * s)) + rng.choice((-1, 0, 0, 1))) for b in base]
        if dims[0] * dims[1] * dims[2] <= top:
            break
        s *= 0.99
    c = _case("", call, system, dims, precision, gradient)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _system(name):
    """Cell (rows), periodic axes, density cutoff, pair cutoff, noise and atoms
    [(position, [(amplitude, decay), ...])] of a system, undisplaced."""
    if name == "slab":
        atoms = []
        dz = 5.0 * math.sqrt(2.0 / 3.0)
        for k in range(4):
            for j in range(6):
                for i in range(6):
                    x = (i * 5.0 + (j % 2) * 2.5 + 2.5 * k) % 30.0
                    y = (j * 26.0 / 6.0 + 26.0 / 18.0 * k) % 26.0
                    atoms.append(((x, y, 8.0 + k * dz), inputs.single_exponential(11.0, 0.6)))
        for rad, cnt, Z in ((2.7, 6, 6.0), (5.0, 12, 6.0), (7.0, 12, 1.0)):
            for m in range(cnt):
                t = 2.0 * math.pi * m / cnt
                atoms.append(((15.0 + rad * math.cos(t), 13.0 + rad * math.sin(t), 8.0 + 3 * dz + 6.0),
                              inputs.single_exponential(Z, 0.4 + 0.3 * (m % 7) / 6.0)))
        return np.diag((30.0, 26.0, 48.0)), (True, True, False), 1e-5, 20.0, 0.005, atoms
    w = {"dimer": inputs.kr_dimer, "monolayer": inputs.xe_monolayer, "hex": inputs.xe_monolayer_hex,
         "chain": inputs.rare_gas_chain, "molecule": inputs.molecule24}[name]((4, 4, 4))
    cell = w["cell"] if "cell" in w else np.diag(w["lengths"])
    noise = 0.01 if any(w["periodic"]) else 0.0
    return np.asarray(cell), w["periodic"], w["n_cut"], w["r_cut"], noise, w["atoms"]


def _curve(dims):
    """The binding curve's instances: (dims, cell, atoms); 16 dimers 6 .. 12 bohr apart
    and one atom in the first and in the last cell, the grids growing with the
    separation from `dims` by a quarter of 8 and of 2 cells of 4 points."""
    shells = inputs.rare_gas_shells()
    f = [d / b for d, b in zip(dims, (32, 24, 24))]
    out = []
    for k in list(range(16)) + [0, 15]:
        s = 6.0 + 0.4 * k
        nat = (32 + 4 * int(8.0 * (s - 6.0) / 6.0 + 0.5),) + 2 * (24 + 4 * int(2.0 * (s - 6.0) / 6.0 + 0.5),)
        grid = tuple(max(5, int(round(n * x))) for n, x in zip(nat, f))
        L = np.array([0.5 * n for n in nat])
        c = L / 2.0
        x = (s / 2.0,) if len(out) >= 16 else (-s / 2.0, s / 2.0)
        atoms = [((c[0] + (0.0 if len(out) >= 16 else d), c[1], c[2]), shells) for d in x]
        out.append((grid, np.diag(L), atoms))
    return out


def _density(dims, cell, periodic, atoms, noise, seed, dev=DEV):
    """Exponential atoms on the grid, displaced by up to 0.05 bohr per axis, with
    multiplicative noise: FP64 [n0][n1][n2]."""
    rng = np.random.Generator(np.random.PCG64(seed))
    u = [torch.arange(d, dtype=torch.float64, device=dev) / d for d in dims]
    M = [[float(x) for x in row] for row in cell]
    orth = all(M[a][b] == 0.0 for a in range(3) for b in range(3) if a != b)
    if not orth:
        P = [u[0][:, None, None] * M[0][c] + u[1][None, :, None] * M[1][c] + u[2][None, None, :] * M[2][c]
             for c in range(3)]
    out = torch.zeros(tuple(dims), dtype=torch.float64, device=dev)
    shifts = [(-1, 0, 1) if p else (0,) for p in periodic]
    for pos, comps in atoms:
        pos = np.asarray(pos, dtype=np.float64) + rng.uniform(-0.05, 0.05, 3)
        reach = max(a * math.log(max(A / 1e-10, 1.0)) for A, a in comps)
        for s0 in shifts[0]:
            for s1 in shifts[1]:
                for s2 in shifts[2]:
                    c = pos + s0 * cell[0] + s1 * cell[1] + s2 * cell[2]
                    if orth:
                        gap = [max(0.0, -c[k], c[k] - M[k][k]) for k in range(3)]
                        if gap[0] ** 2 + gap[1] ** 2 + gap[2] ** 2 > reach ** 2:
                            continue
                        d = [(u[k] * M[k][k] - c[k]) ** 2 for k in range(3)]
                        r = torch.sqrt(d[0][:, None, None] + d[1][None, :, None] + d[2][None, None, :])
                    else:
                        r = torch.sqrt(sum((P[k] - c[k]) ** 2 for k in range(3)))
                    for A, a in comps:
                        out += A * torch.exp(r * (-1.0 / a))
    if noise:
        g = torch.Generator(device=dev)
        g.manual_seed(seed)
        out *= 1.0 + noise * (2.0 * torch.rand(out.shape, generator=g, dtype=torch.float64, device=dev) - 1.0)
    return out


@functools.lru_cache(maxsize=1)
def _table():
    """The kernel table a program builds (or loads) once: 400 x 200 nodes."""
    return V.Table.build(400, 30.0, 200, 0)


def _lengths(cell):
    d = np.diag(cell)
    return tuple(float(x) for x in d) if np.array_equal(np.diag(d), cell) else cell


def prepare(case, seed):
    st = {"case": case, "table": _table()}
    dims = (case["n0"], case["n1"], case["n2"])
    if case["system"] == "curve":
        inst = _curve(dims)
        st["ns"] = [_density(g, c, (False,) * 3, a, 0.0, 100 * seed + k) for k, (g, c, a) in enumerate(inst)]
        st["lengths"] = [_lengths(c) for _, c, _ in inst]
        st["periodic"] = [(False,) * 3] * len(inst)
        st["n_cut"], st["r_cut"] = 1e-6, 0.0
        return st
    cell, periodic, n_cut, r_cut, noise, atoms = _system(case["system"])
    n = _density(dims, cell, periodic, atoms, noise, seed)
    if case["call"] == "autograd":
        n = n.float().requires_grad_(True)  # the density a single-precision model puts out
    st.update(n=n, lengths=_lengths(cell), periodic=periodic, n_cut=n_cut, r_cut=r_cut)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    c, T = state["case"], state["table"]
    single = c["precision"] == "fp32"
    num = np.float32 if single else float
    if c["call"] == "batched":
        E, res = V.energy_batched(state["ns"], state["lengths"], state["periodic"], state["n_cut"], state["r_cut"], T,
                                  c["precision"])
        return {"E": E.astype(num), "pairs": res["pairs"]}
    n, args = state["n"], (state["lengths"], state["periodic"], state["n_cut"], state["r_cut"])
    if c["call"] == "energy":
        E, res = V.energy(n, *args, T, c["precision"], gradient=c["gradient"])
        return {"E": num(E), "pairs": res["pairs"], "n_active": res["n_active"]}
    if c["call"] == "potential":
        E, v, res = V.potential(n, *args, T, c["precision"], gradient=c["gradient"])
        return {"E": num(E), "v": v.float() if single else v, "pairs": res["pairs"], "n_active": res["n_active"]}
    if c["call"] == "autograd":
        spec = dict(lengths=args[0], periodic=args[1], n_cut=args[2], r_cut=args[3], table=T, precision=c["precision"])
        E = V.nonlocal_energy(n.double(), spec).float()
        (g,) = torch.autograd.grad(E, n)
        return {"E": E.detach(), "grad": g}
    if c["call"] == "semilocal":
        r = V.semilocal(n, args[0], args[1], gradient=c["gradient"])
        return {k: r[k] for k in ("Ex_lda", "Ec_lda", "Ex_pbe", "Ec_pbe", "Ex_revpbe", "n_points")}
    r, v = V.far_tail(n, *args, want_v=True)
    return {"T": r["T"], "v": v, "n_active": r["n_active"]}


# ---------------------------------------------------------------------------
# the least work of a pass
# ---------------------------------------------------------------------------
def _count(dims, cell, periodic, atoms, n_cut, r_cut, pairs=True):
    """Active points and ordered pair interactions, estimated on a coarse grid."""
    N = dims[0] * dims[1] * dims[2]
    f = min(1.0, (6000.0 / N) ** (1.0 / 3.0))
    cd = [max(4, int(round(d * f))) for d in dims]
    n = _density(cd, cell, periodic, atoms, 0.0, 0, "cpu").numpy()
    act = np.argwhere(n >= n_cut)
    n_act = len(act) * N / float(n.size)
    if not pairs:
        return n_act, 0.0
    if r_cut <= 0.0:
        return n_act, n_act ** 2
    P = (act / np.asarray(cd, dtype=np.float64)) @ cell
    Q = P[:: max(1, len(P) // 300)]
    cnt = 0
    m = [range(-3, 4) if p else (0,) for p in periodic]
    for a in m[0]:
        for b in m[1]:
            for c in m[2]:
                L = a * cell[0] + b * cell[1] + c * cell[2]
                d2 = ((Q[:, None, :] - P[None, :, :] + L) ** 2).sum(-1)
                cnt += int((d2 <= r_cut * r_cut).sum())
    return n_act, cnt / float(len(Q) * len(P)) * n_act ** 2


def work(case):
    dims = (case["n0"], case["n1"], case["n2"])
    N = dims[0] * dims[1] * dims[2]
    if case["call"] == "batched":
        b = f = 0.0
        for g, cell, atoms in _curve(dims):
            n_act, pairs = _count(g, cell, (False,) * 3, atoms, 1e-6, 0.0)
            b += 8.0 * g[0] * g[1] * g[2]
            f += OPS_E * pairs
        return {"bytes": b, "flops": f}
    cell, periodic, n_cut, r_cut, _, atoms = _system(case["system"])
    n_act, pairs = _count(dims, cell, periodic, atoms, n_cut, r_cut, case["call"] not in ("semilocal", "far_tail"))
    if case["call"] == "energy":
        return {"bytes": 8.0 * N, "flops": OPS_E * pairs}
    if case["call"] in ("potential", "autograd"):
        return {"bytes": (16.0 if case["call"] == "potential" else 8.0) * N, "flops": OPS_V * pairs}
    if case["call"] == "semilocal":
        return {"bytes": 8.0 * N, "flops": 250.0 * N}
    # the far field: an exponential and two sums per point and quadrature node, both ways
    return {"bytes": 16.0 * N, "flops": 2.0 * 165 * 25.0 * n_act}


# ---------------------------------------------------------------------------
# the same outputs from plain torch in 64 bits
# ---------------------------------------------------------------------------
def _roll_grad(f, dims, B):
    """4th-order periodic central differences along the grid axes, to Cartesian."""
    g = [torch.zeros_like(f) for _ in range(3)]
    for a in range(3):
        d = (8.0 * (torch.roll(f, -1, a) - torch.roll(f, 1, a)) - (torch.roll(f, -2, a) - torch.roll(f, 2, a))) / 12.0
        for c in range(3):
            if B[a][c] != 0.0:
                g[c] += d * (dims[a] * float(B[a][c]))
    return g


def _fft_grad(f, dims, B):
    """The band-limited derivative along each axis (Nyquist to zero), to Cartesian."""
    g = [torch.zeros_like(f) for _ in range(3)]
    for a in range(3):
        N = dims[a]
        m = torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device=f.device)
        if N % 2 == 0:
            m[N // 2] = 0.0
        shape = [1, 1, 1]
        shape[a] = N
        d = torch.fft.ifft(torch.fft.fft(f, dim=a) * (2j * math.pi * m).reshape(shape), dim=a).real
        for c in range(3):
            if B[a][c] != 0.0:
                g[c] += d * float(B[a][c])
    return g


def _pw92(rs):
    """Perdew-Wang 1992 correlation energy per electron (unpolarised) and d/d rs."""
    A, a1, b1, b2, b3, b4 = 0.031091, 0.21370, 7.5957, 3.5876, 1.6382, 0.49294
    s = torch.sqrt(rs)
    den = 2.0 * A * (b1 * s + b2 * rs + b3 * rs * s + b4 * rs * rs)
    dden = A * (b1 / s + 2.0 * b2 + 3.0 * b3 * s + 4.0 * b4 * rs)
    lg = torch.log1p(1.0 / den)
    pre = -2.0 * A * (1.0 + a1 * rs)
    return pre * lg, -2.0 * A * a1 * lg - pre * dden / (den * (den + 1.0))


def _q0(n, g):
    """q0 (Dion eqs. 11-12, Zab = -0.8491) and its partials at points of density n."""
    Z = -0.8491
    kF = (3.0 * math.pi ** 2 * n) ** (1.0 / 3.0)
    rs = (3.0 / (4.0 * math.pi * n)) ** (1.0 / 3.0)
    ec, de = _pw92(rs)
    g2 = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
    w = 1.0 / (kF * n * n)
    q = kF - Z / 36.0 * g2 * w - 4.0 * math.pi / 3.0 * ec
    qn = kF / (3.0 * n) + 7.0 * Z / 108.0 * g2 * w / n + 4.0 * math.pi / 3.0 * de * rs / (3.0 * n)
    return q, qn, [-Z / 18.0 * w * x for x in g]


def _spline_matrix(m):
    """Coefficients (m + 2) of the cubic B-spline through m equidistant values, with zero
    slope at the first and zero curvature at the last: rows of the inverse system."""
    S = np.zeros((m + 2, m + 2))
    S[0, 0], S[0, 2] = -1.0, 1.0
    for k in range(m):
        S[k + 1, k:k + 3] = 1.0 / 6.0, 4.0 / 6.0, 1.0 / 6.0
    S[m + 1, m - 1:m + 2] = 1.0, -2.0, 1.0
    return np.linalg.inv(S)[:, 1:m + 1]


def _weights(t):
    """Cubic B-spline weights and derivatives of four neighbours at offset t."""
    s = 1.0 - t
    w = [s ** 3 / 6.0, (3.0 * t ** 3 - 6.0 * t ** 2 + 4.0) / 6.0, (-3.0 * t ** 3 + 3.0 * t ** 2 + 3.0 * t + 1.0) / 6.0,
         t ** 3 / 6.0]
    d = [-s ** 2 / 2.0, (9.0 * t ** 2 - 12.0 * t) / 6.0, (-9.0 * t ** 2 + 6.0 * t + 3.0) / 6.0, t ** 2 / 2.0]
    return w, d


class _Kernel:
    """phi(q_i, q_j, r) and r dphi/dd1 of a node table (D up to Dmax, delta = l/nd):
    bicubic spline, linear past the last delta node, g(delta*) times the asymptote
    past Dmax."""

    C = 12.0 * (4.0 * math.pi / 9.0) ** 3

    def __init__(self, nodes, Dmax):
        self.nD, self.nd = nodes.shape
        self.Dmax = Dmax
        c = _spline_matrix(self.nD) @ nodes @ _spline_matrix(self.nd).T
        self.c = torch.from_numpy(np.ascontiguousarray(c)).to(DEV).reshape(-1)
        dl = np.arange(self.nd) / self.nd
        p17 = -self.C / (Dmax ** 6 * (1.0 + dl) ** 2 * (1.0 - dl) ** 2 * ((1.0 + dl) ** 2 + (1.0 - dl) ** 2))
        rho = nodes[-1] / p17
        self.rho0 = float(rho[0])
        self.rho = torch.from_numpy(_spline_matrix(self.nd) @ rho).to(DEV)

    def _delta(self, d):
        x = d * self.nd
        xc = x.clamp(0.0, self.nd - 1.0)
        l = xc.floor().clamp(max=self.nd - 2)
        w, dw = _weights(xc - l)
        e = x.clamp(min=0.0) - xc
        return l.long(), [a + e * b for a, b in zip(w, dw)], dw

    def __call__(self, r, qi, qj):
        sq = qi + qj
        D = 0.5 * r * sq
        ds = (qi - qj) / sq
        l, wd, dwd = self._delta(ds.abs())
        x = (D * ((self.nD - 1) / self.Dmax)).clamp(max=self.nD - 1.0)
        k = x.floor().clamp(max=self.nD - 2)
        wD, dwD = _weights(x - k)
        at = k.long() * (self.nd + 2) + l
        phi = torch.zeros_like(r)
        pD = torch.zeros_like(r)
        pd = torch.zeros_like(r)
        for m in range(4):
            row = torch.zeros_like(r)
            drow = torch.zeros_like(r)
            for j in range(4):
                c = self.c[at + (m * (self.nd + 2) + j)]
                row += wd[j] * c
                drow += dwd[j] * c
            phi += wD[m] * row
            pD += dwD[m] * row
            pd += wD[m] * drow
        pD *= (self.nD - 1) / self.Dmax
        pd *= self.nd * torch.sign(ds)
        u = 0.5 * r * pD + (1.0 - ds) / sq * pd
        far = (D > self.Dmax).nonzero()[:, 0]
        if len(far):
            r, qi, qj, D = r[far], qi[far], qj[far], D[far]
            s2 = qi ** 2 + qj ** 2
            p17 = -self.C / (r ** 6 * qi ** 2 * qj ** 2 * s2)
            ts = 1.0 - r * torch.minimum(qi, qj) / self.Dmax
            l, w, dw = self._delta(ts)
            rho = sum(w[j] * self.rho[l + j] for j in range(4))
            dr = sum(dw[j] * self.rho[l + j] for j in range(4)) * self.nd * (ts > 0.0)
            D2 = (self.Dmax / D) ** 2
            g = rho + (1.0 - self.rho0) * (1.0 - D2)
            dg = (1.0 - self.rho0) * D2 * r / D - (qi < qj) * dr * r / self.Dmax
            phi[far] = g * p17
            u[far] = g * -2.0 * p17 * (1.0 / qi + qi / s2) + p17 * dg
        return phi, u


def _pair_sums(P, q, n, L, rc, K, want_U):
    """A_i = sum_{j, L} n_j phi and U_i = n_i sum n_j r dphi/dd1 over Cartesian points P
    and image vectors L within rc (all pairs when rc <= 0), and the ordered pairs."""
    m = len(q)
    A = torch.zeros(m, dtype=torch.float64, device=DEV)
    U = torch.zeros_like(A)
    pairs = 0
    rc2 = rc * rc * (1.0 + 1e-12) if rc > 0.0 else math.inf
    step = max(1, (1 << 24) // m)
    lo, hi = P.min(0).values, P.max(0).values
    for i0 in range(0, m, step):
        Pi = P[i0:i0 + step]
        for v in L:
            gap = torch.maximum((Pi.min(0).values + v) - hi, lo - (Pi.max(0).values + v)).clamp(min=0.0)
            if float((gap ** 2).sum()) > rc2 * 1.001:
                continue
            r2 = torch.zeros((len(Pi), m), dtype=torch.float64, device=DEV)
            for c in range(3):
                r2 += ((Pi[:, c, None] + v[c]) - P[None, :, c]) ** 2
            i, j = (r2 <= rc2).nonzero(as_tuple=True)
            if not len(i):
                continue
            r = r2[i, j].sqrt()
            pairs += int((r > 0.0).sum())
            phi, u = K(r, q[i0:i0 + step][i], q[j])
            A[i0:i0 + step].index_add_(0, i, phi * n[j])
            if want_U:
                U[i0:i0 + step].index_add_(0, i, u * n[j])
    return A, U * n, pairs


def _exact_tail(n, q, dV, cell, dims, rc, act):
    """Far field past rc with periodic x, y: T and the sums S0, S1 per active point
    (trapezoid in ln s with a fine step)."""
    area = float(np.linalg.norm(np.cross(cell[0], cell[1])))
    dz = float(cell[2][2]) / dims[2]
    p = act[:, 2]
    z = torch.arange(dims[2], dtype=torch.float64, device=DEV)
    R = ((z[:, None] - z[None, :]).abs() * dz).clamp(min=rc)
    Kpp = 2.0 * math.pi / area / (4.0 * R ** 4)
    u = q * q
    h = 0.1
    x0, x1 = math.log(1e-19 / (2.0 * float(u.max()))), math.log(60.0 / (2.0 * float(u.min())))
    T, S0, S1 = 0.0, torch.zeros_like(q), torch.zeros_like(q)
    for k in range(int(math.ceil((x1 - x0) / h)) + 1):
        s = math.exp(x0 + h * k)
        e = torch.exp(-u * s)
        F = torch.zeros(dims[2], dtype=torch.float64, device=DEV).index_add_(0, p, n / u * e)
        G = Kpp @ F
        T += h * s * float(F @ G)
        t = h * s * e * G[p]
        S0 += t
        S1 += s * t
    C = _Kernel.C
    return -0.5 * dV * dV * C * T, -C * S0 / u, 2.0 * C * n * q * (S0 / (u * u) + S1 / u)


def exact(case, seed):
    dims = (case["n0"], case["n1"], case["n2"])
    call = case["call"]
    if call == "batched":
        return None
    cell, periodic, n_cut, r_cut, noise, atoms = _system(case["system"])
    if call not in ("semilocal", "far_tail") and work(case)["flops"] / OPS_E > 6e9:
        return None
    n = _density(dims, cell, periodic, atoms, noise, seed)
    if call == "autograd":
        n = n.float().double()
    N = n.numel()
    dV = abs(float(np.linalg.det(cell))) / N
    B = np.linalg.inv(cell).T
    grad = _fft_grad if case["gradient"] == "spectral" else _roll_grad
    g = grad(n, dims, B)
    if call == "semilocal":
        m = n > 0.0
        x, g2 = n[m], (g[0] ** 2 + g[1] ** 2 + g[2] ** 2)[m]
        kF = (3.0 * math.pi ** 2 * x) ** (1.0 / 3.0)
        ec, _ = _pw92((3.0 / (4.0 * math.pi * x)) ** (1.0 / 3.0))
        ex = -3.0 * kF / (4.0 * math.pi)
        s2 = g2 / (2.0 * kF * x) ** 2
        beta, gam = 0.06672455060314922, (1.0 - math.log(2.0)) / math.pi ** 2
        mu = beta * math.pi ** 2 / 3.0
        t2 = g2 * math.pi / (16.0 * kF * x * x)
        At = beta / gam / torch.expm1(-ec / gam) * t2
        H = gam * torch.log1p(beta / gam * t2 * (1.0 + At) / (1.0 + At + At * At))
        F = [1.0 + k - k / (1.0 + mu * s2 / k) for k in (0.804, 1.245)]
        e = [ex, ec, ex * F[0], ec + H, ex * F[1]]
        out = dict(zip(("Ex_lda", "Ec_lda", "Ex_pbe", "Ec_pbe", "Ex_revpbe"), [dV * float((x * y).sum()) for y in e]))
        out["n_points"] = None
        return out
    mask = n >= n_cut
    act = mask.nonzero()
    nm = n[mask]
    q, qn, qg = _q0(nm, [x[mask] for x in g])
    if call == "far_tail":
        E, A, U = _exact_tail(nm, q, dV, cell, dims, r_cut, act)
    else:
        P = sum((act[:, a].double() / dims[a])[:, None] * torch.tensor(cell[a], device=DEV) for a in range(3))
        m = [range(-4, 5) if p else (0,) for p in periodic]
        ext = [r_cut * float(np.linalg.norm(B[a])) + 1.0 for a in range(3)]
        L = [torch.tensor(a * cell[0] + b * cell[1] + c * cell[2], dtype=torch.float64, device=DEV)
             for a in m[0] if abs(a) <= ext[0] for b in m[1] if abs(b) <= ext[1] for c in m[2] if abs(c) <= ext[2]]
        T = _table()
        K = _Kernel(T.nodes, T.info()[1])
        A, U, pairs = _pair_sums(P, q, nm, L, r_cut, K, call != "energy")
        E = 0.5 * dV * dV * float((nm * A).sum())
        if call == "energy":
            return {"E": E, "pairs": None, "n_active": None}
    # v = dV (chi (A + U dq0/dn) - div(U dq0/dgrad n)), the transpose of the gradient
    v = torch.zeros_like(n)
    v[mask] = A + U * qn
    for c in range(3):
        w = torch.zeros_like(n)
        w[mask] = U * qg[c]
        v -= grad(w, dims, B)[c]
    v *= dV
    if call == "far_tail":
        return {"T": E, "v": v, "n_active": None}
    if call == "autograd":
        return {"E": E, "grad": v * dV}
    return {"E": E, "v": v, "pairs": None, "n_active": None}
