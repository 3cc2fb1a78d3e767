"""What a user of this library has it do, as measurable cases.

Every case is one call of a public entry point (``rpa_probe_density``, ``rpa_energy_density``,
``rpa_chi0``, ``rpa_interpolate``) on a synthetic cell of the kinds that the benchmark and the
tests use: Si-like cells with s/p projectors, rock-salt LiH-like cells without projectors, a
Gaussian cluster between Dirichlet walls, and the small periodic toy cell.  The cells, their
ground states and the sampled probe-points are made on the GPU from the seed.

Whole Lanczos runs are in the FP64 form.  The mixed form's solves stop at a loose tolerance
after FP32 iterations whose sums have no fixed order, so single numbers at the end of a
Lanczos run differ from run to run by amounts that vary a lot; its cases return the whole
field chi0 u instead, over many solves.  (Its iteration counts are no result and vary too.)
"""
import math
from fractions import Fraction

import numpy as np
import torch

import paper_2609_16408_gb300 as R

DEV = "cuda"
F64 = torch.float64


# -------------------------------------------------------------------------------------------
# cases
# -------------------------------------------------------------------------------------------
def listed():
    return [
        # one probe-point of the toy cell in the FP64 form: the smallest solve, all latency
        dict(name="toy_point_fp64", kind="points", cell="toy", nx=12, ny=12, nz=12, cx=1, cy=1,
             cz=1, states=8, radius=6, precision="fp64", nw=8, nl=20, tol=1e-10, count=1),
        # a whole E_c of the toy cell (every coarse point and frequency, interpolation)
        dict(name="toy_energy_fp64", kind="energy", cell="toy", nx=12, ny=12, nz=12, cx=1, cy=1,
             cz=1, states=8, radius=6, precision="fp64", nw=4, nl=4, tol=1e-10, stride=3),
        # sampled probe-points of the 8-atom Si-like cell in the plain FP64 form, which gives
        # the reference values for the mixed form
        dict(name="si8_points_fp64", kind="points", cell="si", nx=26, ny=26, nz=26, cx=1, cy=1,
             cz=1, states=16, radius=6, precision="fp64", nw=10, nl=2, tol=1e-8, count=10),
        # the (LiH)32-like cell without projectors at the settings of the paper's LiH runs
        dict(name="lih32_points_fp64", kind="points", cell="lih", nx=32, ny=32, nz=32, cx=2, cy=2,
             cz=2, states=64, radius=6, precision="fp64", nw=8, nl=2, tol=0.1, count=8),
        # chi0 on a wave of vectors, the step that a Lanczos run in the mixed form consists of,
        # on the 8-atom cell
        dict(name="si8_chi0", kind="chi0", cell="si", nx=26, ny=26, nz=26, cx=1, cy=1, cz=1,
             states=16, radius=6, precision="mixed", nw=4, nl=1, tol=1e-8, count=20),
        # 16 atoms on an odd, uneven grid (a spacing chosen by convergence, not by tiles)
        dict(name="si16_odd_chi0", kind="chi0", cell="si", nx=27, ny=25, nz=53, cx=1, cy=1, cz=2,
             states=32, radius=6, precision="mixed", nw=4, nl=1, tol=1e-8, count=10),
        # one vector of the 32-atom cell: a user looking at a single point
        dict(name="si32_one_chi0", kind="chi0", cell="si", nx=26, ny=52, nz=52, cx=1, cy=2, cz=2,
             states=64, radius=6, precision="mixed", nw=10, nl=1, tol=1e-4, count=1),
        # a molecule-like cluster between Dirichlet walls
        dict(name="cluster_chi0", kind="chi0", cell="cluster", nx=40, ny=40, nz=40, cx=1, cy=1,
             cz=1, states=24, radius=6, precision="mixed", nw=4, nl=1, tol=1e-4, count=8),
        # the 64-atom cell on the 40^3 grid at the tolerance of the paper's Si64 run
        dict(name="si64_40_chi0", kind="chi0", cell="si", nx=40, ny=40, nz=40, cx=2, cy=2, cz=2,
             states=128, radius=6, precision="mixed", nw=8, nl=1, tol=0.1, count=16),
        # the 64-atom cell on the 52^3 grid, ten frequencies: the benchmark's headline
        # workload and the largest case
        dict(name="si64_52_chi0", kind="chi0", cell="si", nx=52, ny=52, nz=52, cx=2, cy=2, cz=2,
             states=128, radius=6, precision="mixed", nw=10, nl=1, tol=1e-4, count=10),
        # interpolation of a finished coarse array (10 frequencies) to the fine grid and E_c
        dict(name="interp_52", kind="interp", cell="none", nx=52, ny=52, nz=52, nw=10, stride=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["si", "si", "si", "si", "si", "cluster", "toy", "fp64", "interp"])
    if kind == "interp":
        n = [_log_int(rng, 12, 52) for _ in range(3)]
        return dict(kind="interp", cell="none", nx=n[0], ny=n[1], nz=n[2],
                    nw=rng.choice([4, 8, 10]), stride=rng.choice([1, 2, 3]))
    if kind == "toy":
        n = [rng.randint(12, 16) for _ in range(3)]
        return dict(kind="points", cell="toy", nx=n[0], ny=n[1], nz=n[2], cx=1, cy=1, cz=1,
                    states=8, radius=rng.choice([4, 6]), precision="fp64", nw=8,
                    nl=rng.randint(4, 20), tol=1e-10, count=_log_int(rng, 1, 32))
    if kind == "fp64":
        c = rng.choice([(1, 1, 1), (1, 1, 2)])
        cell = rng.choice(["si", "lih"])
        n = [rng.randint(20, 26) * k if cell == "si" else rng.randint(14, 17) * k for k in c]
        return dict(kind="points", cell=cell, nx=n[0], ny=n[1], nz=n[2], cx=c[0], cy=c[1],
                    cz=c[2], states=(16 if cell == "si" else 8) * c[2], radius=6,
                    precision="fp64", nw=8, nl=rng.randint(1, 2), tol=1e-8,
                    count=_log_int(rng, 1, 8))
    if kind == "cluster":
        n = [rng.randint(32, 40) for _ in range(3)]
        return dict(kind="chi0", cell="cluster", nx=n[0], ny=n[1], nz=n[2], cx=1, cy=1, cz=1,
                    states=24, radius=6, precision="mixed", nw=4, nl=1, tol=1e-4,
                    count=rng.randint(6, 9))
    # the small cells are solved tighter: they are the ones that convergence is studied on
    c = rng.choice([(1, 1, 1), (1, 1, 2), (1, 2, 2), (2, 2, 2)])
    n = [rng.randint(20, 26) * k - rng.choice([0, 0, 1]) for k in c]
    states = 16 * c[0] * c[1] * c[2]
    if states <= 32:
        nw, tol, count = 4, 1e-8, _log_int(rng, 8, 20)
    else:
        # at most the work of the largest listed case: ten vectors of 128 states on 52^3
        most = 52 ** 3 * 128 * 10 // (n[0] * n[1] * n[2] * states)
        nw, tol = 10, rng.choice([0.1, 1e-3, 1e-4] if states == 128 else [1e-3, 1e-4])
        count = _log_int(rng, 1, min(20, most))
    return dict(kind="chi0", cell="si", nx=n[0], ny=n[1], nz=n[2], cx=c[0], cy=c[1], cz=c[2],
                states=states, radius=6, precision="mixed", nw=nw, nl=1, tol=tol, count=count)


# -------------------------------------------------------------------------------------------
# the discrete problem: grid, wells, projectors, ground state
# -------------------------------------------------------------------------------------------
def _weights(radius):
    """Central second-derivative weights from the moment conditions, exactly."""
    m = radius + 1
    a = []
    for k in range(0, 2 * radius + 1, 2):
        row = [Fraction(1 if k == 0 else 0)] + [Fraction(2 * j ** k) for j in range(1, m)]
        a.append(row + [Fraction(2 if k == 2 else 0)])
    for c in range(m):
        p = next(i for i in range(c, m) if a[i][c] != 0)
        a[c], a[p] = a[p], a[c]
        a[c] = [v / a[c][c] for v in a[c]]
        for i in range(m):
            if i != c and a[i][c] != 0:
                a[i] = [x - a[i][c] * y for x, y in zip(a[i], a[c])]
    return [float(a[i][m]) for i in range(m)]


def _lap1d(n, h, periodic, radius):
    w = _weights(radius)
    L = np.zeros((n, n))
    for i in range(n):
        L[i, i] += w[0]
        for m in range(1, radius + 1):
            for j in (i + m, i - m):
                if periodic:
                    L[i, j % n] += w[m]
                elif 0 <= j < n:
                    L[i, j] += w[m]
    return L / (h * h)


def _diamond(c):
    fcc = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    basis = np.concatenate([fcc, fcc + 0.25])
    return np.concatenate([basis + [i, j, k] for i in range(c[0]) for j in range(c[1])
                           for k in range(c[2])])


def _rocksalt(c):
    fcc = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    off = [np.array([i, j, k]) for i in range(c[0]) for j in range(c[1]) for k in range(c[2])]
    return (np.concatenate([fcc + o for o in off]),
            np.concatenate([fcc + [0.5, 0, 0] + o for o in off]))


class _Cell:
    """Grid, V_loc, projector groups and H of one synthetic cell."""

    def __init__(self, case, rng):
        self.n = n = (case["nx"], case["ny"], case["nz"])
        c = (case["cx"], case["cy"], case["cz"])
        kind = case["cell"]
        self.periodic = kind != "cluster"
        self.radius = case["radius"]
        if kind == "si":
            a = 10.26
            site = _diamond(c) * a
            pos = site + 0.1 * a * math.sqrt(3) / 4 * rng.uniform(-0.5, 0.5, site.shape)
            depth = rng.uniform(1.2, 1.8, len(pos))
            sigma = np.full(len(pos), 1.0)
        elif kind == "lih":
            a = 7.71
            li, hy = _rocksalt(c)
            site = np.concatenate([li, hy]) * a
            pos = site + 0.05 * a * rng.uniform(-0.5, 0.5, site.shape)
            depth = np.concatenate([rng.uniform(4.5, 5.5, len(li)), rng.uniform(1.3, 1.7, len(hy))])
            sigma = np.concatenate([np.full(len(li), 0.5), np.full(len(hy), 0.8)])
        elif kind == "cluster":
            a = 16.0
            pos = 8.0 + rng.uniform(-3.0, 3.0, (12, 3))
            depth = rng.uniform(1.2, 1.8, 12)
            sigma = np.full(12, 1.0)
        else:
            a = 6.0
            pos = rng.uniform(0.0, a, (4, 3))
            depth = rng.uniform(0.5, 2.0, 4)
            sigma = rng.uniform(0.8, 1.5, 4)
        L = [a * k for k in c]
        self.h = tuple(L[i] / (n[i] if self.periodic else n[i] + 1) for i in range(3))
        self.dV = self.h[0] * self.h[1] * self.h[2]
        self.nd = n[0] * n[1] * n[2]
        first = 0 if self.periodic else 1
        axis = [(torch.arange(n[i], dtype=F64, device=DEV) + first) * self.h[i] for i in range(3)]
        # Gaussian wells are products over the axes; periodic axes sum the nearest images
        v = torch.zeros(n[2], n[1], n[0], dtype=F64, device=DEV)
        for p, d, s in zip(pos, depth, sigma):
            g = []
            for i in range(3):
                im = (-1, 0, 1) if self.periodic else (0,)
                g.append(sum(torch.exp(-(axis[i] - (p[i] + k * L[i])) ** 2 / (2 * s * s))
                             for k in im))
            v -= d * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
        self.v = v
        # s and p projectors per atom of the Si-like cells and the cluster
        self.groups = []
        if kind in ("si", "cluster"):
            sp = 1.1
            for p in pos:
                d = []
                for i in range(3):
                    x = axis[i] - p[i]
                    d.append(x - L[i] * torch.round(x / L[i]) if self.periodic else x)
                r2 = (d[2] ** 2)[:, None, None] + (d[1] ** 2)[None, :, None] + (d[0] ** 2)[None, None]
                idx = torch.nonzero(r2.reshape(-1) <= (3.5 * sp) ** 2).reshape(-1)
                ix, iy, iz = idx % n[0], (idx // n[0]) % n[1], idx // (n[0] * n[1])
                e = torch.exp(-r2.reshape(-1)[idx] / (2 * sp * sp))
                chi = torch.stack([e, d[0][ix] * e, d[1][iy] * e, d[2][iz] * e])
                chi /= torch.sqrt(self.dV * (chi * chi).sum(1, keepdim=True))
                gam = np.concatenate([rng.uniform(1.5, 2.5, 1), rng.uniform(-3.5, -2.5, 3)])
                self.groups.append((idx, chi, gam))
        self.lap = [torch.from_numpy(_lap1d(n[i], self.h[i], self.periodic, self.radius)).to(DEV)
                    for i in range(3)]
        self._op = {}

    def _data(self, dtype):
        """V_loc, kinetic matrices and projectors in one type: by group (padded) for the dot
        products, by point (padded) for the sum, so that nothing is added in a random order."""
        if dtype in self._op:
            return self._op[dtype]
        op = dict(v=self.v.to(dtype), k=[(-0.5 * m).to(dtype) for m in self.lap])
        if self.groups:
            G = len(self.groups)
            top = max(len(g[0]) for g in self.groups)
            idx = torch.zeros(G, top, dtype=torch.int64, device=DEV)
            chi = torch.zeros(G, 4, top, dtype=F64, device=DEV)
            for k, (i, x, _) in enumerate(self.groups):
                idx[k, : len(i)] = i
                chi[k, :, : len(i)] = x
            gam = torch.from_numpy(np.stack([g[2] for g in self.groups])).to(DEV) * self.dV
            pts = torch.cat([g[0] for g in self.groups])
            grp = torch.cat([torch.full((len(g[0]),), k, device=DEV)
                             for k, g in enumerate(self.groups)])
            val = torch.cat([g[1].T for g in self.groups])
            order = torch.sort(pts, stable=True).indices
            pts, grp, val = pts[order], grp[order], val[order]
            rank = torch.arange(len(pts), device=DEV) - torch.searchsorted(pts, pts)
            layers = []
            for k in range(int(rank.max()) + 1):
                m = rank == k
                layers.append((pts[m], grp[m], val[m].to(dtype)))
            op.update(idx=idx, chi=chi.to(dtype), gam=gam.to(dtype), layers=layers)
        self._op[dtype] = op
        return op

    def apply(self, X):
        """H X for real rows X (m, N_d)."""
        op = self._data(X.dtype)
        nx, ny, nz = self.n
        m = X.shape[0]
        V = X.view(m, nz, ny, nx)
        Y = V * op["v"]
        Y += V @ op["k"][0]
        Y += op["k"][1] @ V
        Y = Y.view(m, -1)
        Y += (op["k"][2] @ X.view(m, nz, ny * nx)).view(m, -1)
        if self.groups:
            G, top = op["idx"].shape
            part = X[:, op["idx"].reshape(-1)].view(m, G, top).transpose(0, 1)
            c = (part @ op["chi"].transpose(1, 2)).transpose(0, 1) * op["gam"]   # (m, G, 4)
            for pts, grp, val in op["layers"]:
                Y[:, pts] += (c[:, grp] * val).sum(-1)
        return Y

    def ground_state(self, ns, rng):
        """Lowest ns eigenpairs: Chebyshev-filtered subspace iteration, FP32 then FP64."""
        m = ns + max(8, ns // 3)
        X = torch.from_numpy(rng.standard_normal((m, self.nd))).to(DEV)
        top = -0.5 * sum(float(torch.linalg.eigvalsh(k)[0]) for k in self.lap)
        top += max(0.0, float(self.v.max())) + (6.0 if self.groups else 0.0)
        X = _orth(X)
        HX = self.apply(X)
        th, W = torch.linalg.eigh(_sym(X @ HX.T))
        X, HX = W.T @ X, W.T @ HX
        for it in range(60):
            res = float((HX - th[:, None] * X)[:ns].norm(dim=1).max())
            if res < 1e-8:
                break
            low = torch.float64 if res < 5e-4 else torch.float32
            a, a0 = float(th[-1]), float(th[0])
            c, e = 0.5 * (top + a), 0.5 * (top - a)
            t0 = (a0 - c) / e
            rp, r = 1.0, t0
            Yp = X.to(low)
            Y = (self.apply(Yp) - c * Yp) / (e * r)
            for _ in range(2, 25 if low == torch.float32 else 31):
                rn = 2.0 * t0 * r - rp
                Yn = self.apply(Y)
                Yn.add_(Y, alpha=-c).mul_(2.0 * r / (e * rn)).add_(Yp, alpha=-rp / rn)
                Yp, Y = Y, Yn
                rp, r = r, rn
            X = _orth(Y.to(F64))
            HX = self.apply(X)
            th, W = torch.linalg.eigh(_sym(X @ HX.T))
            X, HX = W.T @ X, W.T @ HX
        return X[:ns] / math.sqrt(self.dV), th[:ns].clone()


def _sym(S):
    return 0.5 * (S + S.T)


def _orth(Y):
    for _ in range(2):
        L = torch.linalg.cholesky(_sym(Y @ Y.T))
        Y = torch.linalg.solve_triangular(L, Y, upper=False)
    return Y


def _problem(case, seed):
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["nz"], case["states"]])
    cell = _Cell(case, rng)
    psi, eps = cell.ground_state(case["states"], rng)
    return cell, psi, eps, rng


def _frequencies(nw):
    """Gauss-Legendre nodes mapped to [0, inf) by w = (1 + x) / (1 - x)."""
    x, w = np.polynomial.legendre.leggauss(nw)
    return (1 + x) / (1 - x), 2 * w / (1 - x) ** 2


def _nodes(n, g, periodic=True):
    k = list(range(0, n, g))
    return k if periodic or k[-1] == n - 1 else k + [n - 1]


def _points(case, cell, rng):
    """Probe-points sampled evenly over the frequencies, as the benchmark does."""
    cnt = case["count"]
    freqs = np.arange(cnt) * case["nw"] // cnt if cnt > 1 else np.array([case["nw"] // 2])
    return (rng.choice(cell.nd, cnt, replace=False).astype(np.int64), freqs.astype(np.int32))


# -------------------------------------------------------------------------------------------
# prepare / run
# -------------------------------------------------------------------------------------------
def prepare(case, seed):
    if case["kind"] == "interp":
        n = (case["nx"], case["ny"], case["nz"])
        om, w = _frequencies(case["nw"])
        ctx = R.Context(n, (0.39,) * 3, (0, 0, 0))
        R.rpa_set_frequencies(ctx.ctx, om, w)
        R.rpa_set_options(ctx.ctx, stride=(case["stride"],) * 3, interp="cubic")
        return dict(case=case, ctx=ctx, coarse=_coarse(case, seed))
    cell, psi, eps, rng = _problem(case, seed)
    bc = (0, 0, 0) if cell.periodic else (1, 1, 1)
    ctx = R.Context(cell.n, cell.h, bc, cell.radius)
    R.rpa_set_potential(ctx.ctx, cell.v.reshape(-1))
    R.rpa_set_projectors(ctx.ctx, [(i.cpu().numpy(), x.cpu().numpy(), g)
                                   for i, x, g in cell.groups])
    R.rpa_set_occupied(ctx.ctx, psi, eps)
    R.rpa_set_frequencies(ctx.ctx, *_frequencies(case["nw"]))
    opts = dict(precision=case["precision"], lanczos_max=case["nl"], stern_tol=case["tol"])
    state = dict(case=case, ctx=ctx)
    if case["kind"] == "energy":
        R.rpa_set_options(ctx.ctx, stride=(case["stride"],) * 3, interp="cubic", **opts)
        state["P"] = R.rpa_num_probes(ctx.ctx)
    else:
        R.rpa_set_options(ctx.ctx, **opts)
        state["points"] = _points(case, cell, rng)
    if case["kind"] == "chi0":
        # the vectors of a first Lanczos step, u = nu^(1/2) e_j
        points, freqs = state["points"]
        e = np.zeros((len(points), cell.nd))
        e[np.arange(len(points)), points] = 1.0
        state["u"] = R.rpa_apply_nu_half(ctx.ctx, e)
        state["omega"] = _frequencies(case["nw"])[0][freqs]
    return state


def run(state):
    case, ctx = state["case"], state["ctx"].ctx
    if case["kind"] == "interp":
        fine, ec = R.rpa_interpolate(ctx, state["coarse"], state["ctx"].nd)
        return dict(fine=fine, ec=ec)
    if case["kind"] == "energy":
        coarse, fine, ec, _ = R.rpa_energy_density(ctx, case["nw"], state["P"], state["ctx"].nd)
        return dict(coarse=coarse, fine=fine, ec=ec)
    if case["kind"] == "chi0":
        r, _ = R.rpa_chi0(ctx, state["omega"], state["u"], case["states"])
        return r
    out = R.rpa_probe_density(ctx, *state["points"], nl=case["nl"], want_tridiag=True,
                              allow_nonconv=True)
    return dict(d=out["d"], alpha=out["alpha"], beta=out["beta"], steps=out["steps"])


def work(case):
    nd = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "interp":
        m = [len(_nodes(case[a], case["stride"])) for a in ("nx", "ny", "nz")]
        nw = case["nw"]
        flops = 8 * nw * (case["nx"] * m[1] * m[2] + case["nx"] * case["ny"] * m[2] + nd)
        return dict(bytes=8 * nw * (m[0] * m[1] * m[2] + nd), flops=flops)
    if case["kind"] == "energy":
        cnt = case["nw"] * math.prod(len(_nodes(case[a], case["stride"]))
                                     for a in ("nx", "ny", "nz"))
    else:
        cnt = case["count"]
    # per Sternheimer system and COCG iteration: the vectors x, r, p and w = (H - sigma) p read
    # and written once each but for w (7 passes), 6 R + 1 complex by real multiply-adds for
    # the stencil and 5 complex multiply-adds; the iterations to the tolerance are taken as
    # 4 per decimal digit, what an average frequency needs at the least
    its = max(2.0, -4.0 * math.log10(case["tol"]))
    systems = cnt * case["states"] * case["nl"]
    size = 16 if case["precision"] == "fp64" else 8
    gram = 4.0 * case["states"] * nd            # Galerkin projection, per system
    return dict(bytes=systems * its * 7.0 * size * nd,
                flops=systems * (its * nd * (4.0 * (6 * case["radius"] + 1) + 40.0) + 1.5 * gram))


# -------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits, solved to convergence
# -------------------------------------------------------------------------------------------
def _coarse(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    P = math.prod(len(_nodes(case[a], case["stride"])) for a in ("nx", "ny", "nz"))
    # densities d_j(i w) are negative and vary over the cell
    return -torch.rand(case["nw"], P, generator=g, dtype=F64, device=DEV) * 1e-2 - 1e-4


def _interp_matrix(n, g, periodic):
    """Four-point Lagrange interpolation from the coarse nodes of one axis."""
    nodes = _nodes(n, g, periodic)
    m = len(nodes)
    W = np.zeros((n, m))
    for i in range(n):
        c = int(np.searchsorted(nodes, i, side="right")) - 1
        if periodic:
            ids = [c - 1 + t for t in range(4)]
            xs = [nodes[k % m] + n * (k // m) for k in ids]
            cols = [k % m for k in ids]
        else:
            k = min(4, m)
            f = min(max(min(c, m - 2) - (k // 2 - 1), 0), m - k)
            cols = list(range(f, f + k))
            xs = [nodes[q] for q in cols]
        for a, col in enumerate(cols):
            W[i, col] += math.prod((i - xs[b]) / (xs[a] - xs[b])
                                   for b in range(len(xs)) if b != a)
    return torch.from_numpy(W).to(DEV)


def _interpolate(case, coarse, periodic=True):
    n = [case["nx"], case["ny"], case["nz"]]
    W = [_interp_matrix(k, case["stride"], periodic) for k in n]
    D = coarse.view(case["nw"], W[2].shape[1], W[1].shape[1], W[0].shape[1])
    F = torch.einsum("ia,jb,kc,wcba->wkji", W[0], W[1], W[2], D).reshape(case["nw"], -1)
    weight = torch.from_numpy(_frequencies(case["nw"])[1]).to(DEV)
    return F, float((weight * F.sum(1)).sum()) / (2 * math.pi)


class _Exact:
    """chi0 and nu^(1/2) in 64 bits."""

    def __init__(self, cell, psi, eps, tol):
        self.cell, self.psi, self.eps = cell, psi, eps
        self.tol = max(1e-12, 0.01 * tol)
        self.mode = [torch.linalg.eigh(-m) for m in cell.lap]
        lam = (self.mode[2][0][:, None, None] + self.mode[1][0][None, :, None]
               + self.mode[0][0][None, None, :])
        keep = lam > 1e-10 * lam.max() if cell.periodic else lam > 0
        self.root = torch.where(keep, torch.sqrt(4 * math.pi / torch.where(keep, lam, 1.0)), 0.0)

    def nu_half(self, q):
        U = [m[1] for m in self.mode]
        t = q.view(-1, *self.root.shape)
        t = torch.einsum("bkji,ia,jd,kc->bcda", t, U[0], U[1], U[2])
        t = torch.einsum("bcda,ia,jd,kc->bkji", t * self.root, U[0], U[1], U[2])
        return t.reshape(q.shape)

    def _h(self, x, shift):
        y = self.cell.apply(torch.view_as_real(x).permute(2, 0, 1).reshape(-1, x.shape[1]))
        return torch.complex(y[: x.shape[0]], y[x.shape[0]:]) - shift[:, None] * x

    def chi0(self, u, omega):
        """u (b, N_d), omega (b,): 4 sum_n psi_n Re dpsi_n."""
        cell, psi, eps = self.cell, self.psi, self.eps
        ns, nd = psi.shape
        omega = torch.as_tensor(omega, dtype=F64, device=DEV)
        out = []
        few = max(1, int(2.5e7 / (ns * nd)))        # probe-points solved together
        for ub, ob in zip(u.split(few), omega.split(few)):
            b = -(psi[None] * ub[:, None])
            den = eps[None, :, None] - eps[None, None, :] - 1j * ob[:, None, None]
            C = cell.dV * (psi @ b.transpose(1, 2)) / den
            x = (C.transpose(1, 2) @ psi.to(C.dtype)).reshape(-1, nd)
            shift = (eps[None] + 1j * ob[:, None]).reshape(-1)
            b = b.reshape(-1, nd)
            r = b - self._h(x, shift)
            target = self.tol * b.norm(dim=1)
            live = torch.arange(len(b), device=DEV)
            xs, p = x.clone(), r.clone()
            rho = (r * r).sum(1)
            for it in range(4000):
                w = self._h(p, shift[live])
                a = (rho / (p * w).sum(1))[:, None]
                x += a * p
                r -= a * w
                new = (r * r).sum(1)
                p = r + (new / rho)[:, None] * p
                rho = new
                if it % 16 == 15:
                    go = r.norm(dim=1) > target[live]
                    xs[live[~go]] = x[~go]
                    if not bool(go.any()):
                        break
                    live, x, r, p, rho = live[go], x[go], r[go], p[go], rho[go]
            out.append(4 * (psi[None] * xs.real.view(-1, ns, nd)).sum(1))
        return torch.cat(out)

    def lanczos(self, points, omega, nl):
        nb = len(points)
        Q = [torch.zeros(nb, self.cell.nd, dtype=F64, device=DEV)]
        Q[0][torch.arange(nb), torch.from_numpy(points).to(DEV)] = 1.0
        al, be = [], []
        for _ in range(nl):
            v = self.nu_half(self.chi0(self.nu_half(Q[-1]), omega))
            al.append((Q[-1] * v).sum(1))
            for _ in range(2):
                for q in Q:
                    v = v - (q * v).sum(1, keepdim=True) * q
            be.append(v.norm(dim=1))
            Q.append(v / be[-1][:, None])
        al, be = torch.stack(al, 1), torch.stack(be, 1)
        T = torch.diag_embed(al)
        if nl > 1:
            T = T + torch.diag_embed(be[:, :-1], 1) + torch.diag_embed(be[:, :-1], -1)
        lam, W = torch.linalg.eigh(T)
        d = (W[:, 0, :] ** 2 * (torch.log1p(-lam) + lam)).sum(1)
        be[:, -1] = 0.0      # the last step makes no further vector
        return d, al, be


def exact(case, seed):
    if case["kind"] == "interp":
        fine, ec = _interpolate(case, _coarse(case, seed))
        return dict(fine=fine, ec=ec)
    cell, psi, eps, rng = _problem(case, seed)
    om = _frequencies(case["nw"])[0]
    ex = _Exact(cell, psi, eps, case["tol"])
    if case["kind"] == "energy":
        axis = [_nodes(k, case["stride"], cell.periodic) for k in cell.n]
        pts = np.array([x + cell.n[0] * (y + cell.n[1] * z) for z in axis[2] for y in axis[1]
                        for x in axis[0]])
        coarse = torch.stack([ex.lanczos(pts, np.full(len(pts), o), case["nl"])[0] for o in om])
        fine, ec = _interpolate(case, coarse, cell.periodic)
        return dict(coarse=coarse, fine=fine, ec=ec)
    points, freqs = _points(case, cell, rng)
    if case["kind"] == "chi0":
        e = torch.zeros(len(points), cell.nd, dtype=F64, device=DEV)
        e[torch.arange(len(points)), torch.from_numpy(points).to(DEV)] = 1.0
        return ex.chi0(ex.nu_half(e), om[freqs])
    d, al, be = ex.lanczos(points, om[freqs], case["nl"])
    return dict(d=d, alpha=al, beta=be, steps=None)
