"""The resident COCG kernel (one cluster per system) against the launched iteration.

Both solve the same systems to the same tolerance.  H is real symmetric, so every
eigenvalue of H - eps_n - i omega is at least omega away from zero and a solve that meets
||b - A x|| <= tol ||b|| is within tol ||b|| / omega of the exact x; the density is
4 sum_n psi_n Re x_n, so two runs differ by at most
2 * 4 sum_n max|psi_n| tol ||b_n|| / omega in the 2-norm.  (FP64 rounding, 1e-14 of the
result, is far below that at the tolerances used.)
"""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R

pytestmark = pytest.mark.gpu


def plane_waves(n, h, bc, ns):
    """The ns smoothest products of cosines and sines, normalised on the grid."""
    axes = []
    for m, p in zip(n, bc):
        i = np.arange(m)
        if p == 0:
            f = [np.ones(m)] + [g(2 * np.pi * k * i / m) for k in (1, 2) for g in (np.cos, np.sin)]
            e = [0.0, 1.0, 1.0, 4.0, 4.0]
        else:
            f = [np.sin(np.pi * k * (i + 1) / (m + 1)) for k in range(1, 6)]
            e = [0.25 * k * k for k in range(1, 6)]
        axes.append(list(zip(e, f)))
    q = sorted(((a[0] + b[0] + c[0], i) for i, (a, b, c) in enumerate(
        (a, b, c) for c in axes[2] for b in axes[1] for a in axes[0])), key=lambda t: t)
    every = [(a, b, c) for c in axes[2] for b in axes[1] for a in axes[0]]
    psi = []
    for _, i in q[:ns]:
        a, b, c = every[i]
        v = (c[1][:, None, None] * b[1][None, :, None] * a[1][None, None, :]).ravel()
        psi.append(v / np.sqrt(np.prod(h) * (v @ v)))
    return np.array(psi), np.linspace(-0.4, -0.1, ns)


def context(n, bc, radius, ns, groups, seed, **opts):
    rng = np.random.default_rng(seed)
    h = (0.45, 0.5, 0.4)
    nd = int(np.prod(n))
    psi, eps = plane_waves(n, h, bc, ns)
    c = R.Context(n, h, bc, radius)
    R.rpa_set_potential(c.ctx, -rng.uniform(0.0, 1.5, nd))
    gr = []
    for g in range(groups):
        idx = np.sort(rng.choice(nd, size=min(nd, 40 + 23 * g), replace=False)).astype(np.int32)
        gr.append((idx, rng.standard_normal((1 + g % 6, len(idx))), rng.uniform(-0.4, 0.4, 1 + g % 6)))
    R.rpa_set_projectors(c.ctx, gr)
    R.rpa_set_occupied(c.ctx, psi, eps)
    R.rpa_set_options(c.ctx, **opts)
    return c, psi


CASES = [
    # n, bc, radius, states, vectors, projector groups
    ((12, 12, 12), (0, 0, 0), 6, 8, 1, 3),      # few systems: clusters of 16
    ((6, 6, 48), (0, 0, 0), 6, 2, 3, 1),        # two extents are the radius
    ((11, 12, 13), (0, 1, 0), 6, 4, 2, 3),
    ((13, 17, 9), (1, 1, 1), 4, 5, 3, 0),
    ((16, 9, 11), (0, 0, 1), 6, 6, 60, 4),      # many systems: one block each
    ((71, 8, 10), (0, 0, 0), 4, 3, 2, 2),       # rows longer than two warps
    ((25, 26, 27), (0, 0, 0), 6, 4, 12, 5),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])))
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("mixed", 1e-9)])
def test_resident_matches_launched(case, prec, tol):
    n, bc, radius, ns, cnt, groups = case
    check(n, bc, radius, ns, cnt, groups, prec, tol)


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-9), ("mixed", 1e-4), ("fp64", 1e-10)])
def test_handover_on_a_large_grid(prec, tol):
    """A grid that needs clusters of 8 or 16: launched iterations first, the resident kernel
    for the last systems (at 1e-4 with a recurrence continued across refinement rounds)."""
    check((40, 38, 41), (0, 0, 0), 6, 7, 40, 6, prec, tol)


def check(n, bc, radius, ns, cnt, groups, prec, tol):
    rng = np.random.default_rng(3)
    u = rng.standard_normal((cnt, int(np.prod(n))))
    om = np.linspace(0.3, 2.0, cnt)
    out = []
    for graphs in (2, 1):
        c, psi = context(n, bc, radius, ns, groups, 11, precision=prec, stern_tol=tol, refine=6,
                         graphs=graphs)
        r, it = R.rpa_chi0(c.ctx, om, u, ns)
        assert it.min() > 0
        out.append(r)
        c.close()
    top = np.abs(psi).max(axis=1)
    for i in range(cnt):
        bn = np.linalg.norm(psi * u[i], axis=1)
        bound = 8.0 * float(top @ bn) * tol / om[i]
        assert np.linalg.norm(out[0][i] - out[1][i]) <= bound


def test_resident_iteration_cap():
    c, _ = context((12, 12, 12), (0, 0, 0), 6, 4, 2, 11, precision="fp64", stern_tol=1e-12,
                   stern_maxit=3)
    with pytest.raises(R.RpaError) as e:
        R.rpa_chi0(c.ctx, np.array([0.3]), np.ones((1, 12 ** 3)) + np.arange(12 ** 3) % 5, 4)
    assert e.value.status == R.RPA_ENOCONV
    c.close()
