"""FP64 Galerkin guesses at state counts around the tile sizes (8 and 16 states) against the
formula in numpy.  Error bound, element by element: the sum over N_d points of products rounds
by at most (N_d + 4) 2^-53 of its terms' moduli, the sum over states by (N_s + 4) 2^-53."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [1, 7, 8, 9, 15, 16, 17, 33])
@pytest.mark.parametrize("n", [(5, 6, 7), (12, 12, 12), (16, 17, 18)], ids=lambda n: "x".join(map(str, n)))
def test_galerkin_fp64(n, ns):
    rng = np.random.default_rng(ns)
    nd, h = int(np.prod(n)), (0.4, 0.5, 0.6)
    dV = float(np.prod(h))
    psi = np.linalg.qr(rng.standard_normal((nd, ns)))[0].T / np.sqrt(dV)
    psi = np.ascontiguousarray(psi)
    eps = np.linspace(-0.5, 0.1, ns)
    c = R.Context(n, h, (0, 0, 0), 4)
    R.rpa_set_potential(c.ctx, np.zeros(nd))
    R.rpa_set_projectors(c.ctx, [])
    R.rpa_set_occupied(c.ctx, psi, eps)
    R.rpa_set_options(c.ctx, precision="fp64", lanczos_max=1)
    om, u = np.array([0.3, 2.0, 0.7]), rng.standard_normal((3, nd))
    x0 = R.rpa_galerkin(c.ctx, om, u, ns)
    # the same guesses start a solve, whose chunks are cut differently
    r, _ = R.rpa_chi0(c.ctx, om, u, ns)
    assert np.isfinite(r).all()
    c.close()
    for i in range(3):
        G = -dV * (psi * u[i]) @ psi.T
        A = dV * np.abs(psi * u[i]) @ np.abs(psi).T
        den = eps[:, None] - eps[None, :] - 1j * om[i]
        ref = (G / den).T @ psi
        bound = (nd + ns + 8) * 2.0 ** -53 * 2 * (A / np.abs(den)).T @ np.abs(psi)
        assert (np.abs(x0[i] - ref) <= 2 * bound).all()
