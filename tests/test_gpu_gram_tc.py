"""Mixed-form Galerkin guesses (three TF32 MMAs, FP32 accumulation) at state counts around the
groups of 8, the K stages of 32 and the tiles of 128, on grids with and without 16-byte rows.
Error bound, element by element: each product is off by at most 2^-21 of its modulus (FP32
operands and the dropped low x low part), each of the N_d + N_s additions by 2^-22 of the sum of
moduli (truncation to 23 bits)."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns", [1, 7, 8, 9, 31, 33, 64, 127, 129])
@pytest.mark.parametrize("n", [(5, 6, 7), (15, 17, 19), (16, 17, 18)], ids=lambda n: "x".join(map(str, n)))
def test_galerkin_mixed(n, ns):
    rng = np.random.default_rng(ns)
    nd, h = int(np.prod(n)), (0.4, 0.5, 0.6)
    dV = float(np.prod(h))
    psi = np.ascontiguousarray(np.linalg.qr(rng.standard_normal((nd, ns)))[0].T / np.sqrt(dV))
    eps = np.linspace(-0.5, 0.1, ns)
    c = R.Context(n, h, (0, 0, 0), 4)
    R.rpa_set_potential(c.ctx, np.zeros(nd))
    R.rpa_set_projectors(c.ctx, [])
    R.rpa_set_occupied(c.ctx, psi, eps)
    R.rpa_set_options(c.ctx, precision="mixed", lanczos_max=1)
    om, u = np.array([0.3, 2.0, 0.7]), rng.standard_normal((3, nd))
    x0 = R.rpa_galerkin(c.ctx, om, u, ns)
    # the same guesses start a solve
    r, _ = R.rpa_chi0(c.ctx, om, u, ns)
    assert np.isfinite(r).all()
    c.close()
    for i in range(3):
        G = -dV * (psi * u[i]) @ psi.T
        A = dV * np.abs(psi * u[i]) @ np.abs(psi).T
        den = eps[:, None] - eps[None, :] - 1j * om[i]
        ref = (G / den).T @ psi
        bound = (nd + ns + 8) * 2.0 ** -22 * (A / np.abs(den)).T @ np.abs(psi)
        assert (np.abs(x0[i] - ref) <= 2 * bound).all()
