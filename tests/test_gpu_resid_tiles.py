"""The tiles of the true residual: solves of the mixed form against the FP64 form on planes
whose extents make full-row, half-row and ragged tiles.  Both forms end with a true residual
(double-float at 1e-8, FP64 below it) at or under the tolerance, so they differ by at most
2 * 4 sum_n max|psi_n| tol ||b_n|| / omega (see test_gpu_resident.py); a wrong residual at any
point of the plane would leave an error of the order of b there."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R
from tests.test_gpu_resident import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [4, 6, 8])
@pytest.mark.parametrize("n", [(40, 9, 8), (52, 13, 8), (26, 26, 9), (27, 25, 8), (64, 9, 9),
                               (65, 8, 10), (8, 70, 9), (130, 9, 8), (12, 12, 66)],
                         ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 1, 0)], ids=["per", "walls"])
def test_residual_tiles(n, radius, bc):
    cnt, ns, tol = 2, 3, 1e-8
    u = np.random.default_rng(2).standard_normal((cnt, int(np.prod(n))))
    om = np.array([0.5, 1.0])
    out = []
    for prec in ("mixed", "fp64"):
        c, psi = context(n, bc, radius, ns, 3, 7, precision=prec, stern_tol=tol, refine=6)
        out.append(R.rpa_chi0(c.ctx, om, u, ns)[0])
        c.close()
    top = np.abs(psi).max(axis=1)
    for i in range(cnt):
        bn = np.linalg.norm(psi * u[i], axis=1)
        # FP32 inputs of the mixed form (u and psi enter its right-hand side as pairs, V and the
        # projectors too, so only the 2^-24 rounding of u on entry): relative 2^-24 of b
        bound = 8.0 * float(top @ bn) * (tol + 2.0 ** -24) / om[i]
        assert np.linalg.norm(out[0][i] - out[1][i]) <= bound
