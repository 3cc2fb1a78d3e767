"""The resident COCG kernel on very small and very large vectors: the FP64 form solves whatever
the launched iteration solves, down to |p^T A p|^2 among the subnormal numbers, where a
reciprocal of it overflows."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R
from tests.test_gpu_resident import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** -236, 2.0 ** 240], ids=["tiny", "huge"])
@pytest.mark.parametrize("graphs", [2, 1], ids=["resident", "launched"])
def test_fp64_range(scale, graphs):
    """chi0 (s u) = s chi0 u: each solve meets ||b - A x|| <= tol ||b||, so the two differ by at
    most the bound of test_gpu_resident.py."""
    n, ns, tol, om = (12, 12, 12), 4, 1e-8, np.array([0.3, 1.0])
    u = np.random.default_rng(5).standard_normal((2, 12 ** 3))
    c, psi = context(n, (0, 0, 0), 6, ns, 3, 11, precision="fp64", stern_tol=tol, graphs=graphs)
    ref = R.rpa_chi0(c.ctx, om, u, ns)[0]
    got = R.rpa_chi0(c.ctx, om, scale * u, ns)[0] / scale
    c.close()
    top = np.abs(psi).max(axis=1)
    for i in range(2):
        bn = np.linalg.norm(psi * u[i], axis=1)
        assert np.linalg.norm(got[i] - ref[i]) <= 8.0 * float(top @ bn) * tol / om[i]
