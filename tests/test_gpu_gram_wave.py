"""The FP64 Galerkin guess of a probe-point does not depend on what else is in its wave, and
rpa_galerkin returns the guess that starts a solve: equal to the bit."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R
from tests.test_gpu_resident import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ns", [((12, 12, 12), 8), ((9, 10, 11), 3), ((20, 18, 22), 17),
                                  ((26, 26, 26), 40)], ids=["12^3-8", "9x10x11-3", "20x18x22-17", "26^3-40"])
def test_guess_is_the_same_alone_and_in_a_wave(n, ns):
    cnt = 37
    c, psi = context(n, (0, 0, 0), 4, ns, 0, 11, precision="fp64", stern_tol=1e30)  # the guess is accepted
    u = np.random.default_rng(3).standard_normal((cnt, int(np.prod(n))))
    om = np.linspace(0.3, 2.0, cnt)
    wave = R.rpa_chi0(c.ctx, om, u, ns)[0]
    x0 = R.rpa_galerkin(c.ctx, om, u, ns)
    for i in (0, 5, cnt - 1):
        one, it = R.rpa_chi0(c.ctx, om[i:i + 1], u[i:i + 1], ns)
        assert it.max() == 0
        assert np.array_equal(one[0], wave[i])
        assert np.array_equal(R.rpa_galerkin(c.ctx, om[i:i + 1], u[i:i + 1], ns)[0], x0[i])
        # the density 4 sum_n psi_n Re x_n as the kernel adds it: fused multiply-adds in state order
        acc = np.zeros(u.shape[1], dtype=np.longdouble)
        for k in range(ns):
            acc = (acc + psi[k].astype(np.longdouble) * x0[i, k].real).astype(np.float64)
        rel = np.abs(4.0 * acc.astype(np.float64) - one[0])
        assert (rel <= (ns + 2) * 2.0 ** -53 * 4.0 * (np.abs(psi) * np.abs(x0[i].real)).sum(axis=0)).all()
    c.close()
