"""The choice of the resident COCG kernel's cluster size is the same in every call."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R
from tests.test_gpu_resident import plane_waves

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-6)])
@pytest.mark.parametrize("groups", [8, 34, 90])
def test_calls_do_not_depend_on_earlier_ones(groups, prec, tol):
    """12^3 points in 16 bricks leave 117 values per brick for the projector sums, four per
    group that touches the brick: with 34 groups that touch every brick clusters of 16 are
    ruled out, with 90 clusters of 4 to 16.  The first call and the second take the same size: the
    sums, and so the results, are equal to the bit."""
    n, ns, nd, h = (12, 12, 12), 4, 1728, (0.45, 0.5, 0.4)
    rng = np.random.default_rng(8)
    psi, eps = plane_waves(n, h, (0, 0, 0), ns)
    c = R.Context(n, h, (0, 0, 0), 6)
    R.rpa_set_potential(c.ctx, -rng.uniform(0.0, 1.5, nd))
    R.rpa_set_projectors(c.ctx, [
        (np.sort(rng.choice(nd, size=300, replace=False)).astype(np.int32),
         0.2 * rng.standard_normal((4, 300)), rng.uniform(-0.1, 0.1, 4)) for _ in range(groups)])
    R.rpa_set_occupied(c.ctx, psi, eps)
    R.rpa_set_options(c.ctx, precision=prec, stern_tol=tol)
    u = rng.standard_normal((1, nd))
    first, second = (R.rpa_chi0(c.ctx, np.array([0.7]), u, ns) for _ in range(2))
    c.close()
    assert np.array_equal(first[1], second[1]) and np.array_equal(first[0], second[0])


def test_size_counts_systems_that_refinement_takes_up():
    """A guess that meets the inner tolerance is not done: the rounds that follow run the whole wave, on the
    cluster size of a whole wave (320 systems on 26^3: clusters of two, no launched iterations)."""
    n, ns, cnt, h = (26, 26, 26), 16, 20, (0.45, 0.5, 0.4)
    nd = int(np.prod(n))
    rng = np.random.default_rng(8)
    psi, eps = plane_waves(n, h, (0, 0, 0), ns)
    c = R.Context(n, h, (0, 0, 0), 6)
    R.rpa_set_potential(c.ctx, -rng.uniform(0.0, 1.5, nd))
    R.rpa_set_projectors(c.ctx, [])
    R.rpa_set_occupied(c.ctx, psi, eps)
    R.rpa_set_frequencies(c.ctx, np.array([0.5, 2.0]), np.array([1.0, 1.0]))
    R.rpa_set_options(c.ctx, precision="mixed", stern_tol=1e-6, inner_tol=2.0, refine=2, lanczos_max=1,
                      profile=1)
    out = R.rpa_probe_density(c.ctx, rng.choice(nd, cnt, replace=False).astype(np.int64),
                              (np.arange(cnt) % 2).astype(np.int32), allow_nonconv=True)
    c.close()
    assert out["stats"]["refine_rounds"] > 0
    assert out["stats"]["tile_rows"] == out["stats"]["tile_rows_tail"] == -7
