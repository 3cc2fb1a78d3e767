"""Statistics of the resident COCG kernel: a slot of its own, the bytes that it moves, the launches
counted, and the tiling of launches that did not happen not named."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R
from tests.test_gpu_resident import context

pytestmark = pytest.mark.gpu

CASES = [
    # n, precision, probe-points, resident alone
    ((12, 12, 12), "fp64", 1, True),     # clusters of 16
    ((12, 12, 12), "mixed", 200, True),  # one block per system
    ((26, 26, 26), "mixed", 40, True),   # x in global memory
    ((26, 26, 26), "fp64", 2, True),
    ((44, 46, 42), "mixed", 40, False),  # launched iterations first
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0][0]}-{c[1]}-{c[2]}")
def test_resident_slot(case):
    n, prec, cnt, alone = case
    nd, ns = int(np.prod(n)), 8
    c, _ = context(n, (0, 0, 0), 6, ns, 3, 11, precision=prec, stern_tol=1e-6, lanczos_max=2,
                   profile=1)
    R.rpa_set_frequencies(c.ctx, np.array([0.5, 2.0]), np.array([1.0, 1.0]))
    pts = np.random.default_rng(1).choice(nd, cnt, replace=False).astype(np.int64)
    l0 = R.rpa_kernel_launches()
    st = R.rpa_probe_density(c.ctx, pts, (np.arange(cnt) % 2).astype(np.int32))["stats"]
    assert R.rpa_kernel_launches() - l0 >= st["kernel_launches"][7]
    c.close()
    ks, kl, kb = st["kernel_seconds"], st["kernel_launches"], st["kernel_bytes"]
    size = 16 if prec == "fp64" else 8
    assert st["tile_rows_tail"] == -7 and (st["tile_rows"] == -7) == alone
    assert kl[7] > 0 and 0.0 < ks[7] <= 1.05 * st["seconds_phase"][2]
    # at most p, r and x in every iteration, and r, x (twice), p (twice) once per loop and solve
    assert 0.0 < kb[7] <= (5.0 * st["cocg_iters"] + 5.0 * (st["solves"] + st["refine_rounds"]) * 2) * size * nd
    assert (sum(kl[:5]) == 0) == alone and (sum(ks[:5]) == 0.0) == alone
    assert st["precision_bytes"] == size // 2
