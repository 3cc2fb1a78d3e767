"""What the interpolation keeps between calls is bounded (64 MiB): larger workspaces are given back."""
import numpy as np
import pytest

import paper_2609_16408_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dev", [False, True], ids=["host", "device"])
def test_large_workspace_is_given_back(dev):
    import torch
    n, nw = (64, 64, 64), 64   # 134 MB for each array
    nd = int(np.prod(n))
    c = R.Context(n, (0.4,) * 3, (0, 0, 0), 2)
    R.rpa_set_frequencies(c.ctx, *R.rpa_gl_frequencies(nw))
    R.rpa_set_options(c.ctx, stride=(4, 4, 4), interp="cubic")
    small = -np.ones((nw, R.rpa_num_probes(c.ctx)))
    R.rpa_interpolate(c.ctx, small, nd)  # operators, and the driver's own allocations
    R.rpa_set_options(c.ctx, stride=(1, 1, 1), interp="cubic")
    d = -np.ones((nw, nd))
    if dev:
        d = torch.from_numpy(d).cuda()
        warm = torch.empty_like(d)  # the result's place in torch's pool
        del warm
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    fine, _ = R.rpa_interpolate(c.ctx, d, nd)
    torch.cuda.synchronize()
    after = torch.cuda.mem_get_info()[0]
    c.close()
    assert float(fine[0, 0]) == -1.0
    assert before - after <= 64 << 20
