"""rpa_interpolate on device arrays at addresses that the kernels cannot use in place: they go
through a copy and give the same values to the bit."""
import ctypes as C

import numpy as np
import pytest

import oracle
import paper_2609_16408_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["cubic", "fourier"])
@pytest.mark.parametrize("off", [(0, 0, 0), (4, 0, 0), (0, 4, 0), (0, 0, 4), (4, 2, 1)],
                         ids=lambda o: "-".join(map(str, o)))
def test_any_alignment(off, kind):
    import torch
    n, nw = (8, 10, 12), 3
    nd = int(np.prod(n))
    c = R.Context(n, (0.4,) * 3, (0, 0, 0), 2)
    R.rpa_set_frequencies(c.ctx, *oracle.gl_frequencies(nw))
    R.rpa_set_options(c.ctx, stride=(2, 2, 2), interp=kind)
    P = R.rpa_num_probes(c.ctx)
    d = -np.random.default_rng(1).uniform(0.0, 1.0, (nw, P))
    ref, ec = R.rpa_interpolate(c.ctx, d, nd)
    raw = [torch.zeros(8 * k + 16, dtype=torch.uint8, device="cuda") for k in (nw * P, nw * nd, 1)]
    raw[0][off[0]:off[0] + d.nbytes] = torch.from_numpy(np.frombuffer(d.tobytes(), np.uint8).copy()).cuda()
    torch.cuda.synchronize()
    p = [C.c_void_p(t.data_ptr() + o) for t, o in zip(raw, off)]
    assert R.load().rpa_interpolate(c.ctx, p[0], p[1], p[2], R.RPA_DEVICE) == R.RPA_OK
    out = [t.cpu().numpy()[o:o + 8 * k].tobytes() for t, o, k in zip(raw, off, (nw * P, nw * nd, 1))]
    assert out[0] == d.tobytes()
    assert out[1] == ref.tobytes()
    assert np.frombuffer(out[2]) == ec
    for t, o, k in zip(raw, off, (nw * P, nw * nd, 1)):  # nothing written beside the arrays
        t = t.cpu().numpy()
        assert not t[:o].any() and not t[o + 8 * k:].any()
    c.close()
