"""Interpolation by at most four taps per axis against the oracle's dense operators: ragged
grids around the 1,024-output blocks, host and device arrays, in place at stride 1.

Tolerance: a fine value is a sum of at most 64 products of three weights (each of modulus at
most 1.2) and a coarse value, so its rounding error is below 64 * 1.2^3 * 4 * 2^-53 of the
largest coarse value; E_c adds N_d n_w values in FP64 trees (depth below 40).
"""
import numpy as np
import pytest

import oracle
import paper_2609_16408_gb300 as R

pytestmark = pytest.mark.gpu

CASES = [
    # n, bc, stride, kind, frequencies
    ((16, 16, 4), (0, 0, 0), (1, 1, 1), "cubic", 1),      # exactly one block of outputs
    ((16, 16, 5), (0, 0, 0), (2, 3, 1), "cubic", 3),
    ((9, 13, 11), (0, 1, 1), (2, 2, 3), "cubic", 4),
    ((9, 13, 11), (1, 0, 0), (4, 3, 2), "linear", 2),
    ((3, 2, 7), (1, 1, 1), (2, 1, 3), "cubic", 2),        # fewer coarse nodes than taps
    ((1, 1, 33), (1, 1, 0), (1, 1, 4), "cubic", 1),       # one coarse node on two axes
    ((52, 50, 47), (0, 0, 0), (2, 2, 3), "cubic", 10),
    ((7, 8, 9), (0, 0, 0), (1, 1, 1), "none", 2),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}-{c[2]}-{c[3]}")
@pytest.mark.parametrize("dev", [False, True], ids=["host", "device"])
def test_taps_match_dense_operators(case, dev):
    n, bc, g, kind, nw = case
    nd = int(np.prod(n))
    om, w = oracle.gl_frequencies(max(nw, 1))
    c = R.Context(n, (0.4,) * 3, bc, 2)
    R.rpa_set_frequencies(c.ctx, om, w)
    R.rpa_set_options(c.ctx, stride=g, interp=kind)
    P = R.rpa_num_probes(c.ctx)
    d = -np.random.default_rng(1).uniform(0.0, 1.0, (nw, P))
    ref = np.stack([oracle.interpolate(x, n, g, bc, kind) for x in d])
    if dev:
        import torch
        fine, ec = R.rpa_interpolate(c.ctx, torch.from_numpy(d).cuda(), nd)
        fine = fine.cpu().numpy()
    else:
        fine, ec = R.rpa_interpolate(c.ctx, d, nd)
    tol = 64 * 1.2 ** 3 * 4 * 2.0 ** -53 * np.abs(d).max()
    assert np.abs(fine - ref).max() <= tol
    want = float(w @ ref.sum(axis=1)) / (2 * np.pi)
    assert abs(ec - want) <= float(w @ np.abs(ref).sum(axis=1)) / (2 * np.pi) * 64 * 2.0 ** -53 + tol * nd * w.sum()
    c.close()


def test_in_place_at_stride_one():
    import ctypes as C

    import torch
    n = (8, 9, 10)
    c = R.Context(n, (0.4,) * 3, (0, 0, 0), 2)
    R.rpa_set_frequencies(c.ctx, *oracle.gl_frequencies(2))
    R.rpa_set_options(c.ctx, stride=(1, 1, 1), interp="cubic")
    a = torch.rand(2, 720, dtype=torch.float64, device="cuda")
    b = a.clone()
    ptr = C.c_void_p(a.data_ptr())
    assert R.load().rpa_interpolate(c.ctx, ptr, ptr, None, R.RPA_DEVICE) == R.RPA_OK
    assert torch.equal(a, b)
    c.close()
