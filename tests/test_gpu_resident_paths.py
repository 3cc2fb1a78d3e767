"""The resident COCG kernel in the calls that reach it: that it runs, at every cluster size and with r and
x in shared or global memory, against the oracle, and its failure statuses, lanes and threads.

Which kernel ran is read from the statistics (tile_rows -7: no launched iterations), and from the
vector passes over global memory per iteration: one for p where a cluster has more than one block, two
each for r and x where they are not in shared memory.
"""
import threading

import numpy as np
import pytest

import oracle
import paper_2609_16408_gb300 as R
from synth import DIRICHLET, PERIODIC
from tests.systems_small import small
from tests.test_gpu_resident import CASES, context

pytestmark = pytest.mark.gpu


def density(c, nd, cnt, **kw):
    """Probe-points spread over two frequencies, with the statistics."""
    R.rpa_set_frequencies(c.ctx, np.array([0.5, 2.0]), np.array([1.0, 1.0]))
    pts = np.random.default_rng(1).choice(nd, cnt, replace=False).astype(np.int64)
    return R.rpa_probe_density(c.ctx, pts, (np.arange(cnt) % 2).astype(np.int32), **kw)


# Bytes of a vector in one block: 16 (FP64) or 8 times the row pitch (odd) times the brick's rows;
# p and w, then r, then x take what fits of 227 KB
SIZES = [
    # n, precision, probe-points of 8 states, passes per iteration
    ((12, 12, 12), "fp64", 64, 0),    # one block, 4 x 29 KB
    ((18, 18, 18), "fp64", 40, 4),    # one block, 2 x 98 KB
    ((20, 20, 20), "fp64", 40, 3),    # two, 3 x 67 KB
    ((23, 23, 23), "fp64", 40, 5),    # two, 2 x 101 KB
    ((26, 26, 26), "fp64", 20, 5),    # four, 2 x 73 KB and no room for a third
    ((26, 26, 26), "fp64", 2, 1),     # eight, 4 x 36 KB
    ((30, 30, 30), "fp64", 2, 3),     # eight, 3 x 59 KB
    ((12, 12, 12), "fp64", 1, 1),     # sixteen
    ((12, 12, 12), "mixed", 64, 0),
    ((20, 20, 20), "mixed", 40, 2),   # one block, 3 x 67 KB
    ((23, 23, 23), "mixed", 40, 4),   # one block, 2 x 97 KB
    ((26, 26, 26), "mixed", 40, 3),   # two, 3 x 73 KB
    ((30, 30, 30), "mixed", 40, 5),   # two, 2 x 112 KB
    ((31, 31, 31), "mixed", 20, 3),   # four, 3 x 63 KB
    ((33, 33, 33), "mixed", 20, 5),   # four, 2 x 76 KB
    ((26, 26, 26), "mixed", 1, 1),    # sixteen or eight
]


@pytest.mark.parametrize("case", SIZES, ids=lambda c: f"{c[0][0]}-{c[1]}-{c[2]}")
def test_sizes(case):
    n, prec, cnt, passes = case
    nd, ns = int(np.prod(n)), 8
    c, _ = context(n, (0, 0, 0), 6, ns, 3, 11, precision=prec, stern_tol=1e-8, lanczos_max=1,
                   profile=1)
    st = density(c, nd, cnt)["stats"]
    c.close()
    assert st["tile_rows"] == st["tile_rows_tail"] == -7
    q = st["kernel_bytes"][7] / ((16 if prec == "fp64" else 8) * nd * st["cocg_iters"])
    # at most five passes per loop, at most 1 + refinement rounds loops of 20 iterations or more
    assert passes < q < passes + 0.6, (passes, q)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])))
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("mixed", 1e-9)])
def test_resident_cases_take_the_kernel(case, prec, tol):
    n, bc, radius, ns, cnt, groups = case
    c, _ = context(n, bc, radius, ns, groups, 11, precision=prec, stern_tol=tol, refine=6,
                   lanczos_max=1, profile=1)
    st = density(c, int(np.prod(n)), cnt)["stats"]
    c.close()
    assert st["tile_rows"] == st["tile_rows_tail"] == -7 and st["kernel_launches"][7] > 0


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-9), ("mixed", 1e-4), ("fp64", 1e-10)])
def test_handover_case_takes_both(prec, tol):
    n = (40, 38, 41)
    c, _ = context(n, (0, 0, 0), 6, 7, 6, 11, precision=prec, stern_tol=tol, refine=6, lanczos_max=1,
                   profile=1)
    st = density(c, int(np.prod(n)), 40)["stats"]
    c.close()
    assert st["tile_rows"] != -7 and st["tile_rows_tail"] == -7 and st["kernel_launches"][7] > 0


SMALL = {
    "per": dict(n=(12, 12, 13), L=(6.0, 6.0, 6.5)),
    "walls": dict(n=(12, 13, 12), L=(6.0, 6.5, 6.0), bc=(DIRICHLET,) * 3),
    "mixed": dict(n=(16, 11, 12), L=(8.0, 5.5, 6.0), bc=(PERIODIC, DIRICHLET, PERIODIC)),
    "r4": dict(n=(13, 12, 12), L=(6.5, 6.0, 6.0), radius=4),
    "bare": dict(n=(12, 12, 13), L=(6.0, 6.0, 6.5), proj=False),
}
_S = {}


def system(name):
    if name not in _S:
        _S[name] = small(**SMALL[name])
    return _S[name]


def solver(s, **opts):
    om, w = oracle.gl_frequencies(4)
    return R.Context.from_system(s, om, w, **opts), om


@pytest.mark.parametrize("name", list(SMALL))
def test_against_the_oracle(name):
    """Tolerances as in the parity tests: solves at 1e-12 on both sides agree to 1e-9 (FP64); the
    mixed form at 1e-10 to 1e-7 of the largest value."""
    s = system(name)
    probes, freqs = np.array([5, 700, 1500], dtype=np.int64), np.array([0, 2, 3], dtype=np.int32)
    c, om = solver(s, precision="fp64", lanczos_max=3, stern_tol=1e-12, stern_maxit=5000, profile=1)
    out = R.rpa_probe_density(c.ctx, probes, freqs, nl=3)
    c.close()
    assert out["stats"]["tile_rows"] == -7
    ref = oracle.lanczos(s, probes, om[freqs], 3, tol=1e-12)
    assert np.max(np.abs(out["d"] - ref["d"])) <= 1e-9
    c, _ = solver(s, precision="mixed", stern_tol=1e-10, refine=4, stern_maxit=5000)
    u = np.random.default_rng(7).standard_normal((2, s.N_d))
    r, _ = R.rpa_chi0(c.ctx, om[[0, 2]], u, s.ns)
    c.close()
    for i, o in enumerate((om[0], om[2])):
        want, _ = oracle.chi0(s, o, u[i], tol=1e-12)
        assert np.max(np.abs(r[i] - want)) <= 1e-7 * np.max(np.abs(want))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_iteration_cap(prec):
    s = system("per")
    c, _ = solver(s, precision=prec, stern_tol=1e-12, stern_maxit=3, lanczos_max=2, profile=1)
    probes, freqs = np.array([5, 300], dtype=np.int64), np.array([0, 3], dtype=np.int32)
    out = R.rpa_probe_density(c.ctx, probes, freqs, nl=2, allow_nonconv=True)
    assert out["stats"]["tile_rows"] == -7 and out["stats"]["nonconv_solves"] > 0
    assert out["status"] == R.RPA_ENOCONV and np.isfinite(out["d"]).all()
    R.rpa_set_options(c.ctx, precision=prec, stern_tol=1e-8, stern_maxit=20000, lanczos_max=2)
    assert R.rpa_probe_density(c.ctx, probes, freqs, nl=2)["status"] == R.RPA_OK
    c.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("where", ["orbital", "potential", "projector"])
def test_non_finite_input_breaks_down(prec, where):
    """NaN in one input: every solve that meets it ends with a breakdown, and the context works again
    with the clean input."""
    s = system("per")
    c, _ = solver(s, precision=prec, stern_tol=1e-8, lanczos_max=2)
    probes, freqs = np.array([5, 44], dtype=np.int64), np.array([1, 2], dtype=np.int32)
    good = R.rpa_probe_density(c.ctx, probes, freqs, nl=2)["d"]
    groups = [(g.idx, g.chi, g.gamma) for g in s.groups]
    if where == "orbital":
        a = np.array(s.psi, copy=True)
        a[1, 17] = np.nan
        R.rpa_set_occupied(c.ctx, a, s.eps)
    elif where == "potential":
        a = np.array(s.vloc, copy=True)
        a.reshape(-1)[17] = np.nan
        R.rpa_set_potential(c.ctx, a)
    else:
        a = np.array(groups[0][1], copy=True)
        a[0, 3] = np.nan
        R.rpa_set_projectors(c.ctx, [(groups[0][0], a, groups[0][2])] + groups[1:])
    with pytest.raises(R.RpaError) as e:
        R.rpa_probe_density(c.ctx, probes, freqs, nl=2)
    assert e.value.status == R.RPA_EBREAKDOWN
    R.rpa_set_occupied(c.ctx, s.psi, s.eps)
    R.rpa_set_potential(c.ctx, s.vloc)
    R.rpa_set_projectors(c.ctx, groups)
    again = R.rpa_probe_density(c.ctx, probes, freqs, nl=2)["d"]
    c.close()
    assert np.allclose(again, good, rtol=1e-9 if prec == "fp64" else 1e-6, atol=0)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_lanes(prec):
    s = system("per")
    probes = np.arange(5, s.N_d, 131, dtype=np.int64)[:11]
    freqs = (np.arange(len(probes)) % 4).astype(np.int32)
    out = {}
    for lanes in (1, 3):
        c, _ = solver(s, precision=prec, lanczos_max=4, stern_tol=1e-10, stern_maxit=5000,
                      lanes=lanes, profile=1)
        out[lanes] = R.rpa_probe_density(c.ctx, probes, freqs, nl=4, want_tridiag=True)
        c.close()
    a, b = out[1], out[3]
    assert a["stats"]["tile_rows"] == b["stats"]["tile_rows"] == -7
    rt = 1e-9 if prec == "fp64" else 1e-6
    assert np.allclose(a["d"], b["d"], rtol=rt, atol=0)
    assert np.array_equal(a["steps"], b["steps"])
    assert a["stats"]["solves"] == b["stats"]["solves"]


def test_contexts_on_threads():
    """Contexts of one grid, one thread and stream each, at the same time: the results of each alone."""
    s = system("per")
    om = np.array([0.3, 1.0])
    u = np.random.default_rng(2).standard_normal((4, 2, s.N_d))
    cs = [solver(s, precision="fp64", stern_tol=1e-9)[0] for _ in range(4)]
    alone = [R.rpa_chi0(c.ctx, om, x, s.ns)[0] for c, x in zip(cs, u)]
    got = [None] * 4

    def work(i):
        for _ in range(5):
            got[i] = R.rpa_chi0(cs[i].ctx, om, u[i], s.ns)[0]
    th = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for c in cs:
        c.close()
    for a, b in zip(alone, got):
        assert np.array_equal(a, b)
