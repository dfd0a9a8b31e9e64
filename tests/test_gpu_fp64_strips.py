"""The FP64 stage's work split: blocks of 32 consecutive cells in linear order, axes of one cell
skipped, components that vanish in a whole warp skipped.  Against the oracle at the sizes where the
split can go wrong: cell counts around multiples of 32, every combination of one-cell axes, a single
cell, and events of a batch that end inside a strip."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import FIELDS, assert_parity, field_errors, run_pair
from workload.problem import hotspot_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()
    oracle.build()


def _viscous(nx, ny, nz, baseline_eos, **kw):
    p = hotspot_problem(nx=nx, ny=ny, neta=nz, nhot=5, seed=3, r_max=0.8, eos_table=baseline_eos, **kw)
    X, Y, Z = p.coords_xyz()
    p.u = np.stack([0.1 * np.tanh(X + 0.3).ravel(), -0.05 * np.tanh(Y + 0.2).ravel(), 0.2 * np.tanh(Z + 0.1).ravel()])
    p.pi = np.zeros((10, p.ncells))
    p.pi[4], p.pi[7] = 0.01 * p.e, -0.01 * p.e
    p.Pi = -0.01 * p.e
    return p


# 1e-12 per field: the tolerance of every FP64 parity test (rounding of ~1e3 operations per cell and
# ten steps, 1e-16 each, far below it)
@pytest.mark.parametrize("shape", [(1, 1, 1), (31, 1, 1), (33, 1, 1), (1, 37, 1), (1, 1, 35), (9, 7, 1), (11, 1, 3),
                                   (1, 13, 5), (7, 3, 3), (32, 2, 2), (3, 11, 4)])
@pytest.mark.parametrize("theta", [1.0, 1.6])
def test_one_cell_axes_and_strip_remainders(shape, theta, baseline_eos):
    p = _viscous(*shape, baseline_eos, theta=theta)
    g, r, _ = run_pair(p, 6)
    assert_parity(g, r)


@pytest.mark.parametrize("shape", [(19, 1, 5), (6, 9, 1)])
def test_one_cell_axes_periodic_and_inverted_faces(shape, baseline_eos):
    from dataclasses import replace
    p = replace(_viscous(*shape, baseline_eos), bc="periodic")
    g, r, _ = run_pair(p, 6)
    assert_parity(g, r)
    g, r, _ = run_pair(replace(p, bc="copy", iface="invert"), 6)
    assert_parity(g, r)


def test_batch_of_strips_matches_oracle(baseline_eos):
    from paper_1608_06577_gb300 import KT
    probs = [_viscous(*s, baseline_eos) for s in ((33, 1, 1), (8, 4, 1), (5, 5, 5), (1, 1, 1))]
    k = KT(probs)
    k.set_problem_state()
    k.step(5)
    for ev, p in enumerate(probs):
        o = oracle.Oracle(p)
        assert o.step(5) == 0
        r = o.get_state()
        errs = field_errors(k.get_state(event=ev), r)
        assert all(v <= 1e-12 for v in errs.values()), (ev, errs)
        single = KT(p)
        single.set_problem_state()
        single.step(5)
        a, b = k.get_state(event=ev), single.get_state()
        for f in FIELDS:
            assert np.array_equal(a[f], b[f]), (ev, f)


@pytest.mark.parametrize("theta", [1.0, 1.6])
@pytest.mark.parametrize("ideal", [False, True])
def test_four_warp_and_one_warp_kernels_agree_bitwise(theta, ideal, baseline_eos):
    """A grid of few strips runs four warps per strip, a larger one (here: the batch) one; the values are
    added in the same order, so an event gives the same bits in both."""
    from dataclasses import replace
    from paper_1608_06577_gb300 import KT
    probs = [_viscous(*s, baseline_eos, theta=theta)
             for s in ((33, 1, 1), (1, 37, 1), (1, 1, 34), (9, 7, 1), (1, 1, 1), (6, 9, 5), (64, 52, 4))]
    if ideal:
        probs = [replace(p, eta_over_s=("const", 0.0, 0.0, 1.0), zeta_over_s=("const", 0.0, 0.0, 1.0),
                         pi=np.zeros_like(p.pi), Pi=np.zeros_like(p.Pi)) for p in probs]
    k = KT(probs)
    k.set_problem_state()
    k.step(5)
    assert k.tuning()["grid_blocks"] > 304  # one warp per strip
    for ev, p in enumerate(probs[:-1]):
        single = KT(p)
        single.set_problem_state()
        single.step(5)
        assert single.tuning()["grid_blocks"] <= 304
        a, b = k.get_state(event=ev), single.get_state()
        for f in FIELDS:
            assert np.array_equal(a[f], b[f]), (ev, f)
