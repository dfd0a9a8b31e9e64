"""Face root-finds in FP64 (KT_IFACE_INVERT) whose start lies where E + P0(e) + Pi < 0: with a bulk pressure
near -(e + P0) the face state has its root close to E while the cell it was extrapolated from has its e below
the sign change.  Against the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_acceptance import _hermite
from test_gpu_parity import assert_parity, run_pair
from workload.problem import Problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()
    oracle.build()


def _problem(t, axis):
    n = [1, 1, 1]
    n[axis] = 24
    p = Problem("strong_bulk", *n, 0.1, 0.1, 0.1, 1e-3, 1.0, 1, coords="cartesian", eos=t, iface="invert", regulate=False,
                zeta_over_s=("const", 0.1, 0.0, 1.0), tau_relax_min=1.0)
    i = np.arange(24)
    p.e = 2.0 * 1.25 ** i
    p.u = np.zeros((3, 24))
    p.u[axis] = 2e-3 * np.cos(0.7 * i)
    p.pi = np.zeros((10, 24))
    P0, _ = _hermite(t, p.e)
    p.Pi = -(p.e + P0) + 0.008 * p.e
    return p


def _right_faces(t, p):
    """E + Pi of the left state of every inner right face (theta = 1), A there at the start e_i and at E."""
    P0, _ = _hermite(t, p.e)
    u2 = np.sum(p.u ** 2, axis=0)
    E = (p.e + P0 + p.Pi) * (1.0 + u2) - P0 - p.Pi

    def ext(x):
        d = np.diff(x)
        s = np.where(d[:-1] * d[1:] > 0, np.where(np.abs(d[:-1]) < np.abs(d[1:]), d[:-1], d[1:]), 0.0)
        return x[1:-1] + 0.5 * s
    Ef, Pf = ext(E), ext(p.Pi)
    return Ef + Pf + P0[1:-1], Ef + Pf + _hermite(t, Ef)[0]


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_face_states_with_a_sign_change(axis, baseline_eos):
    p = _problem(baseline_eos, axis)
    at_start, at_E = _right_faces(baseline_eos, p)
    assert np.sum((at_start < 0) & (at_E > 0)) >= 5, (at_start, at_E)
    g, r, _ = run_pair(p, 1)
    assert_parity(g, r)
