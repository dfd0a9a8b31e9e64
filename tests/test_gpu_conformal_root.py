"""FP64 mode, conformal EOS: the closed form e = 3 (E - M)(E + M) / (sqrt(4 E^2 - 3 M^2) + E) with every
operation rounded once, bit for bit against rational arithmetic."""
import math
from fractions import Fraction

import numpy as np
import pytest

from workload.problem import Problem, conformal_eos

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


def _closed_form(E, M2):
    M = math.sqrt(M2)
    r = Fraction(-3.0 * M2) + Fraction(4.0 * E) * Fraction(E)
    return (3.0 * (E - M) * (E + M)) / (math.sqrt(float(r)) + E)  # float(r): rounded to nearest, as fma


def test_conformal_energy_density_is_correctly_rounded():
    from paper_1608_06577_gb300 import KT
    n = 3000
    # uniform pressure gradients vanish only at rest; dtau = 1e-30 leaves the state as it was put in
    p = Problem("conformal", n, 1, 1, 0.1, 0.1, 0.1, 1e-30, 1.0, 1, coords="cartesian", eos=conformal_eos())
    rng = np.random.default_rng(5)
    p.e = np.exp(rng.uniform(np.log(1e-3), np.log(1e3), n))
    p.u = np.zeros((3, n))
    p.u[0] = rng.uniform(-3.0, 3.0, n)
    k = KT(p)
    k.set_problem_state()
    k.step(1)
    s = k.get_state(fields=("e", "q"))
    want = np.array([_closed_form(s["q"][0, c], s["q"][1, c] * s["q"][1, c]) for c in range(n)])
    assert np.sum(s["e"] != want) == 0, np.max(np.abs(s["e"] / want - 1.0))
