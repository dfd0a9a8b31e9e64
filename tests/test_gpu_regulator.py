"""The regulator of Eq. (regPimunu) where the norm of Pi Delta + pi leaves the arithmetic's range: rho is
then as large as it gets and pi goes to zero, in every precision and storage mode."""
import numpy as np
import pytest

from test_gpu_fp64_strips import _viscous

pytestmark = pytest.mark.gpu

MODES = {"fp64": {}, "mixed": {"precision": 1}, "pi32": {"precision": 1, "pi_fp32": True},
         "conformal": {"precision": 1, "inversion": 2}}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


# A single cell at rest has no neighbours and (Cartesian, no bulk pressure) no velocity gradient: pi^{xx}
# only relaxes.  Its square overflows FP32 above 1.8e19, FP64 above 1.3e154.
@pytest.mark.parametrize("mode,size", [(m, s) for m in MODES for s in (1e17, 1e18, 3e19, 1e25, 1e37)] +
                         [("fp64", 1e153), ("fp64", 2e154), ("fp64", 1e200)])
def test_overflowing_norm_means_full_suppression(mode, size, baseline_eos):
    from paper_1608_06577_gb300 import KT
    p = _viscous(1, 1, 1, baseline_eos).replace(coords="cartesian", zeta_over_s=("const", 0.0, 0.0, 1.0),
                                                tau_relax_min=0.1)
    p.u[:] = 0.0
    p.pi[:] = 0.0
    p.Pi[:] = 0.0
    p.pi[4] = size
    k = KT(p, **MODES[mode])
    k.set_problem_state()
    k.step(1)
    s, f = k.get_state(), k.diagnostics()["regulation"][0]
    # the last stage's pi^{xx} before the regulator is between 0.4 and 1 of `size` (a tenth of it relaxes per
    # stage at most, and the second stage averages with a first one that was suppressed)
    P0 = k.get_state(fields=("e",))["e"][0] / 3.0
    assert 0.0 <= f <= 10.0 * p.rho_max * np.sqrt(p.e[0] ** 2 + 3 * P0 ** 2) / size, f
    assert np.all(np.abs(s["pi"]) <= 10.0 * p.e[0]) and np.all(s["Pi"] == 0.0)
    assert s["e"][0] == pytest.approx(p.e[0], rel=1e-6)
    assert k.stats()["reg_min"] == f and k.stats()["regulated"] == 2
