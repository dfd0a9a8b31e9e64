"""The generalised minmod of the mixed-precision stencil (clamped mean, x and y in pairs) against the
FP64 mode's, over theta and on grids whose edges cut the tiles."""
import numpy as np
import pytest

from test_gpu_fp64_strips import _viscous

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


# A flux difference sums about a dozen products of size |q|/dx, each good to a few 2^-24; with dtau/dx =
# 0.05 that is 3e-7 of the largest |q| per stage, 3e-6 over ten stages: 1e-5 allowed.
@pytest.mark.parametrize("theta", [1.0, 1.0 + 2.0 ** -20, 1.3, 1.8, 2.0])
@pytest.mark.parametrize("shape", [(5, 3, 1), (33, 5, 3), (64, 9, 6)])
def test_mixed_slopes_match_fp64(theta, shape, baseline_eos):
    from paper_1608_06577_gb300 import KT, KT_MIXED
    p = _viscous(*shape, baseline_eos, theta=theta)
    ref = KT(p)
    ref.set_problem_state()
    ref.step(5)
    a = ref.get_state()["q"]
    out = []
    for cand in (11, 0, 35):  # split launches on two tile shapes, the fused launch
        kt = KT(p, precision=KT_MIXED)
        kt.set_tuning(cand)
        kt.set_problem_state()
        kt.step(5)
        out.append(kt.get_state()["q"])
    assert np.max(np.abs(out[0] - a)) <= 1e-5 * np.max(np.abs(a[0]))
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
