"""Face velocities by root-finds in mixed precision (one thread per face, every face once): against the
FP64 mode, on grids with one-cell axes and edges inside a block, in every storage mode and in a batch."""
from dataclasses import replace

import numpy as np
import pytest

from test_gpu_fp64_strips import _viscous

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


SHAPES = [(1, 1, 1), (5, 3, 1), (127, 1, 1), (1, 9, 7), (33, 5, 3), (64, 9, 6)]


# A face root stops at 2^-21 E, so v^d carries up to ~1e-6: with dtau/dx = 0.05 and six faces 3e-7 of the
# largest |q| per stage, as much again from the FP32 fluxes: 6e-6 over ten stages, 2e-5 allowed.
@pytest.mark.parametrize("mode", ["mixed", "pi32"])
@pytest.mark.parametrize("theta", [1.0, 1.6])
def test_inverted_faces_match_fp64(mode, theta, baseline_eos):
    from paper_1608_06577_gb300 import KT, KT_MIXED
    kw = {"precision": KT_MIXED, "pi_fp32": mode == "pi32"}
    probs = [replace(_viscous(*s, baseline_eos, theta=theta), iface="invert") for s in SHAPES]
    batch = KT(probs, **kw)
    batch.set_problem_state()
    batch.step(5)
    for ev, p in enumerate(probs):
        ref, kt = KT(p), KT(p, **kw)
        for k in (ref, kt):
            k.set_problem_state()
            k.step(5)
        a, b = ref.get_state()["q"], kt.get_state()["q"]
        assert np.max(np.abs(a - b)) <= 2e-5 * np.max(np.abs(a[0])), SHAPES[ev]
        assert np.array_equal(b, batch.get_state(event=ev)["q"]), SHAPES[ev]
