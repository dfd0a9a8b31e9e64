"""Face velocities by root-finds keep their results in fields that other parts of a step use too (k_2 in the first
stage, the FP32 copy of q^n in the second): with every start of the root-find, every split update and both kinds
of boundary the results are those of the FP64 mode, and the same bits whatever the layout."""
import numpy as np
import pytest

from test_gpu_fp64_strips import _viscous
from test_gpu_mlp import _newton_counts, _small, trained  # noqa: F401

pytestmark = pytest.mark.gpu

STARTS = {"plain": {}, "conformal": {"inversion": 2}, "learned": {"inversion": 1},
          "learned_pi32": {"inversion": 1, "pi_fp32": True}}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


# 2e-5 of the largest |q| after five steps: the tolerance of test_gpu_faces.py, for the same reasons (an accepted
# root of the learned start is off by 1e-10 E at most)
@pytest.mark.parametrize("start", list(STARTS))
@pytest.mark.parametrize("bc", ["copy", "periodic"])
def test_every_start_and_update(start, bc, baseline_eos):
    from paper_1608_06577_gb300 import KT, KT_MIXED
    kw = dict(STARTS[start], precision=KT_MIXED)
    if "learned" in start:
        kw["mlp_weights"] = (np.random.default_rng(3).normal(size=1313) * 0.05).astype(np.float32)
    probs = [_viscous(*s, baseline_eos, theta=1.3).replace(iface="invert", bc=bc) for s in ((40, 9, 6), (33, 5, 3))]
    ref = []
    for p in probs:
        k = KT(p)
        k.set_problem_state()
        k.step(5)
        ref.append(k.get_state()["q"])
    first = None
    for cand in (0, 11, 12, 22, 23, 35):  # plain updates, TMA-staged ones, and a fused candidate (runs split)
        k = KT(probs, **kw)
        k.set_tuning(cand)
        k.set_problem_state()
        k.step(5)
        out = [k.get_state(event=ev)["q"] for ev in range(2)]
        first = first or out
        for ev in range(2):
            assert np.max(np.abs(out[ev] - ref[ev])) <= 2e-5 * np.max(np.abs(ref[ev][0])), (cand, ev)
            assert np.array_equal(out[ev], first[ev]), (cand, ev)


def test_network_reads_its_own_features(trained):  # noqa: F811
    """With the face velocities in the fields that the network's features come from in the next step, the network
    still saves the steps that it saves with reconstructed faces."""
    params = trained[0].cpu().numpy()
    c = _newton_counts(_small(4).replace(iface="invert"), params, 40)
    (it_l, fb), (it_off, _) = c["trained"], c["network_off"]
    assert fb < 0.02 and it_l <= 0.9 * it_off, (it_l, it_off, fb)
