"""The line between the FP64 kernels of four warps and of one warp per strip of 32 cells: it lies where the
four-warp kernel's blocks no longer are all resident, the reported block says which one runs, and both give
the same bits at the line and beyond it."""
import numpy as np
import pytest

from test_gpu_fp64_strips import _viscous
from test_gpu_parity import FIELDS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


def _strips(n, baseline_eos, **kw):
    """A viscous grid of n strips: rows of 32 cells."""
    return _viscous(32, n, 1, baseline_eos, **kw)


def test_line_and_bits_at_it(baseline_eos):
    import torch
    from paper_1608_06577_gb300 import KT
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    team = [KT(_strips(n, baseline_eos)).tuning() for n in (1, sms, 2 * sms, 3 * sms)]
    one = [KT(_strips(n, baseline_eos)).tuning() for n in (3 * sms + 1, 4 * sms + 1)]
    assert all(t["block"] == (32, 4, 1) for t in team) and all(t["block"] == (32, 1, 1) for t in one)
    assert KT(_strips(4, baseline_eos, ).replace(iface="invert")).tuning()["block"] == (32, 1, 1)
    p = _strips(3 * sms, baseline_eos, theta=1.6)
    single, batch = KT(p), KT([p, _strips(3, baseline_eos, theta=1.6)])  # the batch is three strips over the line
    assert single.tuning()["block"] == (32, 4, 1) and batch.tuning()["block"] == (32, 1, 1)
    for k in (single, batch):
        k.set_problem_state()
        k.step(5)
    a, b = single.get_state(), batch.get_state(event=0)
    for f in FIELDS:
        assert np.array_equal(a[f], b[f]), f


@pytest.mark.parametrize("theta", [1.0, 1.6])
@pytest.mark.parametrize("ideal", [False, True])
def test_small_events_give_the_same_bits_in_a_large_batch(theta, ideal, baseline_eos):
    from dataclasses import replace
    from paper_1608_06577_gb300 import KT
    probs = [_viscous(*s, baseline_eos, theta=theta)
             for s in ((33, 1, 1), (1, 37, 1), (1, 1, 34), (9, 7, 1), (1, 1, 1), (6, 9, 5), (64, 64, 8))]
    if ideal:
        probs = [replace(p, eta_over_s=("const", 0.0, 0.0, 1.0), zeta_over_s=("const", 0.0, 0.0, 1.0),
                         pi=np.zeros_like(p.pi), Pi=np.zeros_like(p.Pi)) for p in probs]
    k = KT(probs)
    k.set_problem_state()
    k.step(5)
    assert k.tuning()["block"] == (32, 1, 1)
    for ev, p in enumerate(probs[:-1]):
        single = KT(p)
        single.set_problem_state()
        single.step(5)
        assert single.tuning()["block"] == (32, 4, 1)
        a, b = k.get_state(event=ev), single.get_state()
        for f in FIELDS:
            assert np.array_equal(a[f], b[f]), (ev, f)
