"""kt_set_state at the ends of the number range: values that round to FP32 numbers below the smallest normal
one are stored as those, and the inversion's admissibility does not depend on the range of FP32."""
import numpy as np
import pytest

from workload.problem import Problem, conformal_eos

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


def _cells(n, **kw):
    p = Problem("cells", n, 1, 1, 0.1, 0.1, 0.1, 0.01, 1.0, 1, eos=conformal_eos(), **kw)
    p.e, p.u, p.pi, p.Pi = np.ones(n), np.zeros((3, n)), np.zeros((10, n)), np.zeros(n)
    return p


@pytest.mark.parametrize("mode", ["mixed", "pi32"])
def test_subnormal_values_round_to_nearest(mode):
    from paper_1608_06577_gb300 import KT
    tiny = np.array([1e-38, 1.2e-38, 3e-39, 1e-40, 7e-43, 1.4e-45, 2.1e-45, 8e-46, 6e-46, 1e-300, 0.0])
    p = _cells(tiny.size)
    p.e[:] = np.where(tiny > 1e-45, tiny, 1.0)
    p.u[0] = np.where(p.e == 1.0, 1.0, 0.0)
    p.pi[4], p.pi[7], p.u[1] = tiny, -tiny, 0.0
    p.Pi[:] = -tiny
    k = KT(p, precision=1, pi_fp32=mode == "pi32")
    k.set_state(p.tau0, p.e, p.u, p.pi, p.Pi * (p.e == 1.0))
    s = k.get_state()
    assert np.array_equal(s["e"], p.e.astype(np.float32).astype(np.float64))
    as_stored = (lambda a: a.astype(np.float32).astype(np.float64)) if mode == "pi32" else (lambda a: a)
    assert np.array_equal(s["pi"][4], as_stored(tiny)) and np.array_equal(s["pi"][7], as_stored(-tiny))
    assert np.array_equal(s["Pi"], as_stored(p.Pi * (p.e == 1.0)))
    _, ck = k.get_checkpoint()  # rows 15-29: the copy the stencil reads
    assert np.array_equal(ck[15 + 8], tiny.astype(np.float32).astype(np.float64))
    p.e[:] = 1.0
    p.u[0], p.u[1] = tiny, -tiny
    k.set_state(p.tau0, p.e, p.u)
    s = k.get_state()
    assert np.array_equal(s["u"][1], tiny.astype(np.float32).astype(np.float64))
    assert np.array_equal(s["u"][2], -tiny.astype(np.float32).astype(np.float64))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("tau", [1e-25, 1e-21, 1e-8, 1.0, 1e8, 1e15, 2e19, 3e20, 1e60, 1e120])
def test_inadmissible_states_at_any_time(precision, tau):
    """e = 100, e + P0 + Pi = -1: T^{tau tau} = 101 - u_tau^2 and |T^{tau i}| = u_tau |u|; tau u^eta = 3 is
    admissible (91 against 9.5), tau u^eta = 9 is not (19 against 81)."""
    from paper_1608_06577_gb300 import KT
    from paper_1608_06577_gb300.binding import KTError
    p = _cells(33)
    p.e[:] = 100.0
    p.Pi[:] = -101.0 - 100.0 / 3.0
    k = KT(p, precision=precision)
    for tu, ok in ((3.0, True), (9.0, False)):
        p.u[2] = 0.0
        p.u[2, -1] = tu / tau
        if ok:
            k.set_state(tau, p.e, p.u, None, p.Pi)
        else:
            with pytest.raises(KTError) as err:
                k.set_state(tau, p.e, p.u, None, p.Pi)
            assert err.value.code == -5  # KT_ERR_STATE
