"""kt_set_state / kt_get_state / kt_get_checkpoint through device arrays and host arrays: the same state
and the same values, at cell counts around a block's 256 and for single cells, in every storage mode."""
import numpy as np
import pytest

from test_gpu_parity import FIELDS
from workload.problem import hotspot_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


@pytest.mark.parametrize("mode", ["fp64", "mixed", "pi32"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 17, 3), (16, 4, 4), (257, 1, 1), (33, 31, 2)])
def test_device_and_host_io_agree(mode, shape, baseline_eos):
    import ctypes as C
    import torch
    from paper_1608_06577_gb300 import KT
    nx, ny, nz = shape
    p = hotspot_problem(nx=nx, ny=ny, neta=nz, nhot=5, seed=3, r_max=0.8, eos_table=baseline_eos)
    rng = np.random.default_rng(5)
    n = p.ncells
    p.u = rng.uniform(-0.3, 0.3, (3, n))
    p.u[0, 0] = 1e-41  # rounds to an FP32 value below the smallest normal
    p.pi = 0.01 * p.e * rng.standard_normal((10, n))
    p.Pi = -0.01 * p.e
    up = 0.9 * p.u
    kw = {"fp64": {}, "mixed": {"precision": 1}, "pi32": {"precision": 1, "pi_fp32": True}}[mode]
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    a, b = KT(p, **kw), KT(p, **kw)
    a.set_state(p.tau0, p.e, p.u, p.pi, p.Pi, up)
    b.set_state(p.tau0, dev(p.e), dev(p.u), dev(p.pi), dev(p.Pi), dev(up))
    sizes = {"e": (n,), "u": (4, n), "pi": (10, n), "Pi": (n,), "q": (15, n)}
    for _ in range(2):
        ha, hb = a.get_state(), b.get_state()
        out = {f: torch.full(sizes[f], float("nan"), dtype=torch.float64, device="cuda") for f in FIELDS}
        assert a.get_state_device(**out) == ha["tau"] == hb["tau"]
        for f in FIELDS:
            assert np.array_equal(ha[f], hb[f]), f
            assert np.array_equal(ha[f], out[f].cpu().numpy()), f
        tau, ck = a.get_checkpoint()
        dck = torch.full((41, n), float("nan"), dtype=torch.float64, device="cuda")
        t = C.c_double()
        assert a.L.kt_get_checkpoint(a.ctx, 0, C.byref(t), C.c_void_p(dck.data_ptr()), 1) == 0
        assert t.value == tau and np.array_equal(ck, dck.cpu().numpy())
        a.step(2)
        b.step(2)
    if mode == "fp64":  # what went in comes out
        c = KT(p)
        c.set_state(p.tau0, dev(p.e), dev(p.u), dev(p.pi), dev(p.Pi))
        s = c.get_state()
        assert np.array_equal(s["e"], p.e) and np.array_equal(s["u"][1:], p.u)
        assert np.array_equal(s["pi"], p.pi) and np.array_equal(s["Pi"], p.Pi)


def test_host_arrays_that_adjoin(baseline_eos):
    """Output arrays pinned one by one that follow one another in memory: no copy spans two of them."""
    import ctypes as C
    import mmap
    import torch
    from paper_1608_06577_gb300 import KT
    p = hotspot_problem(nx=16, ny=16, neta=32, nhot=5, seed=3, r_max=0.8, eos_table=baseline_eos)
    n = p.ncells
    sizes = {"e": (n,), "u": (4, n), "pi": (10, n), "Pi": (n,)}
    buf = mmap.mmap(-1, 16 * n * 8)
    assert (n * 8) % mmap.PAGESIZE == 0
    base = C.addressof(C.c_char.from_buffer(buf))
    out, at, rt, pinned = {}, 0, torch.cuda.cudart(), []
    try:
        for f, s in sizes.items():
            nb = int(np.prod(s)) * 8
            out[f] = np.frombuffer(buf, dtype=np.float64, count=nb // 8, offset=at).reshape(s)
            assert int(rt.cudaHostRegister(base + at, nb, 0)) == 0
            pinned.append(base + at)
            at += nb
        a = KT(p, precision=1)
        a.set_problem_state()
        ref = a.get_state()
        got = a.get_state(fields=tuple(sizes), out=out)
        for f in sizes:
            assert np.array_equal(got[f], ref[f]), f
    finally:
        for q in pinned:
            rt.cudaHostUnregister(q)
