"""Batches whose components hold more elements than a 32-bit byte offset of the FP64 state reaches (2^29):
a context accepts them and every event gets the bits of a context of its own; a single event of that size
is refused in mixed precision (it would not fit on the device) before any device work."""
import ctypes as C

import numpy as np
import pytest

from workload.problem import hotspot_problem


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


def _init(grids, precision):
    """kt_init_batch's status for these grids; a tiny arena keeps every accepted call from allocating."""
    from paper_1608_06577_gb300 import binding
    L = binding.load_library()
    o = binding.Options()
    L.kt_options_default(C.byref(o))
    o.precision = precision
    buf = C.create_string_buffer(256)
    o.arena, o.arena_bytes = C.c_void_p(C.addressof(buf)), 256
    g = (binding.Grid * len(grids))(*[binding.Grid(*s) for s in grids])
    eos = binding.Eos(0, 15.6, 0, None, None, None, None, None)
    z = binding.Coef(0, 0.0, 0.0, 1.0)
    ctx = C.c_void_p()
    return L.kt_init_batch(C.byref(ctx), len(grids), g, 0.1, 0.1, 0.01, C.byref(eos), C.byref(z), C.byref(z), C.byref(o))


# padded cells: 1020+4 times 1020+4 times 508+4 = 2^29 exactly, one plane fewer, and the 240-event batch
@pytest.mark.parametrize("grids,mixed_ok", [([(1020, 1020, 508)], False), ([(1020, 1020, 507)], True),
                                            ([(8, 8, 8), (2044, 1020, 508)], False), ([(128, 128, 128)] * 240, True)])
def test_size_of_one_event_is_what_counts(grids, mixed_ok):
    accepted = (-2, -3)  # no device here, or the arena is too small: past the argument checks
    assert _init(grids, 0) in accepted
    rc = _init(grids, 1)
    assert (rc in accepted) if mixed_ok else rc == -1, rc


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["plain", "fused", "staged", "pi32"])
def test_events_beyond_32_bit_byte_offsets(mode, baseline_eos):
    import torch
    from paper_1608_06577_gb300 import KT, KT_INV_CONFORMAL, KT_MIXED
    nev, n = 236, 128
    elements = nev * 132 ** 3
    assert elements > 1 << 29 and (nev - 4) * 132 ** 3 < 1 << 29
    free = torch.cuda.mem_get_info()[0]
    if free < 434 * elements + (8 << 30):
        pytest.skip(f"needs {434 * elements >> 30} GiB of device memory and 8 GiB of room")
    kw = {"precision": KT_MIXED, "pi_fp32": mode == "pi32", "autotune": False}
    if mode == "fused":
        kw["inversion"] = KT_INV_CONFORMAL
    cand = {"plain": 11, "fused": 35, "staged": 22, "pi32": 10}[mode]
    p = hotspot_problem(nx=n, ny=n, neta=n, nhot=20, seed=3, r_max=4.0, eos_table=baseline_eos)
    if mode == "plain":
        p = p.replace(iface="invert")  # the face velocities go through borrowed fields too
    X, Y, Z = p.coords_xyz()
    u = torch.as_tensor(np.stack([0.2 * np.tanh(X).ravel(), -0.1 * np.tanh(Y).ravel(), 0.1 * np.tanh(Z).ravel()]),
                        device="cuda")
    pi = torch.zeros((10, p.ncells), dtype=torch.float64, device="cuda")
    e0 = torch.as_tensor(p.e, device="cuda")
    scale = (1.0, 1.25, 0.75)
    es = [s * e0 for s in scale]
    p.e = p.u = p.pi = p.Pi = None
    ref, diag = [], []
    for e in es:
        pi[4], pi[7] = 0.02 * e, -0.02 * e
        k = KT(p, **kw)
        k.set_tuning(cand)
        k.set_state(p.tau0, e, u, pi, -0.02 * e)
        k.step(2)
        q = torch.empty((15, p.ncells), dtype=torch.float64, device="cuda")
        k.get_state_device(q=q)
        ref.append(q)
        diag.append(k.diagnostics())
        del k
    big = KT([p] * nev, use_graph=False, **kw)
    big.set_tuning(cand)
    for ev in range(nev):
        e = es[ev % 3]
        pi[4], pi[7] = 0.02 * e, -0.02 * e
        big.set_state(p.tau0, e, u, pi, -0.02 * e, event=ev)
    big.step(2)
    q = torch.empty((15, p.ncells), dtype=torch.float64, device="cuda")
    for ev in range(nev):
        big.get_state_device(q=q, event=ev)
        assert torch.equal(q, ref[ev % 3]), ev
    for ev in (0, nev - 1):
        d = big.diagnostics(event=ev)
        assert all(np.array_equal(d[f], diag[ev % 3][f]) for f in d), ev
    del big, ref
    torch.cuda.empty_cache()
