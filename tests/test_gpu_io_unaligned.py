"""Device arrays that kernels cannot use in place (here: at an odd offset of four bytes) are copied in and out:
kt_set_state, kt_get_state and kt_get_checkpoint give the same values as with aligned ones, also where some
arrays of a call are aligned and others are not."""
import ctypes as C

import numpy as np
import pytest

from test_gpu_fp64_strips import _viscous

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1608_06577_gb300 import build
    build.build()


class _At:
    """A device array of `n` doubles `off` bytes into an allocation."""

    def __init__(self, n, off, values=None):
        import torch
        self.buf = torch.full((8 * n + 16,), 0xff, dtype=torch.uint8, device="cuda")
        self.n, self.off = n, off
        if values is not None:
            b = np.ascontiguousarray(values, dtype=np.float64).ravel().view(np.uint8)
            self.buf[off:off + 8 * n] = torch.as_tensor(b, device="cuda")
        self.ptr = C.c_void_p(self.buf.data_ptr() + off)

    def get(self):
        return self.buf[self.off:self.off + 8 * self.n].cpu().numpy().view(np.float64)


@pytest.mark.parametrize("mode", ["fp64", "mixed"])
@pytest.mark.parametrize("offsets", [(4, 4, 4, 4, 4), (0, 4, 0, 4, 0), (8, 0, 1, 0, 7)])
def test_odd_offsets(mode, offsets, baseline_eos):
    import torch
    from paper_1608_06577_gb300 import KT
    p = _viscous(13, 7, 5, baseline_eos)
    n, kw = p.ncells, ({"precision": 1} if mode == "mixed" else {})
    a, b = KT(p, **kw), KT(p, **kw)
    up = 0.9 * p.u
    a.set_state(p.tau0, p.e, p.u, p.pi, p.Pi, up)
    ins = [_At(v.size, o, v) for v, o in zip((p.e, p.u, p.pi, p.Pi, up), offsets)]
    torch.cuda.synchronize()
    assert b.L.kt_set_state_event(b.ctx, 0, p.tau0, *[i.ptr for i in ins], 1) == 0
    for _ in range(2):
        ref = a.get_state()
        outs = [_At(r * n, o) for r, o in zip((1, 4, 10, 1, 15), offsets)]
        torch.cuda.synchronize()
        assert b.L.kt_get_state_event(b.ctx, 0, None, *[o.ptr for o in outs], 1) == 0
        for f, o in zip(("e", "u", "pi", "Pi", "q"), outs):
            assert np.array_equal(o.get(), ref[f].ravel()), f
            assert bool((o.buf[:o.off] == 0xff).all()) and bool((o.buf[o.off + 8 * o.n:] == 0xff).all()), f
        ck = _At(41 * n, offsets[1])
        torch.cuda.synchronize()
        assert b.L.kt_get_checkpoint(b.ctx, 0, None, ck.ptr, 1) == 0
        assert np.array_equal(ck.get(), a.get_checkpoint()[1].ravel())
        a.step(2)
        b.step(2)
