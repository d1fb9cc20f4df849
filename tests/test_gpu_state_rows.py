"""Device rows of the state exchange that a kernel cannot move with 8-byte accesses: the runtime's
copies take them (f of the FP64 form, W of every form)."""
import numpy as np
import pytest

from paper_1810_08137_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["FP64", "FP32F", "DF64"])
@pytest.mark.parametrize("offset", [0, 4, 8])
def test_state_rows_at_any_offset(form, offset):
    torch = pytest.importorskip("torch")
    from paper_1810_08137_gb300 import build, ugks
    build.build()
    cfg = I.Config(nx=9, ny=4, nu=6, nv=5)
    foff = offset if form == "FP64" else 0  # the other forms' f rows are FP64 numbers, 8-byte aligned
    f = np.ldexp(np.round(np.ldexp(I.uniform01(41, cfg.nc * cfg.nq * 2), 10)), -8)  # exact in every form
    W = I.uniform01(42, 4 * cfg.nc)

    def buffer(n, off):
        return torch.zeros(8 * n + 16, dtype=torch.uint8, device="cuda")[off:off + 8 * n]

    def put(b, a):
        b.copy_(torch.from_numpy(a.view(np.uint8)))

    fb, Wb = buffer(f.size, foff), buffer(W.size, offset)
    put(fb, f)
    put(Wb, W)
    with ugks.Solver(cfg, getattr(ugks, form)) as s:
        s.set_state_device(fb.data_ptr(), Wb.data_ptr())
        s.sync()
        fb.zero_()
        Wb.zero_()
        s.get_state_device(fb.data_ptr(), Wb.data_ptr())
        s.sync()
        fh, Wh = s.get_state()
    assert np.array_equal(Wb.cpu().numpy().view(np.float64), W) and np.array_equal(Wh.reshape(-1), W)
    got = fb.cpu().numpy().view(np.float64)
    assert np.array_equal(got, fh.reshape(-1))
    tol = 0.0 if form == "FP64" else 1e-7  # FP32-f: one rounding of f - g_ref
    assert np.max(np.abs(got - f)) <= tol * np.max(np.abs(f))
