"""State exchange of the FP32-f and DF64 forms in the range of FP32 subnormals, where the tails of f
lie on a wide velocity grid.
"""
import numpy as np
import pytest

from paper_1810_08137_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def U():
    from paper_1810_08137_gb300 import build, ugks
    build.build()
    return ugks


def tail_state(cfg, lo, hi):
    """f of magnitude 2^lo .. 2^hi with 53-bit significands and both signs; any W."""
    r = I.uniform01(31, 2 * cfg.nc * cfg.nq * 2).reshape(2, cfg.nc, cfg.nq, 2)
    f = np.ldexp(1.0 + r[0], np.floor(lo + (hi - lo) * r[1]).astype(int))
    f[:, ::3] *= -1.0
    return f, np.ones((4, cfg.nc))


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("shift", [0, 1])
def test_fp32f_subnormals_pass_in_and_out(U, device, shift):
    """With g_ref = 0 at the velocities compared (exp(-|c|^2 / 1e-4) underflows from |c| = 0.3) the
    stored value is f rounded to FP32, ties to even, subnormals kept.  shift 1: rows that are
    8-byte but not 16-byte aligned."""
    torch = pytest.importorskip("torch")
    cfg = I.Config(nx=5, ny=3, nu=8, nv=6, ref=(1.0, 0.0, 0.0, 1e-4))  # no node within 0.3 of c = 0
    f, W = tail_state(cfg, -152, -120)
    with U.Solver(cfg, U.FP32F) as s:
        if device:
            a = torch.zeros(f.size + shift, dtype=torch.float64, device="cuda")
            a[shift:] = torch.from_numpy(f).reshape(-1)
            w = torch.from_numpy(W).cuda()
            s.set_state_device(a[shift:], w)
            a.zero_()
            s.get_state_device(a[shift:], w)
            s.sync()
            got = a[shift:].cpu().numpy().reshape(f.shape)
        else:
            s.set_state(f, W)
            got, _ = s.get_state()
    assert np.array_equal(got, f.astype(np.float32).astype(np.float64))


def test_df64_subnormal_low_words_pass_out(U):
    """2^-103 <= |f|: the low word of the pair holds the remainder, at these sizes as an FP32
    subnormal: half a unit of 2^-149, and the pair's 2^-47 of the value."""
    cfg = I.Config(nx=5, ny=3, nu=8, nv=6)
    f, W = tail_state(cfg, -102, -98)
    with U.Solver(cfg, U.DF64) as s:
        s.set_state(f, W)
        got, _ = s.get_state()
    assert np.all(np.abs(got - f) <= 2.0 ** -47 * np.abs(f) + 2.0 ** -150)


def test_fp32f_resume_on_a_wide_grid_bitwise(U):
    """A checkpoint of a flow on [-20, 20]^2, whose tails reach from normal numbers through the
    subnormals to zero, resumes bitwise."""
    cfg = I.channel_config(nx=12, ny=6, n_vel=101, vrange=20.0, kn=0.01, rho_in=1.05)
    r = I.uniform01(5, 4 * cfg.nc).reshape(4, cfg.nc)
    prim = (1.0 + 0.05 * r[0], 0.1 * r[1], 0.1 * r[2], 0.9 + 0.2 * r[3])
    with U.Solver(cfg, U.FP32F) as s:
        s.init_maxwellian(*prim)
        s.step(3)
        fc, Wc = s.get_state()
        s.step(2)
        fa, Wa = s.get_state()
    with U.Solver(cfg, U.FP32F) as s:
        s.set_state(fc, Wc)
        s.step(2)
        fb, Wb = s.get_state()
    assert np.array_equal(Wa, Wb) and np.array_equal(fa, fb)
