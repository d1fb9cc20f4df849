"""One-block-per-cell kernels of the FP64 and DF64 forms, the interface in the moving frame and
the one-pass ghost ring: one step against the oracle at the edges of their splits -- u tables of
40 (40, 41, 81 and 512 columns), the smallest velocity grids, meshes of one row or column, 8 x 4
tiles with remainders, every kind of boundary meeting at a corner -- and in flows up to about Mach
1.5, where the half-range error function leaves its series (U^2 / T > 0.25).  Bounds: one step of
the FP64 and DF64 forms <= 1e-12 per field, of the FP32-f form <= 1e-6 (f <= 1e-5).
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


P, WL, PR = I.BC(I.BC_PERIODIC), I.BC(I.BC_WALL, T=1.1, U=0.1), I.BC(I.BC_PRESSURE, 1.1, 1.05)
BOX = [P, P, P, P]
CHANNEL = [I.BC(I.BC_PRESSURE, 1.2), I.BC(I.BC_PRESSURE, 1.0), WL, I.BC(I.BC_WALL)]

CASES = [  # nx, ny, nu, nv, boundaries, K, flow
    (3, 2, 40, 5, CHANNEL, 1, 0.3),
    (3, 2, 41, 8, CHANNEL, 1, 0.3),
    (2, 5, 81, 9, BOX, 2, 0.3),
    (2, 2, 512, 4, BOX, 0, 0.3),
    (1, 2, 4, 512, CHANNEL, 1, 0.3),
    (1, 1, 3, 3, CHANNEL, 1, 0.3),
    (1, 1, 6, 4, CHANNEL, 1, 0.3),
    (4, 3, 7, 1, BOX, 1, 0.3),
    (4, 3, 1, 7, BOX, 1, 0.3),
    (17, 9, 6, 5, CHANNEL, 1, 0.3),
    (8, 4, 12, 12, [PR, PR, P, P], 1, 0.3),
    (9, 5, 12, 12, [WL, PR, PR, WL], 1, 0.3),
    (7, 5, 12, 12, [P, P, PR, WL], 2, 0.3),
    (12, 7, 24, 24, BOX, 1, 1.2),
    (12, 7, 25, 25, [PR, PR, PR, PR], 0, 1.2),
]


@pytest.mark.parametrize("form", ["FP64", "DF64", "FP32F"])
@pytest.mark.parametrize("nx,ny,nu,nv,bc,K,flow", CASES)
def test_one_step_against_oracle(U, oracle, form, nx, ny, nu, nv, bc, K, flow):
    one_u, one_v = nu == 1, nv == 1
    cfg = I.Config(nx=nx, ny=ny, lx=1.0, ly=1.0, nu=nu, nv=nv, K=K, kn=0.05, bc=list(bc),
                   umin=0.0 if one_u else -4.0, umax=0.0 if one_u else 4.0,
                   vmin=0.0 if one_v else -4.0, vmax=0.0 if one_v else 4.0)
    r = I.uniform01(23, 4 * cfg.nc).reshape(4, cfg.nc)
    f, W = oracle.init_maxwellian(cfg, 0.8 + 0.4 * r[0], flow * (2 * r[1] - 1), flow * (2 * r[2] - 1),
                                  0.8 + 0.4 * r[3])
    f = f * I.perturbation(24, f.shape, 0.2)
    fr, Wr = oracle.step(cfg, f, W, 1)
    with U.Solver(cfg, getattr(U, form)) as s:
        s.set_state(f, W)
        s.step(1)
        fg, Wg = s.get_state()
    wtol, ftol = (1e-6, 1e-5) if form == "FP32F" else (1e-12, 1e-12)
    ew = np.max(np.abs(Wg - Wr), axis=1) / np.maximum(np.max(np.abs(Wr), axis=1), 1e-300)
    assert np.all(ew <= wtol), ew
    assert np.max(np.abs(fg - fr)) <= ftol * np.max(np.abs(fr))
