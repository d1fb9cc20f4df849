"""Velocity sums with one thread per cell (FP32-f form, meshes that fill the GPU with 8 x 4
tiles): one step against the oracle at the edges of the tiles (ragged meshes, one column, one
row), of the row sums (odd and even velocity counts, more than one segment of u, more than one
FP32 chunk) and on every kind of boundary.  Bounds: those of the FP32-f form's one-step parity.
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


PERIODIC = [I.BC(I.BC_PERIODIC)] * 4
WALLS_X = [I.BC(I.BC_WALL, T=1.1), I.BC(I.BC_WALL, T=1.0, U=0.1),
           I.BC(I.BC_PRESSURE, 1.15, 1.05), I.BC(I.BC_PRESSURE, 0.95, 1.0)]
CHANNEL = [I.BC(I.BC_PRESSURE, 1.2), I.BC(I.BC_PRESSURE, 1.0), I.BC(I.BC_WALL), I.BC(I.BC_WALL, U=0.1)]


@pytest.mark.parametrize("nx,ny,nu,nv,bc,K", [
    (127, 62, 4, 4, CHANNEL, 1),
    (121, 61, 5, 7, CHANNEL, 2),      # u = 0 column and v = 0 row
    (126, 63, 37, 10, WALLS_X, 1),    # two segments of u per half, the second of 2 and 3 columns
    (120, 60, 9, 41, PERIODIC, 1),    # more than one FP32 chunk per quadrant
    (124, 59, 70, 6, PERIODIC, 0),
    (1, 1000, 6, 5, CHANNEL, 1),
    (2000, 1, 5, 6, WALLS_X, 1),
])
def test_one_step_against_oracle(U, oracle, nx, ny, nu, nv, bc, K):
    cfg = I.Config(nx=nx, ny=ny, lx=1.0, ly=1.0, nu=nu, nv=nv, K=K, kn=0.05, bc=list(bc))
    r = I.uniform01(17, 4 * cfg.nc).reshape(4, cfg.nc)
    f, W = oracle.init_maxwellian(cfg, 0.8 + 0.4 * r[0], 0.6 * r[1] - 0.3, 0.6 * r[2] - 0.3, 0.8 + 0.4 * r[3])
    f = f * I.perturbation(18, f.shape, 0.2)
    fr, Wr = oracle.step(cfg, f, W, 1)
    with U.Solver(cfg, U.FP32F) as s:
        s.set_state(f, W)
        s.step(1)
        fg, Wg = s.get_state()
    ew = np.max(np.abs(Wg - Wr), axis=1) / np.maximum(np.max(np.abs(Wr), axis=1), 1e-300)
    assert np.all(ew <= 1e-6), ew
    assert np.max(np.abs(fg - fr)) <= 1e-5 * np.max(np.abs(fr))
