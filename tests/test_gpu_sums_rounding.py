"""Rounding of the FP32-f velocity sums with a thread per cell: one step's error in W against the FP64
form from the same f is no larger than that of the kernel with several warps per cell, which adds
the same FP32 products in another order.  Both errors are rms over 8160 cells (1 / sqrt(2 n) = 0.8 %
sampling error each): their ratio may exceed 1 by 5 % at most.
"""
import numpy as np
import pytest

from paper_1810_08137_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_vel,vrange,rough", [(28, 4.0, False), (28, 4.0, True), (37, 4.0, False), (64, 4.0, True),
                                                (51, 20.0, False)])
def test_error_of_w_no_larger_than_a_warp_per_cell(n_vel, vrange, rough):
    from paper_1810_08137_gb300 import build, ugks
    build.build()
    cfg = I.channel_config(nx=120, ny=68, n_vel=n_vel, vrange=vrange, kn=0.05)
    r = I.uniform01(61, 4 * cfg.nc).reshape(4, cfg.nc)
    if rough:
        prim = (0.8 + 0.4 * r[0], 0.6 * r[1] - 0.3, 0.6 * r[2] - 0.3, 0.8 + 0.4 * r[3])
    else:
        x = (np.arange(cfg.nc) % cfg.nx + 0.5) / cfg.nx
        prim = (1.2 - 0.2 * x + 2e-3 * r[0], 0.05 + 2e-3 * r[1], 2e-3 * r[2], 1.0 + 2e-3 * r[3])

    def step(form, split, f, W, steps=1):
        with ugks.Solver(cfg, form) as s:
            if form == ugks.FP32F:
                s.set_sums_split(split)
            s.set_state(f, W)
            s.step(steps)
            return s.get_state()

    with ugks.Solver(cfg, ugks.FP32F) as s:  # f as the FP32-f form holds it, after a few steps
        s.init_maxwellian(*prim)
        s.step(0 if rough else 10)
        f, W = s.get_state()
    ref = step(ugks.FP64, 0, f, W)[1]
    err = {}
    for split in (0, 2):
        d = step(ugks.FP32F, split, f, W)[1] - ref
        err[split] = np.sqrt(np.mean(d * d, axis=1))
    assert np.all(err[0] <= 1.05 * err[2]), (err[0], err[2], err[0] / err[2])
