"""Tracing reports the launches that a step has: the ghost ring is one of them, under ghost_x."""
import pytest

from paper_1810_08137_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["FP64", "FP32F", "DF64"])
def test_no_time_without_a_launch(form):
    from paper_1810_08137_gb300 import build, ugks
    build.build()
    cfg = I.channel_config(nx=12, ny=6, n_vel=8)
    with ugks.Solver(cfg, getattr(ugks, form)) as s:
        s.init_maxwellian(*I.initial_prim(cfg, 1))
        s.profile(True)
        s.step(3)
        t = s.kernel_times()
    assert t.pop("ghost_y") == (0, 0.0)
    assert sorted(t) == ["cells", "faces", "ghost_x", "sums", "update"]
    assert all(n == 3 and ms > 0.0 for n, ms in t.values())
