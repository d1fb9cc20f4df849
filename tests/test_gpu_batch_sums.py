"""Batches that hold instances of every kind of the FP32-f velocity sums: a thread per cell (meshes
that fill the device with 8 x 4 tiles), one warp per cell, several warps per cell, and the Shakhov
model.  Each instance must be bitwise the same alone and in the batch, in both step modes, when
an admission brings another kind after an odd number of steps, and when the sums of an instance
in the batch are set anew.
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


def tiled():  # 16 x 16 = 256 ragged tiles, nodes at u = 0 and v = 0
    return I.Config(nx=127, ny=62, lx=1.0, ly=1.0, nu=5, nv=7, kn=0.05,
                    bc=[I.BC(I.BC_PRESSURE, 1.2), I.BC(I.BC_PRESSURE, 1.0), I.BC(I.BC_WALL), I.BC(I.BC_WALL, U=0.1)])


def warps():
    return I.channel_config(nx=37, ny=18, n_vel=33, kn=0.003, rho_in=1.1)


def shakhov():
    return I.channel_config(nx=21, ny=10, n_vel=16, kn=0.1).replace(pr=2.0 / 3.0)


def prim_of(cfg, k):
    return I.initial_prim(cfg, I.seed_for(4, 70 + k), amp=0.02)


def alone(U, cfg, prim, steps, split=0):
    with U.Solver(cfg, U.FP32F) as s:
        s.set_sums_split(split)
        s.init_maxwellian(*prim)
        s.step(steps)
        return s.get_state()


def check(B, slot, ref):
    f, W = B.instance(slot).get_state()
    assert np.array_equal(f, ref[0]) and np.array_equal(W, ref[1])


@pytest.mark.parametrize("persistent", [True, False])
def test_every_kind_of_sums_alone_and_in_a_batch(U, persistent):
    cfgs = [tiled(), warps(), shakhov()]
    prims = [prim_of(c, k) for k, c in enumerate(cfgs)]
    with U.Batch(4) as B:
        B.set_persistent(persistent)
        slots = [B.admit(c) for c in cfgs]
        for s, p in zip(slots, prims):
            B.instance(s).init_maxwellian(*p)
        B.step(5)
        B.sync()
        for c, p, s in zip(cfgs, prims, slots):
            check(B, s, alone(U, c, p, 5))


@pytest.mark.parametrize("persistent", [True, False])
@pytest.mark.parametrize("first", [tiled, warps, shakhov])
def test_admission_of_another_kind_after_odd_steps(U, persistent, first):
    cfgs = [first()] + [f() for f in (tiled, warps, shakhov) if f is not first]
    prims = [prim_of(c, 10 + k) for k, c in enumerate(cfgs)]
    with U.Batch(3) as B:
        B.set_persistent(persistent)
        slots = []
        for c, p in zip(cfgs, prims):  # three steps, then one after each admission
            slots.append(B.admit(c))
            B.instance(slots[-1]).init_maxwellian(*p)
            B.step(3 if len(slots) == 1 else 1)
        B.retire(slots[1])
        B.step(1)
        B.sync()
        check(B, slots[0], alone(U, cfgs[0], prims[0], 6))
        check(B, slots[2], alone(U, cfgs[2], prims[2], 2))


@pytest.mark.parametrize("persistent", [True, False])
def test_sums_set_on_an_instance_of_a_batch(U, persistent):
    """The work table and the descriptors that the device reads agree after the sums of an
    instance were set, before and after other instances come and go."""
    a, b = tiled(), warps()
    pa, pb = prim_of(a, 20), prim_of(b, 21)
    ref = alone(U, a, pa, 3, split=2)
    with U.Batch(2) as B:
        B.set_persistent(persistent)
        sa = B.admit(a)
        B.instance(sa).set_sums_split(2)
        B.instance(sa).init_maxwellian(*pa)
        B.step(1)
        sb = B.admit(b)
        B.instance(sb).init_maxwellian(*pb)
        B.step(1)
        B.retire(sb)
        B.step(1)
        B.sync()
        check(B, sa, ref)
        assert B.instance(sa).sums_split == 2
        B.instance(sa).set_sums_split(0)  # back to a thread per cell
        B.instance(sa).init_maxwellian(*pa)
        B.step(2)
        B.sync()
        check(B, sa, alone(U, a, pa, 2))


@pytest.mark.parametrize("persistent", [True, False])
def test_interface_blocks_follow_the_batch_not_the_result(U, persistent):
    """Two instances of 15937 faces: blocks of 32 faces alone, of 128 together (past 152 x 128
    faces), and back to 32 when one leaves."""
    cfg = tiled()
    prims = [prim_of(cfg, 30 + k) for k in range(2)]
    with U.Batch(2) as B:
        B.set_persistent(persistent)
        slots = [B.admit(cfg), B.admit(cfg)]
        for s, p in zip(slots, prims):
            B.instance(s).init_maxwellian(*p)
        B.step(3)
        check(B, slots[1], alone(U, cfg, prims[1], 3))
        B.retire(slots[1])
        B.step(2)
        B.sync()
        check(B, slots[0], alone(U, cfg, prims[0], 5))


@pytest.mark.parametrize("persistent", [True, False])
def test_wide_grid_in_a_batch(U, persistent):
    """On [-20, 20]^2 the pressure ghosts pass through FP32 subnormals."""
    cfg = I.channel_config(nx=9, ny=4, n_vel=67, vrange=20.0, kn=0.02)
    prim = prim_of(cfg, 40)
    with U.Batch(2) as B:
        B.set_persistent(persistent)
        s, other = B.admit(cfg), B.admit(warps())
        B.instance(s).init_maxwellian(*prim)
        B.instance(other).init_maxwellian(*prim_of(warps(), 41))
        B.step(4)
        B.sync()
        check(B, s, alone(U, cfg, prim, 4))
