"""Body regions that cover a periodic x axis entirely (the rows of the shell are
then taken whole), static and moving, against the oracle; and a body that stops:
its covered / uncovered list is applied to the solid flags once and left empty."""
import ctypes as C

import numpy as np
import pytest

from parity_util import TOL_FP16_POP, TOL_FP64_POP, TOL_RED_POP, pop_error
from test_snapshot_versions_gpu import FLAGS, _parse

pytestmark = pytest.mark.gpu

# region of a body: 2 ceil(R) + 13 cells an axis
CASES = {
    "disc_moving": dict(lattice="D2Q9", n=(23, 41), tau=0.7,
                        bodies=[dict(shape="cylinder", R=4.1, X0=(20.3, 19.6), U=(0.05, -0.03), W=0.002)]),
    "disc_static": dict(lattice="D2Q9", n=(15, 30), tau=0.6, u0=(0.02, 0.03),
                        bodies=[dict(shape="cylinder", R=5.0, X0=(0.7, 14.2))]),
    "sphere_moving": dict(lattice="D3Q19", n=(23, 26, 31), tau=0.65, u0=(0.0, 0.01, 0.0),
                          bodies=[dict(shape="sphere", R=4.1, X0=(1.2, 11.3, 27.9), U=(-0.06, 0.02, 0.04))]),
    "ellipse_moving": dict(lattice="D2Q9", n=(23, 40), tau=0.7,
                           bodies=[dict(shape="ellipse", R=4.4, R2=2.5, theta0=0.6, X0=(11.0, 20.0), U=(0.04, 0.0),
                                        W=0.004)]),
}


@pytest.mark.parametrize("prec,tol", [("fp64", TOL_FP64_POP), ("fp32", TOL_RED_POP), ("fp16", TOL_FP16_POP)])
@pytest.mark.parametrize("name", sorted(CASES))
def test_region_covers_the_periodic_x_axis(oracle_mod, name, prec, tol):
    from paper_1407_4524_gb300 import lbm
    spec = dict(CASES[name], precision=prec)
    R = spec["bodies"][0]["R"]
    assert spec["n"][0] <= 2 * int(np.ceil(R)) + 13
    dom, ref = lbm.Domain(spec, device=0), oracle_mod.Oracle(spec)
    dom.step(60)
    ref.step(60)
    assert np.array_equal(dom.solid(), ref.solid())
    assert pop_error(dom.populations(), ref.fhat(), ref.solid()) <= tol
    if prec == "fp64":
        assert np.array_equal(dom.series(), ref.series())


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_stopped_body_leaves_no_list(prec):
    from paper_1407_4524_gb300 import lbm
    bodies = [dict(shape="cylinder", R=6.2, X0=(15.3, 20.1), U=(0.11, 0.05)),
              dict(shape="cylinder", R=5.0, X0=(50.0, 30.0), U=(-0.07, 0.0))]
    spec = dict(lattice="D2Q9", n=(70, 50), tau=0.7, precision=prec, bodies=bodies)
    dom = lbm.Domain(spec, device=0)
    dom.step(23)

    def state():
        bufs = _parse(dom.save_state(), 2, C.sizeof(lbm.lbm_body))[-1]
        return (np.frombuffer(bufs[FLAGS], np.uint8).reshape(dom.solid().shape) & 1,
                np.frombuffer(bufs[25], np.int64))  # solid flags, lengths of the covered / uncovered lists

    while not state()[1][0]:  # a step in which the first body covers or uncovers a node
        dom.step(1)
    t = dom.t
    at = dom.body_state()
    stopped = [dict(b, X0=tuple(at[k, :2]), U=(0.0, 0.0) if k == 0 else b["U"], t0=t) for k, b in enumerate(bodies)]
    dom.update_bodies(stopped)
    dom.step(1)
    flags, lengths = state()
    assert lengths[0] == 0
    owner = dom.solid()
    _, y, x = np.indices(owner.shape)
    near = np.hypot(x - at[0, 0], y - at[0, 1]) < 12.0  # (the other body still moves)
    assert np.array_equal(flags[near] != 0, owner[near] >= 0)
    dom.update_bodies([dict(b, X0=tuple(x[:2]), U=(0.0, 0.0), t0=dom.t) for b, x in zip(stopped, dom.body_state())])
    dom.step(1)
    flags, lengths = state()
    assert not lengths.any() and np.array_equal(flags != 0, dom.solid() >= 0)
    solid = dom.solid()
    dom.step(40)
    flags, lengths = state()
    assert not lengths.any() and np.array_equal(flags != 0, solid >= 0) and np.array_equal(dom.solid(), solid)
    assert np.isfinite(dom.series()).all()
