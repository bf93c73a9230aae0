"""The stream-collide kernel that brings tiles of whole rows to shared memory
by bulk copies (D3Q19, FP16 storage), against the single-node kernel
(LBM_PAIR=0): the same populations, force/torque series and moments bit for
bit, at sizes just above the number of tiles from which the kernel is used; and
its bounded waits, made to run out by a hook that leaves the copies away."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

IN_OUT = {"x": ("inlet", "outlet")}
CASES = {
    "periodic_partial_tile": dict(  # tiles of 4 rows, the last of a plane of one
        lattice="D3Q19", n=(256, 25, 180), tau=0.6, u0=(0.01, -0.005, 0.002),
        bodies=[dict(shape="sphere", R=5.2, X0=(1.4, 10.6, 17.3), U=(0.02, 0.0, -0.01), W=(0.0, 0.002, 0.0)),
                dict(shape="sphere", R=4.1, X0=(120.2, 19.7, 40.9))]),
    "periodic_row_per_tile": dict(  # the longest rows
        lattice="D3Q19", n=(1024, 16, 80), tau=0.7, eq="standard", u0=(0.02, 0.0, 0.0),
        bodies=[dict(shape="sphere", R=3.2, X0=(1022.9, 0.4, 12.2))]),
    "periodic_plane_per_tile": dict(  # both y seams in every tile; idle lanes past the rows
        lattice="D3Q19", n=(72, 12, 1220), tau=0.8, u0=(0.0, 0.01, 0.02),
        bodies=[dict(shape="sphere", R=2.6, X0=(40.1, 11.4, 600.3))]),
    "channel": dict(  # tiles of 5 rows of 192: lanes past them, a last tile of 4
        lattice="D3Q19", n=(192, 24, 124), tau=0.56, edges=IN_OUT, inlet={"u": 0.04}, u0=(0.04, 0.0, 0.0),
        bodies=[dict(shape="sphere", R=5.4, X0=(40.2, 23.6, 13.9))]),
    "channel_rotating": dict(  # parabolic inlet; a moving body: the kernel that leaves registers free
        lattice="D3Q19", n=(136, 30, 160), tau=0.65, rho0=1.1, edges=IN_OUT, u0=(0.01, 0.0, 0.0),
        inlet={"profile": "parabolic", "u": 0.02},
        bodies=[dict(shape="sphere", R=5.1, X0=(60.3, 12.2, 41.5), W=(0.001, 0.0, 0.002))]),
    "wall_outlet_short_rows": dict(
        lattice="D3Q19", n=(16, 70, 330), tau=0.7, edges={"x": ("wall", "outlet")}, u0=(0.0, 0.01, 0.02),
        bodies=[dict(shape="sphere", R=2.9, X0=(7.8, 33.1, 101.4))]),
}


def _run(spec, pair, monkeypatch):
    from paper_1407_4524_gb300 import lbm
    monkeypatch.setenv("LBM_PAIR", pair)
    dom = lbm.Domain(spec, device=0)
    dom.step(12)
    out = dict(f=dom.populations(), series=dom.series(), mac=dom.macros(), solid=dom.solid())
    dom.close()
    return out


@pytest.mark.parametrize("name", sorted(CASES))
def test_same_bits_as_single_node_kernel(name, monkeypatch):
    spec = dict(CASES[name], precision="fp16")
    a, b = _run(spec, "1", monkeypatch), _run(spec, "0", monkeypatch)
    fluid = a["solid"] < 0
    assert np.array_equal(a["f"][:, fluid], b["f"][:, fluid])
    for k in ("series", "mac", "solid"):
        assert np.array_equal(a[k], b[k]), k


def test_expired_waits_return_a_status(monkeypatch):
    from paper_1407_4524_gb300 import lbm
    spec = dict(CASES["channel"], precision="fp16")
    monkeypatch.setenv("LBM_STAGED_TEST_EXPIRE", "1")
    dom = lbm.Domain(spec, device=0)
    dom.step(1)
    with pytest.raises(lbm.LbmError, match="LBM_ERR_TIMEOUT"):
        dom.series()
    dom.close()
    monkeypatch.delenv("LBM_STAGED_TEST_EXPIRE")
    dom = lbm.Domain(spec, device=0)
    dom.step(4)
    assert np.isfinite(dom.series()).all()
