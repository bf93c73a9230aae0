"""Served solves large enough for the stream-collide kernel on bulk-copied
tiles: its pass leaves the boundary nodes to the kernel beside it, so the two
store single halves of the same words.  The force/torque series is the same
alone, in a mix, on the single-node kernel (LBM_PAIR=0) and on the batched one
(LBM_BATCH_GROUPED=1), bit for bit; and a wait that runs out is reported."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

IN_OUT = {"x": ("inlet", "outlet")}
LARGE = {
    "channel": dict(  # tiles of 5 rows of 192, a last one of 4
        lattice="D3Q19", n=(192, 24, 124), tau=0.56, precision="fp16", edges=IN_OUT, inlet={"u": 0.04},
        u0=(0.04, 0.0, 0.0), steps=56,
        bodies=[dict(shape="sphere", R=5.4, X0=(40.2, 23.6, 13.9)), dict(shape="sphere", R=4.3, X0=(41.0, 11.0, 70.6))]),
    "periodic": dict(
        lattice="D3Q19", n=(256, 25, 180), tau=0.6, precision="fp16", u0=(0.01, -0.005, 0.002), steps=40,
        bodies=[dict(shape="sphere", R=5.2, X0=(1.4, 10.6, 17.3)), dict(shape="sphere", R=4.1, X0=(120.2, 19.7, 40.9))]),
}
BESIDE = [
    dict(lattice="D2Q9", n=(131, 67), tau=0.62, precision="fp16", edges={"x": ("inlet", "outlet"), "y": ("wall", "wall")},
         inlet={"profile": "parabolic", "u": 0.04}, steps=90, bodies=[dict(shape="cylinder", R=7.3, X0=(33.1, 30.2))]),
    dict(lattice="D3Q19", n=(64, 48, 40), tau=0.7, precision="fp16", edges=IN_OUT, inlet={"u": 0.03}, steps=70,
         u0=(0.03, 0.0, 0.0), bodies=[dict(shape="sphere", R=6.2, X0=(16.4, 23.1, 19.7))]),
]


def _serve(specs, ticks=8):
    """series of every spec, all admitted together"""
    from paper_1407_4524_gb300 import lbm
    batch = lbm.Batch(8 << 30, max_slots=len(specs), ticks_per_launch=ticks)
    slots = [batch.admit(s) for s in specs]
    assert None not in slots
    done = set()
    for _ in range(100):
        batch.run(1)
        done.update(batch.poll())
        if len(done) == len(slots):
            break
    out = [{k: batch.force_torque(s, k) for k in ("static", "moving")} for s in slots]
    batch.close()
    return out


@pytest.mark.parametrize("name", sorted(LARGE))
def test_same_bits_however_it_is_served(name, monkeypatch):
    spec = LARGE[name]
    alone = _serve([spec])[0]
    assert alone["static"].shape == (spec["steps"], 2, 6) and np.isfinite(alone["static"]).all()
    runs = {"mix": _serve([BESIDE[0], spec, BESIDE[1], LARGE["channel"]])[1],
            "odd ticks (batched kernel)": _serve([spec], ticks=7)[0]}
    monkeypatch.setenv("LBM_PAIR", "0")
    runs["single-node kernel"] = _serve([spec])[0]
    monkeypatch.delenv("LBM_PAIR")
    monkeypatch.setenv("LBM_BATCH_GROUPED", "1")
    runs["batched kernel"] = _serve([spec])[0]
    for how, got in runs.items():
        for k in alone:
            assert np.array_equal(got[k], alone[k]), (how, k)


@pytest.mark.parametrize("name", sorted(LARGE))
def test_expired_wait_is_reported_for_its_solve_only(name, monkeypatch):
    """(also: these solves do take the kernel on bulk-copied tiles)"""
    from paper_1407_4524_gb300 import lbm
    batch = lbm.Batch(8 << 30, max_slots=2, ticks_per_launch=2)
    small = batch.admit(dict(BESIDE[1], steps=2))
    monkeypatch.setenv("LBM_STAGED_TEST_EXPIRE", "1")
    large = batch.admit(dict(LARGE[name], steps=2))
    batch.run(1)
    assert sorted(batch.poll()) == sorted([small, large])
    with pytest.raises(lbm.LbmError, match="LBM_ERR_TIMEOUT"):
        batch.force_torque(large)
    assert np.isfinite(batch.force_torque(small)).all()
    batch.close()
