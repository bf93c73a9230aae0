"""What a served solve is charged against a batch's budget never grows from one
version of the library to the next: a request that fitted a budget still fits.
The figures are those of the first version with this interface."""
import ctypes as C

import pytest

CHANNEL = {"x": ("inlet", "outlet"), "y": ("wall", "wall")}
SOLVES = [
    (415797, dict(lattice="D2Q9", n=(131, 67), precision="fp16", steps=300, edges=CHANNEL, inlet={"u": 0.04},
                  bodies=[dict(shape="cylinder", R=7.3, X0=(33.1, 30.2))])),
    (270562, dict(lattice="D2Q9", n=(64, 48), precision="fp32", steps=64,
                  bodies=[dict(shape="cylinder", R=2.0, X0=(20.0, 20.0)),
                          dict(shape="ellipse", R=6.0, R2=3.0, theta0=0.3, X0=(45.0, 22.0))])),
    (33018032, dict(lattice="D2Q9", n=(700, 600), precision="fp32", steps=64,
                    bodies=[dict(shape="cylinder", R=120.0, X0=(300.0, 300.0))])),
    (4106738, dict(lattice="D3Q19", n=(40, 36, 33), precision="fp16", steps=95,
                   bodies=[dict(shape="sphere", R=5.5, X0=(20.0, 18.3, 16.1)),
                           dict(shape="sphere", R=1.2, X0=(6.0, 5.0, 5.0))])),
    (148301284, dict(lattice="D3Q19", n=(192, 96, 96), precision="fp16", steps=2000,
                     bodies=[dict(shape="sphere", R=30.5, X0=(60.0, 48.0, 48.0))])),
    (9806170, dict(lattice="D3Q19", n=(64, 40, 24), precision="fp32", steps=10,
                   bodies=[dict(shape="cylinder", R=5.0, X0=(20.0, 20.0))])),
    (178636, dict(lattice="D2Q9", n=(64, 64), precision="fp16", steps=64)),
]


@pytest.mark.parametrize("first,spec", SOLVES)
def test_a_solve_is_charged_no_more_than_before(first, spec):
    from paper_1407_4524_gb300 import lbm
    spec = dict(spec, tau=0.7)
    d, _, _ = lbm.domain_desc(spec, 0)
    bodies = spec.get("bodies", [])
    out = C.c_int64()
    lbm._check(lbm.load().lbm_batch_solve_bytes(C.byref(d), lbm.body_array(bodies), len(bodies), spec["steps"],
                                                C.byref(out)))
    cells = 1
    for v in spec["n"]:
        cells *= v
    q, size = (9 if spec["lattice"] == "D2Q9" else 19), (2 if spec["precision"] == "fp16" else 4)
    assert 2 * cells * q * size < out.value <= first
