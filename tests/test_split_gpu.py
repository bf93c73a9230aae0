"""Steps whose stream-collide pass is divided into the planes that no cut link
touches and the others (static bodies in 3-D), against the undivided pass that
kernel timing takes: the same bits, for runs of planes that wrap and that end
at walls, several bodies, a body across the z seam, plain steps and graphs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SPH = dict(shape="sphere")
CASES = {
    "channel": dict(n=(96, 40, 64), tau=0.6, edges={"x": ("inlet", "outlet")}, inlet={"u": 0.04}, u0=(0.04, 0.0, 0.0),
                    bodies=[dict(SPH, R=6.3, X0=(30.2, 18.7, 30.4))]),
    "across_the_seam": dict(n=(63, 50, 66), tau=0.7, u0=(0.02, 0.01, -0.02),
                            bodies=[dict(SPH, R=5.1, X0=(30.1, 24.6, 0.3)), dict(SPH, R=7.0, X0=(20.0, 20.0, 52.0))]),
    "walls": dict(n=(70, 48, 60), tau=0.65, eq="standard", edges={"y": ("wall", "wall"), "z": ("wall", "wall")},
                  u0=(0.03, 0.0, 0.0), bodies=[dict(SPH, R=6.0, X0=(30.5, 22.1, 41.9))]),
    "forced": dict(n=(64, 48, 48), tau=0.8, force=(1e-5, 0.0, 0.0), edges={"y": ("wall", "wall")},
                   bodies=[dict(SPH, R=5.5, X0=(31.0, 23.0, 11.0))]),
}


def _run(spec, timed):
    from paper_1407_4524_gb300 import lbm
    dom = lbm.Domain(spec, device=0)
    dom.set_kernel_timing(timed)
    dom.step(3)
    dom.step(35)
    out = dict(f=dom.populations()[:, dom.solid() < 0], series=dom.series(), mac=dom.macros())
    dom.close()
    return out


@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_divided_pass_same_bits(name, prec):
    spec = dict(CASES[name], lattice="D3Q19", precision=prec)
    a, b = _run(spec, False), _run(spec, True)
    for k in a:
        assert np.array_equal(a[k], b[k]), k
