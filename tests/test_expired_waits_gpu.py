"""A bounded wait that runs out leaves nodes unstepped: every read of results
says so, with bodies and without, until a good snapshot is loaded.  The waits
are made to run out by a hook that leaves the bulk copies away."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

IN_OUT = {"x": ("inlet", "outlet")}
SPHERE = dict(shape="sphere", R=5.4, X0=(40.2, 23.6, 13.9))
CASES = {
    "bulk_tiles_no_body": (None, dict(lattice="D3Q19", n=(192, 24, 124), tau=0.56, precision="fp16", edges=IN_OUT,
                                      inlet={"u": 0.04}, u0=(0.04, 0.0, 0.0))),
    "bulk_tiles_body": (None, dict(lattice="D3Q19", n=(192, 24, 124), tau=0.56, precision="fp16", edges=IN_OUT,
                                   inlet={"u": 0.04}, u0=(0.04, 0.0, 0.0), bodies=[SPHERE])),
    "staged_no_body": ("1", dict(lattice="D2Q9", n=(64, 24), tau=0.7, precision="fp32", u0=(0.02, 0.0))),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_every_read_reports_it(name, monkeypatch):
    from paper_1407_4524_gb300 import lbm
    staged, spec = CASES[name]
    if staged:
        monkeypatch.setenv("LBM_STAGED", staged)
    good = lbm.Domain(spec, device=0)
    good.step(2)
    blob, want = good.save_state(), good.macros()
    good.close()
    monkeypatch.setenv("LBM_STAGED_TEST_EXPIRE", "1")
    dom = lbm.Domain(spec, device=0)
    dom.step(1)

    def raw_series():
        out = np.zeros((1, max(len(dom.bodies), 1), lbm.SERIES_ROW))
        lbm._check(dom.lib.lbm_get_series(dom.h, 0, 1, out.ctypes.data))

    def no_alloc():
        out = np.empty(dom.q * dom.N)
        lbm._check(dom.lib.lbm_get_populations_noalloc(dom.h, out.ctypes.data))

    reads = [raw_series, dom.macros, dom.populations, dom.save_state, dom.solid]
    if dom.bodies:
        reads += [dom.series, dom.force_torque, dom.body_state]
    if dom.q * dom.N <= 4194304:
        reads.append(no_alloc)
    for read in reads:
        with pytest.raises(lbm.LbmError, match="LBM_ERR_TIMEOUT"):
            read()
    assert dom.stats()["timeouts"] != 0
    dom.load_state(blob)
    assert dom.stats()["timeouts"] == 0
    assert np.array_equal(dom.macros(), want)
    dom.close()


def test_reads_without_a_step():
    """no step yet, no rows asked for: nothing to report"""
    from paper_1407_4524_gb300 import lbm
    dom = lbm.Domain(CASES["staged_no_body"][1], device=0)
    out = (C.c_double * 1)()
    assert dom.lib.lbm_get_series(dom.h, 0, 0, out) == 0
    dom.step(3)
    assert dom.lib.lbm_get_series(dom.h, 0, 3, out) == 0  # no bodies: no rows
    dom.close()
