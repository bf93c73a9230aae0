"""Snapshots that an earlier version of the library wrote: body records without
the served solves' part, other geometry chunks, link tiles of another size and,
in FP64 mode, moments kept within two links of a body only and solid flags
already moved on.  A snapshot of today is turned into one of those (what that
version did not hold is overwritten with rubbish); the domain that loads it
continues with the same bits."""
import ctypes as C
import struct

import numpy as np
import pytest

from test_parity_gpu import CASES_2D, CASES_3D

pytestmark = pytest.mark.gpu

HEADER = "<8s6iq2iq"
RECORD_TAIL = 64  # bytes of a body record that earlier versions do not have
NCHUNKS_AT = 12   # BodyDev::nchunks
FLAGS, COUNTERS, BODIES, DERIVED, TILE_PRE = 6, 7, 8, (10, 11, 12, 13), 30
MAC = {0: 1, 1: 4}  # moments of even / odd steps

CASES = {
    "moving_cylinders": dict(CASES_2D["moving_cylinders_periodic"]),
    "moving_spheres": dict(CASES_3D["moving_spheres_periodic"]),
    "static_sphere": dict(lattice="D3Q19", n=(60, 40, 36), tau=0.6, u0=(0.03, 0.0, 0.01),
                          bodies=[dict(shape="sphere", R=9.3, X0=(20.2, 19.6, 18.4))]),
}


def _parse(blob, nb, body_bytes):
    head = struct.unpack_from(HEADER, blob, 0)
    nbuf = head[-1]
    # the record size is the one that the buffer list fits
    for rec in range(64, 1024, 8):
        at = struct.calcsize(HEADER) + nb * (body_bytes + rec)
        if at + 8 * nbuf > len(blob):
            continue
        sizes = struct.unpack_from("<%dq" % nbuf, blob, at)
        if all(n >= 0 for n in sizes) and at + 8 * nbuf + sum(sizes) == len(blob) and sizes[BODIES] == nb * rec:
            break
    else:
        raise AssertionError("no record size fits")
    at += 8 * nbuf
    bufs = []
    for n in sizes:
        bufs.append(blob[at:at + n])
        at += n
    host = blob[struct.calcsize(HEADER):struct.calcsize(HEADER) + nb * body_bytes]
    records = blob[struct.calcsize(HEADER) + nb * body_bytes:][:nb * rec]
    return head, rec, host, records, bufs


def _hops(solid, c):
    one = np.zeros(solid.shape, bool)
    two = np.zeros(solid.shape, bool)
    for v in c[1:]:
        one |= np.roll(solid, (v[2], v[1], v[0]), (0, 1, 2))
        two |= np.roll(solid, (2 * v[2], 2 * v[1], 2 * v[0]), (0, 1, 2))
    return one, two


def _as_earlier_version(dom, spec, blob):
    from paper_1407_4524_gb300 import lbm
    nb = len(spec["bodies"])
    head, rec, host, records, bufs = _parse(blob, nb, C.sizeof(lbm.lbm_body))

    def shorten(data):
        out = bytearray()
        for k in range(nb):
            r = bytearray(data[k * rec:(k + 1) * rec - RECORD_TAIL])
            r[NCHUNKS_AT:NCHUNKS_AT + 4] = struct.pack("<i", 1)
            out += r
        return bytes(out)

    bufs[BODIES] = shorten(bufs[BODIES])
    for k in DERIVED:
        bufs[k] = b"\xff" * (8 * nb)
    bufs[TILE_PRE] = b"\0" * len(bufs[TILE_PRE])
    if spec["precision"] == "fp64":
        c = np.zeros((dom.q, 3), int)
        t = lbm.lbm_lattice_table(dom.q)[0]
        c[:, :t.shape[1]] = t
        solid = dom.solid() >= 0
        one, two = _hops(solid, c)
        near = (one | two) & ~solid
        flags = np.where(solid, 1, np.where(near, 2, 0) | np.where(one, 4, 0)).astype(np.uint8)
        bufs[FLAGS] = flags.tobytes()
        mac = np.frombuffer(bufs[MAC[dom.t & 1]], dtype=np.float64).copy().reshape(-1, 4)
        mac[~near.ravel()] = np.nan
        bufs[MAC[dom.t & 1]] = mac.tobytes()
    out = struct.pack(HEADER, *head) + host + shorten(records)
    out += struct.pack("<%dq" % len(bufs), *[len(b) for b in bufs])
    return out + b"".join(bufs)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_loads_and_continues(name, prec):
    from paper_1407_4524_gb300 import lbm
    spec = dict(CASES[name], precision=prec)
    a = lbm.Domain(spec, device=0)
    a.step(17)
    blob = a.save_state()
    old = _as_earlier_version(a, spec, blob)
    assert len(old) != len(blob)
    a.step(39)
    b = lbm.Domain(spec, device=0)
    b.load_state(old)
    assert b.t == 17
    b.step(39)
    fluid = a.solid() < 0
    assert np.array_equal(a.solid(), b.solid())
    assert np.array_equal(a.populations()[:, fluid], b.populations()[:, fluid])
    assert np.array_equal(a.series(), b.series())
    again = lbm.Domain(spec, device=0)  # and what it writes is a snapshot of today
    again.load_state(b.save_state())
    assert np.array_equal(again.populations()[:, fluid], b.populations()[:, fluid])


def test_what_does_not_fit_is_refused_and_changes_nothing():
    from paper_1407_4524_gb300 import lbm
    spec = dict(CASES["moving_cylinders"], precision="fp32")
    a = lbm.Domain(spec, device=0)
    a.step(6)
    blob = a.save_state()
    want = a.populations()
    old = _as_earlier_version(a, spec, blob)
    for bad in (blob[:-1], blob + b"\0", old[:-8], old[:200], blob[:56]):
        with pytest.raises(lbm.LbmError, match="LBM_ERR_ARG"):
            a.load_state(bad)
    assert a.t == 6 and np.array_equal(a.populations(), want)
