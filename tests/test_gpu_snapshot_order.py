"""Snapshots of contexts whose three psi' buffers take turns: every order of the
buffers, the fixed order of earlier files, and a context that keeps a fixed order
(needs a GB300)."""
import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu

HEADER, VERSION, CUR = 48, 4, 40  # bytes of the header, offsets of the version and of the two indices


def _cfg(tol, precision="fp32"):
    return dict(W.small(nx=98, ny=35, r1=5.0, r2=10.0, xc=40.0, Bo_m=3.0, alpha_deg=30.0, mag_tol=tol), precision=precision)


def _ints(snap, at, n):
    return snap[at:at + 4 * n].view(np.int32)


def _planes(snap, ch):
    """The three stored buffers, in the order of the file."""
    ps = (ch.nx + 31) // 32 * 32 * ch.ny
    return [snap[HEADER + 4 * ps * (27 + 2 * q):HEADER + 4 * ps * (29 + 2 * q)] for q in range(3)]


def _fixed(snap, ch, cur):
    """The same state as a version-4 file whose buffer `cur` (0 or 1) is the current one."""
    now, prev = _ints(snap, CUR, 2)[0], 2 - _ints(snap, CUR, 2)[1]
    src, out = _planes(snap.copy(), ch), snap.copy()
    dst = _planes(out, ch)
    dst[cur][:], dst[1 - cur][:], dst[2][:] = src[now], src[3 - now - prev], src[prev]
    _ints(out, VERSION, 1)[0] = 4
    _ints(out, CUR, 2)[:] = (cur, 0)
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp32_offset"])
def test_every_order_and_earlier_files(precision):
    from paper_2410_11129_gb300 import fcd
    a, b, ref = (fcd.Channel(_cfg(1e-4, precision)) for _ in range(3))
    pair = fcd.Channel(_cfg(1e-6, precision))
    seen = set()
    for n in range(1, 9):
        a.step(1)
        snap = np.empty(a.state_bytes(), np.uint8)
        a.get_state(snap)
        assert _ints(snap, VERSION, 1)[0] == 5
        seen.add(tuple(_ints(snap, CUR, 2)))
        ref.step(1)
        psi = ref.field("psi")
        for file in (snap, _fixed(snap, a, 0), _fixed(snap, a, 1)):
            b.set_state(file)
            assert np.array_equal(b.field("psi"), psi)
            again = np.empty_like(snap)
            b.get_state(again)
            if file is snap:
                assert np.array_equal(again, snap)
            b.step(3)
            c = [x.copy() for x in b.populations()]
            if file is snap:
                first = c
            assert all(np.array_equal(x, y) for x, y in zip(c, first))
        pair.set_state(snap)  # fixed order, the low planes 0
        assert np.array_equal(pair.field("psi"), psi)
        pair.get_state(again)
        assert _ints(again, VERSION, 1)[0] == 4 and _ints(again, CUR, 1)[0] in (0, 1) and _ints(again, CUR, 2)[1] == 0
        assert np.array_equal(_fixed(again, a, 0), _fixed(snap, a, 0))
        pair.step(1)
        assert pair.observe(allow=(fcd.FCD_ENOCONV,))["step"] == n + 1
    ref.step(3)
    assert all(np.array_equal(x, y) for x, y in zip(ref.populations(), first))
    assert len(seen) >= 3, seen  # the buffers did take turns
    for bad in ((3, 0), (-1, 0), (0, 3), (2, 0), (1, 1), (0, 2)):
        file = snap.copy()
        _ints(file, CUR, 2)[:] = bad
        with pytest.raises(fcd.FcdError) as e:
            b.set_state(file)
        assert e.value.status == fcd.FCD_ESTATE
    for ch in (a, b, ref, pair):
        ch.close()
