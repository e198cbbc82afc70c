"""The bounded wait of the one-kernel potential solve (needs a GB300).

A context's solves are told to give up at a grid barrier after one unsuccessful
poll, so the wait runs out by itself and the kernel returns; nothing faults or
hangs. On the 208 tiles of 402 x 123 some block polls before the last one has
arrived. Every call that delivers results reports FCD_ECUDA until a new state is
set, and the context then continues with the bits of one that never gave up."""
import ctypes as C

import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fcd():
    from paper_2410_11129_gb300 import fcd as F
    L = F.load()
    L.fcd_set_barrier_polls.argtypes = [C.c_void_p, C.c_uint]
    return F


def _cfg(prec, tol, **kw):
    return dict(W.small(nx=402, ny=123, r1=20.0, r2=40.0, xc=120.0, Bo_m=2.0, alpha_deg=20.0, mag_tol=tol,
                        mag_max_iter=300, **kw), precision=prec)


def _polls(fcd, ch, polls):
    assert fcd.load().fcd_set_barrier_polls(ch.h, polls) == fcd.FCD_OK


def _gives_up(fcd, call):
    with pytest.raises(fcd.FcdError) as e:
        call()
    assert e.value.status == fcd.FCD_ECUDA and "barrier" in str(e.value), str(e.value)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-6)])
def test_every_delivering_call_reports_it(fcd, prec, tol):
    ch, ref = fcd.Channel(_cfg(prec, tol)), fcd.Channel(_cfg(prec, tol))
    ch.step(2)
    snap = np.empty(ch.state_bytes(), np.uint8)
    ch.get_state(snap)
    pops = ch.populations()
    _polls(fcd, ch, 1)
    ch.step(2)  # asynchronous
    bad = np.empty_like(snap)
    for call in (ch.observe, lambda: ch.field("psi"), lambda: ch.field("phi1"), ch.populations,
                 lambda: ch.get_state(bad), ch.solve_magnetic, ch.observe):
        _gives_up(fcd, call)
    ref.step(4)
    want = ref.populations()
    for restore, exact in ((lambda: ch.set_state(snap), True),
                           (lambda: ch.set_populations(*pops, step=2), False)):  # no previous potential
        _polls(fcd, ch, 0)
        restore()
        ch.step(2)
        assert ch.observe()["step"] == 4
        got = ch.populations()
        if exact:
            assert all(np.array_equal(x, y) for x, y in zip(got, want))
        _polls(fcd, ch, 1)
        ch.step(1)
        _gives_up(fcd, ch.populations)
    ch.close()
    ref.close()


def test_host_driven_step(fcd, monkeypatch):
    monkeypatch.setenv("FCD_NO_GRAPH", "1")
    ch = fcd.Channel(_cfg("fp64", 1e-10))
    _polls(fcd, ch, 1)
    _gives_up(fcd, lambda: ch.step(1))
    ch.close()


def test_tangent_observation(fcd):
    t = fcd.Tangent(_cfg("fp64", 1e-10))
    t.step(1)
    t.tangent_observe()
    _polls(fcd, t, 1)
    t.step(1)
    _gives_up(fcd, t.tangent_observe)
    t.close()


def test_gradient(fcd):
    """The forward run is sound; the solves of the reverse sweep give up."""
    a = fcd.Adjoint(_cfg("fp64", 1e-10), 4)
    a.step(4)
    a.observe()
    _polls(fcd, a, 1)
    _gives_up(fcd, lambda: a.gradient(1.0, 0.0))
    a.close()


@pytest.mark.parametrize("mode", [0, 1])
def test_batch_instance(fcd, mode):
    """One instance of a batch gives up; the others deliver."""
    b = fcd.Batch([_cfg("fp32", 1e-6, Ca=0.1 + 0.02 * i) for i in range(3)])
    b.set_mode(mode)
    b.step(2)
    _polls(fcd, b.instances[1], 1)
    b.step(2)
    _gives_up(fcd, b.instances[1].populations)
    for i in (0, 2):
        assert b.instances[i].observe()["step"] == 4
    b.close()
