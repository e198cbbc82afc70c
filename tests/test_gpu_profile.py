"""Stage times of a step whose solve does not end at its first residual: the
further cycles belong to the solve, not to the collide-stream (needs a GB300)."""
import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,open_x", [("fp32", 0), ("fp32_offset", 1)])
def test_further_cycles_are_booked_as_solve(precision, open_x):
    """psi' far from the solution takes five residuals or more, each behind a
    cycle of at least four dependent kernels; the collide-stream is one, or two
    with open ends. So the solve takes more than twice as long, and the collide
    no more than twice what it takes in the next steps."""
    from paper_2410_11129_gb300 import fcd
    cfg = dict(W.small(nx=402, ny=123, r1=20.0, r2=40.0, xc=120.0, Bo_m=2.0, mag_tol=1e-4, open_x=open_x),
               precision=precision)
    ch, plain = fcd.Channel(cfg), fcd.Channel(cfg)
    ch.set_profiling(True)
    for c in (ch, plain):  # graphs of both parities
        c.step(1)
        c.step(1)
    ch.step(8)
    plain.step(8)
    usual = ch.last_step_profile()
    f, g, psi = ch.populations()
    psi = psi + ch.derived()["H0"] * np.random.default_rng(1).standard_normal(psi.shape)
    ch.set_populations(f, g, psi)
    plain.set_populations(f, g, psi)
    before = ch.solver_stats()["heads"]
    ch.step(1)
    p = ch.last_step_profile()
    assert ch.solver_stats()["heads"] - before >= 5
    assert p["solve"] > 2 * p["collide"], p
    assert p["collide"] < 2 * usual["collide"], (p, usual)
    assert abs(p["phase"] + p["solve"] + p["collide"] - p["step"]) <= 1e-3 * p["step"]
    plain.step(1)  # profiling changes no bit
    for x, y in zip(ch.populations(), plain.populations()):
        assert np.array_equal(x, y)
    ch.close()
    plain.close()
