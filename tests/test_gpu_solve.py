"""The one-kernel potential solve at the edges of its tiling (needs a GB300):
32 x 8 lattice tiles, rows merged in pairs with three in the last cell of an odd
32 x 8 lattice tiles, rows merged in pairs with three in the last cell of an odd
block and (402 x 123, 800 x 100) across the grid."""
import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(4, 2), (6, 3), (34, 4), (32, 8), (34, 9), (66, 17), (100, 31), (402, 123), (800, 100)]


def _cfg(nx, ny, **kw):
    r2 = 0.3 * min(nx, ny) + 0.5
    return W.small(nx=nx, ny=ny, r1=0.5 * r2, r2=r2, xc=0.93 * nx, yc=0.45 * ny, xi=3.0, Bo_m=2.0,
                   alpha_deg=35.0, mag_max_iter=300, **kw)


def _residual(orc, cfg, ch):
    """max |L(psi0 + psi')| / H0 by the FP64 oracle, for the context's populations."""
    _, g, psi = ch.populations()
    k = orc.phase(cfg, g)[1]
    H0 = ch.derived()["H0"]
    return np.abs(orc.mag_apply(k, psi, 0.0, 0.0) - orc.mag_rhs(k, H0, cfg["alpha"])).max() / H0


@pytest.mark.parametrize("nx,ny", SIZES)
def test_fp64_solve_residual(orc, nx, ny):
    """The residual that ends the solve is the oracle's: below the tolerance, up
    to the rounding of nine terms of a potential of up to r2 H0 (1e-13 H0)."""
    from paper_2410_11129_gb300 import fcd
    cfg = _cfg(nx, ny, mag_tol=1e-11)
    ch = fcd.Channel(dict(cfg, precision="fp64"))
    ch.step(2)
    it, res, st = ch.solve_magnetic(1e-11, 300)
    assert st == fcd.FCD_OK and res <= 1e-11
    assert _residual(orc, cfg, ch) <= 1e-11 + 2e-13
    ch.close()


@pytest.mark.parametrize("nx,ny", SIZES)
def test_pair_solve_residual(orc, nx, ny):
    """The hi + lo pair to 1e-6: the FP32 permeability (6e-8 of k, eight links,
    gradients of up to a few H0) moves the oracle's residual by less than 1e-6."""
    from paper_2410_11129_gb300 import fcd
    cfg = _cfg(nx, ny, mag_tol=1e-6)
    ch = fcd.Channel(dict(cfg, precision="fp32"))
    ch.step(2)
    it, res, st = ch.solve_magnetic(1e-6, 300)
    assert st == fcd.FCD_OK and res <= 1e-6
    assert _residual(orc, cfg, ch) <= 2e-6
    ch.close()


def test_share_of_the_gpu_does_not_change_bits(orc):
    """An instance of a batch solves on fewer blocks than a lone context."""
    from paper_2410_11129_gb300 import fcd
    cfgs = [dict(_cfg(130, 33, mag_tol=1e-10), precision="fp64"), dict(_cfg(98, 41, mag_tol=1e-6), precision="fp32")]
    b = fcd.Batch(cfgs * 4)
    b.set_mode(0)
    b.step(3)
    for cfg, inst in zip(cfgs, b.instances):
        ch = fcd.Channel(cfg)
        ch.step(3)
        for x, y in zip(ch.populations(), inst.populations()):
            assert np.array_equal(x, y)
        ch.close()
    b.close()


@pytest.mark.parametrize("nx,ny,rows", [(130, 33, 2), (402, 123, 4)])
def test_fp64_collide_tile_rows(orc, nx, ny, rows):
    """Both tile heights of the FP64 collide-stream, ragged in both directions,
    against the oracle after two steps (solves at 1e-12: 1e-11 in the populations)."""
    from paper_2410_11129_gb300 import fcd
    cfg = _cfg(nx, ny, mag_tol=1e-12)
    ch = fcd.Channel(dict(cfg, precision="fp64"))
    assert ch.collide_tile_height() == rows
    ch.step(2)
    orc.set_threads(orc.max_threads())
    try:
        sim = orc.Sim(dict(cfg, mag_max_iter=100000))
        sim.step(2)
    finally:
        orc.set_threads(1)
    f, g, _ = ch.populations()
    assert np.abs(f - sim.f).max() <= 1e-11 and np.abs(g - sim.g).max() <= 1e-11
    ch.close()


OPENINGS = [(n, p) for n in [(6, 3), (34, 9), (64, 16), (66, 17), (130, 33), (402, 123)] for p in ("fp32", "fp32_offset")]


def _opening_pair(size, precision, max_iter):
    """Two contexts of the single-plane FP32 solve at one state: populations as
    initialised, the potential moved off its solution, for the last two steps."""
    from paper_2410_11129_gb300 import fcd
    cfg = dict(_cfg(*size, mag_tol=1e-4), mag_max_iter=max_iter, precision=precision)
    a, b = fcd.Channel(cfg), fcd.Channel(cfg)
    f, g, psi = a.populations()
    rng = np.random.default_rng(7)
    psi = (psi + 0.1 * a.derived()["H0"] * rng.standard_normal(psi.shape)).astype(np.float32).astype(np.float64)
    for ch in (a, b):
        ch.set_populations(f, g, psi)
    return a, b, psi


@pytest.mark.parametrize("size,precision", OPENINGS)
def test_opening_of_a_step(size, precision):
    """The kernel that opens a step against the phase recovery and the sweep of a
    solve on its own, one cycle each, at the edges of its 64 x 16 patches: the same
    sums in four dependent colours of about twenty roundings, 80 x 2^-24."""
    a, b, psi = _opening_pair(size, precision, 1)
    a.step(1)
    b.solve_magnetic(1e-30, 1)
    x, y = a.populations()[2], b.populations()[2]
    assert np.abs(x - psi).max() > 0
    assert np.abs(x - y).max() <= 80 * 2.0**-24 * (np.abs(psi).max() + a.derived()["H0"])
    a.close()
    b.close()


@pytest.mark.parametrize("size,precision", OPENINGS[2:6])
def test_potential_buffers_take_turns(size, precision):
    """Without cycles a step leaves exactly 2 psi'(t) - psi'(t-1), through every
    turn of the three buffers, and a snapshot continues with the same bits."""
    a, b, prev = _opening_pair(size, precision, 0)
    a.solve_magnetic(1e-30, 1)
    cur = a.populations()[2].astype(np.float32)
    prev = prev.astype(np.float32)
    assert not np.array_equal(cur, prev)
    buf = np.empty(a.state_bytes(), np.uint8)
    for _ in range(4):
        a.get_state(buf)
        b.set_state(buf)
        a.step(1)
        b.step(1)
        prev, cur = cur, np.float32(2) * cur - prev
        for ch in (a, b):
            assert np.array_equal(ch.populations()[2].astype(np.float32), cur)
    a.close()
    b.close()
