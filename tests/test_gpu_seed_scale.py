"""The reverse sweep is linear in its seed: a power-of-two seed scales every FP64
value it forms without a rounding, so the gradients of s J are s times those of
J, far outside the FP32 range of the potential solve's correction as well. The
tolerance of a solve is relative to its right-hand side, so the solves take the
same cycles. 1e-12 leaves room for the order of the reductions (needs a GB300)."""
import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(exponent, nx, ny):
    from paper_2410_11129_gb300 import fcd
    s = 2.0**exponent
    a = fcd.Adjoint(dict(W.small(nx=nx, ny=ny, xc=0.3 * nx, Bo_m=2.0, alpha_deg=20.0, mag_tol=1e-10,
                                 mag_max_iter=100), precision="fp64"), 4)
    a.step(6)
    o = a.gradient(s * 1.0, s * 0.01, initial=True)
    a.close()
    return np.array(o["grad"]) / s, o["df0"] / s, o["dg0"] / s, o["solve_cycles"]


@pytest.mark.parametrize("nx,ny", [(48, 20), (130, 33)])
@pytest.mark.parametrize("exponent", [-200, -100, 100, 200])
def test_gradient_is_linear_in_the_seed(exponent, nx, ny):
    ref, got = _run(0, nx, ny), _run(exponent, nx, ny)
    assert got[3] == ref[3]
    for x, y in zip(got[:3], ref[:3]):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(y).max()
