"""Observables at the edges of their clusters (needs a GB300): 32 columns a cluster
of ceil(ny / 16) blocks, at most 8 (from 113 rows on), of 8 warps, each a run of
ceil(ny / (8 blocks)) rows; the last runs of a column are short or empty where
that does not divide. 256 or 512 threads over the columns at the end.

Against the FP64 oracle on the same populations: sums of at most 7e4 FP64 terms in
another order agree to 7e4 x 1.1e-16 < 1e-11 of their size; extents and centroids
are quotients of such values."""
import ctypes as C

import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("T_o", "T_i", "lx_o", "ly_o", "lx_i", "ly_i", "xc_core", "yc_core", "xc_shell", "yc_shell")


@pytest.mark.parametrize("open_x", [0, 1])
@pytest.mark.parametrize("nx,ny,yc", [(34, 16, 8.0), (34, 17, 8.0), (34, 112, 100.0), (66, 113, 56.0), (34, 127, 3.0),
                                      (34, 128, 64.0), (34, 129, 126.0), (30, 200, 190.0), (34, 577, 300.0),
                                      (254, 24, 12.0), (256, 24, 12.0), (258, 24, 12.0), (510, 20, 9.0),
                                      (512, 20, 9.0), (514, 20, 9.0)])
def test_observables_at_cluster_edges(orc, nx, ny, yc, open_x):
    import torch
    from paper_2410_11129_gb300 import fcd
    r2 = 0.35 * min(nx, ny) + 0.4
    cfg = W.small(nx=nx, ny=ny, r1=0.9 * r2, r2=r2, xc=0.9 * nx, yc=yc, xi=3.0, Bo_m=0.0, open_x=open_x)
    sim = orc.Sim(cfg)
    ref = sim.observe()
    g = torch.from_numpy(sim.g).to("cuda")
    out = fcd.fcd_obs()
    st = fcd.load().fcd_observe_populations_noalloc(C.c_void_p(g.data_ptr()), nx, ny, open_x,
                                                    C.c_void_p(torch.cuda.current_stream().cuda_stream),
                                                    C.byref(out))
    assert st == fcd.FCD_OK
    got = out.as_dict()
    for k in KEYS:
        assert abs(got[k] - ref[k]) <= 1e-11 * max(1.0, abs(ref[k])), (k, got[k], ref[k])
    for i in range(3):
        assert abs(got["mass"][i] - ref["mass"][i]) <= 1e-11 * nx * ny
    assert got["breakup"] == ref["breakup"]
    if ref["breakup"]:
        assert (got["xb"], got["yb"]) == (ref["xb"], ref["yb"])


@pytest.mark.parametrize("nx,ny", [(34, 113), (30, 129), (34, 200), (514, 24)])
def test_tangent_observables_at_cluster_edges(nx, ny):
    """The derivative form's values are the plain observables', and its derivatives
    the adjoint seed's, to the 1e-9 of the existing comparison of the two forms."""
    from paper_2410_11129_gb300 import fcd
    cfg = dict(W.small(nx=nx, ny=ny, r1=4.0, r2=8.0, xc=0.95 * nx, xi=4.0, Bo_m=2.0, alpha_deg=20.0,
                       mag_tol=1e-13, mag_max_iter=300), precision="fp64")
    t, a = fcd.Tangent(cfg), fcd.Adjoint(cfg, 2)
    t.step(2)
    a.step(2)
    o, p = t.tangent_observe(), t.observe()
    for k in ("T_o", "lx_o", "ly_o"):
        assert abs(o[k] - p[k]) <= 1e-11 * max(1.0, abs(p[k])), k
    for wT, wO, key in ((1.0, 0.0, "dT_o"), (0.0, 1.0, "doverlap")):
        g = np.array(a.gradient(wT, wO)["grad"])
        d = np.array(o[key])
        assert np.abs(g - d).max() <= 1e-9 * np.abs(d).max(), (key, g, d)
    t.close()
    a.close()
