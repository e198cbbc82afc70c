"""Exchange with device memory (written and read by the kernels directly) against
exchange with host memory (through a staging block): the same bits, any of the
pointers missing (needs a GB300). 38 x 13 and 64 x 33 leave ragged 32 x 32 tiles."""
import ctypes as C

import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4), ("fp32_offset", 1e-6)])
@pytest.mark.parametrize("nx,ny", [(38, 13), (64, 33)])
def test_device_exchange_is_host_exchange(prec, tol, nx, ny):
    import torch
    from paper_2410_11129_gb300 import fcd
    L = fcd.load()
    cfg = dict(W.small(nx=nx, ny=ny, r1=2.0, r2=4.0, xc=14.0, xi=3.0, Bo_m=2.0, mag_tol=tol), precision=prec)
    a, b = fcd.Channel(cfg), fcd.Channel(cfg)
    a.step(5)
    host = a.populations()
    ptr = lambda t: C.c_void_p(t.data_ptr()) if t is not None else None
    for keep in ((1, 1, 1), (1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1)):
        dev = [torch.full(h.shape, -7.0, dtype=torch.float64, device="cuda") if k else None
               for h, k in zip(host, keep)]
        assert L.fcd_get_populations(a.h, *[ptr(t) for t in dev]) == fcd.FCD_OK
        for h, t in zip(host, dev):
            assert t is None or np.array_equal(t.cpu().numpy(), h)
    for name in ("phi1", "phi3", "ux", "psi"):
        t = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
        assert np.array_equal(a.field(name, out=t).cpu().numpy(), a.field(name))
    dev = [torch.from_numpy(h).to("cuda") for h in host]
    assert L.fcd_set_populations(b.h, *[ptr(t) for t in dev], 5) == fcd.FCD_OK
    c = fcd.Channel(cfg)
    c.set_populations(*host, step=5)
    for x, y in zip(b.populations(), c.populations()):
        assert np.array_equal(x, y)
    b.step(3)
    c.step(3)
    for x, y in zip(b.populations(), c.populations()):
        assert np.array_equal(x, y)
    for ch in (a, b, c):
        ch.close()
