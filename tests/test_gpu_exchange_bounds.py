"""Device buffers of the exchange that end too early are refused on the host,
before any kernel is launched, and nothing is written; a buffer that ends exactly
with its values is taken (needs a GB300)."""
import ctypes as C

import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture
def alloc():
    """cudaMalloc blocks of exact sizes whose end no other allocation follows."""
    import torch
    torch.cuda.init()
    rt = C.CDLL("libcudart.so")
    drv = C.CDLL("libcuda.so.1")
    blocks = []

    def make(doubles, alone=True):
        for _ in range(8):
            p = C.c_void_p()
            assert rt.cudaMalloc(C.byref(p), C.c_size_t(8 * doubles)) == 0
            blocks.append(p)
            base, size = C.c_uint64(), C.c_size_t()
            assert drv.cuMemGetAddressRange_v2(C.byref(base), C.byref(size), C.c_uint64(p.value)) == 0
            after = C.c_uint64(base.value + size.value)
            if not alone or drv.cuMemGetAddressRange_v2(C.byref(base), C.byref(size), after) != 0:
                return p.value
        pytest.skip("an allocation follows every block")

    yield make
    for p in blocks:
        rt.cudaFree(p)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_short_device_buffers_are_refused(alloc, precision, tol):
    import torch
    from paper_2410_11129_gb300 import fcd
    L = fcd.load()
    cfg = dict(W.small(nx=130, ny=33, mag_tol=tol), precision=precision)
    ch = fcd.Channel(cfg)
    ch.step(2)
    N = ch.nx * ch.ny
    want = ch.populations()
    ok = torch.full((28 * N,), -7.0, dtype=torch.float64, device="cuda")
    at = lambda n: C.c_void_p(ok.data_ptr() + 8 * n)
    short = {k: C.c_void_p(alloc(n * N // 2)) for k, n in (("f", 9), ("g", 18), ("psi", 1))}
    torch.cuda.synchronize()
    for i, k in enumerate(("f", "g", "psi")):
        bufs = [at(0), at(9 * N), at(27 * N)]
        bufs[i] = short[k]
        for st in (L.fcd_get_populations(ch.h, *bufs), L.fcd_set_populations(ch.h, *bufs, 2)):
            assert st == fcd.FCD_ECUDA
        assert b"buffer" in L.fcd_last_error(ch.h)
    assert L.fcd_get_field(ch.h, fcd.FIELDS["psi"], short["psi"], N) == fcd.FCD_ECUDA
    assert (ok == -7.0).all()
    for x, y in zip(ch.populations(), want):  # nothing was imported
        assert np.array_equal(x, y)
    whole = C.c_void_p(alloc(28 * N, alone=False))
    at = lambda n: C.c_void_p(whole.value + 8 * n)
    assert L.fcd_get_populations(ch.h, at(0), at(9 * N), at(27 * N)) == fcd.FCD_OK
    assert L.fcd_set_populations(ch.h, at(0), at(9 * N), at(27 * N), 2) == fcd.FCD_OK
    for x, y in zip(ch.populations(), want):
        assert np.array_equal(x, y)
    ch.close()


def test_buffers_mapped_in_pieces():
    """torch's expandable segments map a tensor piece by piece (20 MiB): taken
    whole. In a process of its own, where the allocator is set up so."""
    import os
    import subprocess
    import sys
    code = """if True:
        import ctypes as C, numpy as np, torch
        from paper_2410_11129_gb300 import fcd, workloads as W
        ch = fcd.Channel(dict(W.C2))
        ch.step(2)
        N = ch.nx * ch.ny
        t = torch.full((28 * N,), -7.0, dtype=torch.float64, device="cuda")
        base, size = C.c_uint64(), C.c_size_t()
        C.CDLL("libcuda.so.1").cuMemGetAddressRange_v2(C.byref(base), C.byref(size), C.c_uint64(t.data_ptr()))
        assert size.value < 8 * 28 * N, "not in pieces"
        at = lambda n: C.c_void_p(t.data_ptr() + 8 * n)
        L = fcd.load()
        assert L.fcd_get_populations(ch.h, at(0), at(9 * N), at(27 * N)) == 0
        got = t.cpu().numpy()
        assert np.array_equal(got, np.concatenate([a.ravel() for a in ch.populations()]))
        assert L.fcd_set_populations(ch.h, at(0), at(9 * N), at(27 * N), 2) == 0
        assert np.array_equal(got, np.concatenate([a.ravel() for a in ch.populations()]))
        print("whole")
    """
    env = dict(os.environ, PYTORCH_CUDA_ALLOC_CONF="expandable_segments:True")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "whole" in r.stdout, r.stdout + r.stderr
