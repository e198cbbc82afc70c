"""Steps of contexts on the legacy default stream, where they run on streams of
the context: the order with work that the caller puts on the default stream (a
device tensor written just before it is imported, populations exported straight
after a step) and between one-step and many-step calls is kept, and the bits are
those of a context on a stream of its own (needs a GB300)."""
import ctypes as C

import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cfg(i, **kw):
    return dict(W.small(nx=130 + 32 * i, ny=41, r1=6.0, r2=12.0, xc=40.0, Bo_m=1.0 + 0.5 * i, mag_tol=1e-4,
                        **kw), precision="fp32")


@pytest.mark.parametrize("open_x", [0, 1])
@pytest.mark.parametrize("calls", [(1, 1, 1, 1, 1, 1), (6,), (1, 3, 1, 1), (2, 1, 3)])
def test_legacy_stream_keeps_its_order(calls, open_x):
    import torch
    from paper_2410_11129_gb300 import fcd
    L = fcd.load()
    assert torch.cuda.current_stream().cuda_stream == 0
    own = torch.cuda.Stream()
    chs = [fcd.Channel(_cfg(i, open_x=open_x)) for i in range(5)]
    refs = [fcd.Channel(_cfg(i, open_x=open_x), stream=own.cuda_stream) for i in range(5)]
    start = [ch.populations() for ch in refs]
    big = torch.empty(1 << 26, device="cuda")
    for rep in range(3):
        ins = []
        for ch, (f, g, psi) in zip(chs, start):
            big.normal_()  # keeps the default stream busy in front of the copies
            dev = [(torch.from_numpy(a).to("cuda") * 0.5) * 2.0 for a in (f, g, psi)]
            ins.append(dev)
            assert L.fcd_set_populations(ch.h, *[C.c_void_p(t.data_ptr()) for t in dev], 0) == fcd.FCD_OK
        for ref, p in zip(refs, start):
            ref.set_populations(*p, step=0)
        for n in calls:
            for ch in chs:
                ch.step(n)
            big.add_(1.0)
        for n in calls:
            for ref in refs:
                ref.step(n)
        for ch, ref in zip(chs, refs):
            f = torch.zeros((9, ch.ny, ch.nx), dtype=torch.float64, device="cuda")
            assert L.fcd_get_populations(ch.h, C.c_void_p(f.data_ptr()), None, None) == fcd.FCD_OK
            want = ref.populations()
            assert np.array_equal(f.cpu().numpy(), want[0])
            for x, y in zip(ch.populations(), want):
                assert np.array_equal(x, y)
    for ch in chs + refs:
        ch.close()


@pytest.mark.parametrize("others", [0, 1])
def test_a_synchronised_legacy_stream_has_no_step_left(others):
    """A caller that moves a context to another stream after synchronising, alone
    on the default stream or not (its single steps take another route then)."""
    import torch
    from paper_2410_11129_gb300 import fcd
    a, b = fcd.Channel(_cfg(0)), fcd.Channel(_cfg(0))
    more = [fcd.Channel(_cfg(1)) for _ in range(others)]
    for ch in more:
        ch.step(1)
    s = torch.cuda.Stream()
    for _ in range(20):
        a.step(1)
        torch.cuda.current_stream().synchronize()
        a.check(fcd.load().fcd_set_stream(a.h, C.c_void_p(s.cuda_stream)))
        a.step(1)
        s.synchronize()
        a.check(fcd.load().fcd_set_stream(a.h, None))
        a.step(2)
    b.step(80)
    for x, y in zip(a.populations(), b.populations()):
        assert np.array_equal(x, y)
    for ch in [a, b] + more:
        ch.close()
