"""Batches whose instances solve in different forms (needs a GB300)."""
import time

import numpy as np
import pytest

from paper_2410_11129_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _small(i):
    return dict(W.small(nx=64, ny=24, Bo_m=1.0 + 0.1 * i, mag_tol=1e-4), precision="fp32")


def _best(step):
    import torch
    t = []
    for _ in range(8):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        step(20)
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t)


def test_only_one_kernel_solves_share_the_gpu():
    """One FP64 channel beside seven small channels of one FP32 plane (64 x 24: a
    few tiles each) steps in no more than half as long again as alone. With an
    eighth of the SMs its solve alone took longer than that."""
    from paper_2410_11129_gb300 import fcd
    one = dict(W.C5)
    ch = fcd.Channel(one)
    ch.step(4)
    alone = _best(ch.step)
    b = fcd.Batch([one] + [_small(i) for i in range(7)])
    b.set_mode(0)
    b.step(4)
    assert _best(b.step) <= 1.5 * alone
    ch.close()
    b.close()


def test_more_solves_than_shares():
    """Eleven pair instances and one FP64 among single-plane ones, each on its own
    stream: the bits of each alone."""
    from paper_2410_11129_gb300 import fcd
    cfgs = [dict(W.small(nx=98 + 32 * (i % 3), ny=33, r1=5.0, r2=10.0, xc=40.0, Bo_m=1.0 + 0.2 * i, mag_tol=1e-6),
                 precision="fp32") for i in range(11)]
    cfgs += [dict(W.small(nx=130, ny=33, mag_tol=1e-10), precision="fp64"), _small(1), _small(2)]
    b = fcd.Batch(cfgs)
    b.set_mode(0)
    b.step(3)
    for cfg, inst in zip(cfgs, b.instances):
        ch = fcd.Channel(cfg)
        ch.step(3)
        for x, y in zip(ch.populations(), inst.populations()):
            assert np.array_equal(x, y)
        ch.close()
    b.close()
