"""Kernel launches of the screened interaction: as many as bench.py counts for it, and no more when
systems below and above the size limit of the sliced products alternate in the call."""
import os
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def launches(ns, nw):
    import paper_1003_0316_gb300 as gw
    from torch.profiler import ProfilerActivity, profile
    Ps = [torch.zeros((nw, n, n), dtype=torch.complex128, device="cuda") for n in ns]
    vs = [torch.ones(n, dtype=torch.float64, device="cuda") for n in ns]
    gw.screened_w(Ps, vs)
    torch.cuda.synchronize()
    for _ in range(2):                       # the first profile of a process can miss its launches
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            gw.screened_w(Ps, vs)
            torch.cuda.synchronize()
    gw.check()
    n = sum(e.count for e in p.key_averages() if "gw::" in e.key)
    if n == 0:
        pytest.skip("the profiler records no kernels here")
    return n


@pytest.mark.parametrize("n,nsys", [(200, 3), (64, 300), (257, 4), (600, 16), (600, 200), (1025, 2)])
def test_bench_counts_the_dielectric_launches(n, nsys):
    import bench
    nw = 50 if nsys % 50 == 0 else nsys
    assert launches([n] * (nsys // nw), nw) == bench.dielectric_launches(n, nsys)


def test_alternating_sizes_share_their_launches():
    mixed = launches([250, 260] * 4, 3)
    assert mixed == launches([250] * 4, 3) + launches([260] * 4, 3)
