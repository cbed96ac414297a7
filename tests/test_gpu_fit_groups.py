"""The fit kernel for many curves (several curves per warp) returns exactly what the kernel for few
curves (one warp per curve) returns: the same curves in one call and in calls of at most 6,000."""
import numpy as np
import pytest

import synth_inputs as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    import paper_1003_0316_gb300 as g
    return g


@pytest.mark.parametrize("n,nw,npole", [(6144, 4, 1), (6200, 24, 2), (6145, 32, 3), (8192, 13, 2),
                                        (9001, 24, 3), (8200, 31, 1)])
def test_many_curves_equal_few(gw, n, nw, npole):
    om = S.omega_mesh(nw)
    y, sg = S.model_sigma_curves(5, n, om)
    y = torch.as_tensor(y, device="cuda")
    sg = torch.as_tensor(sg, device="cuda")
    y[3] = 0.0                                   # a zero curve, and one that is not finite
    y[5, 1] = complex(float("nan"), 0.0)
    many = gw.continue_fit(y, om, npole=npole, sign=sg)
    few = [torch.cat(t) for t in zip(*(gw.continue_fit(y[i:i + 6000].contiguous(), om, npole=npole,
                                                       sign=sg[i:i + 6000].contiguous())
                                       for i in range(0, n, 6000)))]
    for a, b in zip(many, few):
        assert torch.equal(torch.nan_to_num(a.double(), nan=-7.0), torch.nan_to_num(b.double(), nan=-7.0))


def test_learned_start_many_curves_equal_few(gw):
    n, om = 6500, S.omega_mesh(24)
    y, sg = S.model_sigma_curves(8, n, om)
    y, sg = torch.as_tensor(y, device="cuda"), torch.as_tensor(sg, device="cuda")
    w = gw.mlp_init(1)
    for method in ("mlp", "mlp_only"):
        many = gw.continue_fit(y, om, sign=sg, method=method, mlp=w)
        few = [torch.cat(t) for t in zip(*(gw.continue_fit(y[i:i + 3300].contiguous(), om, method=method,
                                                           sign=sg[i:i + 3300].contiguous(), mlp=w)
                                           for i in range(0, n, 3300)))]
        for a, b in zip(many, few):
            assert torch.equal(a, b)


@pytest.mark.parametrize("n,nw,npole", [(5000, 4, 1), (8001, 40, 1), (3500, 24, 2), (5607, 33, 2),
                                        (12200, 16, 2), (2000, 24, 3), (2003, 6, 3), (3210, 64, 3)])
def test_groups_equal_one_curve_per_warp(gw, n, nw, npole):
    """From the smallest numbers of curves that several per warp are taken for; the calls of at most
    1,900 curves take one warp per curve."""
    om = S.omega_mesh(nw)
    y, sg = S.model_sigma_curves(6, n, om)
    y = torch.as_tensor(y, device="cuda")
    sg = torch.as_tensor(sg, device="cuda")
    y[2] = 0.0
    y[4, 3] = complex(0.0, float("inf"))
    many = gw.continue_fit(y, om, npole=npole, sign=sg)
    few = [torch.cat(t) for t in zip(*(gw.continue_fit(y[i:i + 1900].contiguous(), om, npole=npole,
                                                       sign=sg[i:i + 1900].contiguous())
                                       for i in range(0, n, 1900)))]
    for a, b in zip(many, few):
        assert torch.equal(torch.nan_to_num(a.double(), nan=-7.0), torch.nan_to_num(b.double(), nan=-7.0))
