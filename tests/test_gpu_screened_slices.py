"""The screened interaction of larger systems, whose products run on the tensor cores from digit
slices, against an FP64 solve on the device: sizes at the edges of its 128-blocks, 32-blocks and doubling
steps, mixed sizes in one call, in place, and the error of a matrix that is not positive definite.

Bound: relative Frobenius error 1e-12, the bound of the FP64 path (the float-float storage of eps
leaves 2^-48 times the condition number, about 3e-14 here; the slices carry 56 bits).
"""
import numpy as np
import pytest

import synth_inputs as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    import paper_1003_0316_gb300 as g
    return g


def system(n, nw, seed, real=False):
    g = torch.Generator(device="cuda").manual_seed(seed)
    K = 2 * n
    M = torch.randn((K, n, 2), generator=g, dtype=torch.float64, device="cuda")
    M /= 1.0 + torch.arange(n, device="cuda", dtype=torch.float64)[:, None] / 16.0
    M = torch.view_as_complex(M)
    if real:
        M = M.real.to(torch.complex128)
    d = 0.05 + 2.4 * torch.rand(K, generator=g, dtype=torch.float64, device="cuda")
    P = []
    for w in S.omega_mesh(max(nw, 4))[:nw]:
        X = (M * (-12800.0 / K * d / (d * d + w * w))[:, None]).T @ M.conj()
        P.append(0.5 * (X + X.mH))
    v = torch.as_tensor(S.coulomb_eigenvalues(n), device="cuda")
    return torch.stack(P), v


def solve(P, v):
    s = v.sqrt()
    out = []
    for p in P:
        X = s[:, None] * p * s[None, :]
        L = torch.linalg.cholesky(torch.eye(len(s), dtype=X.dtype, device="cuda") - X)
        out.append(s[:, None] * torch.cholesky_solve(X, L) * s[None, :])
    return torch.stack(out)


def err(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("n,nw,real", [(256, 2, False), (257, 3, False), (288, 1, False), (289, 1, False),
                                       (384, 2, False), (385, 1, False), (511, 1, False), (512, 1, False),
                                       (513, 2, False), (640, 1, False), (1025, 1, False), (448, 1, True),
                                       (449, 3, True), (512, 1, True), (777, 2, True)])
def test_sizes(gw, n, nw, real):
    P, v = system(n, nw, n + nw, real)
    W = gw.screened_w([P], [v], real=real)[0]
    gw.check()
    assert err(W, solve(P, v)) <= 1e-12
    assert torch.equal(W, W.mH)
    if real:
        assert torch.count_nonzero(W.imag) == 0


def test_mixed_sizes_in_one_call_and_in_place(gw):
    ns = [300, 40, 513, 260, 256, 129, 700]
    sys_ = [system(n, 2, 7 + n) for n in ns]
    ref = [solve(P, v) for P, v in sys_]
    Ps = [P for P, _ in sys_]
    W = gw.screened_w(Ps, [v for _, v in sys_])
    gw.check()
    for a, b in zip(W, ref):
        assert err(a, b) <= 1e-12
    gw.screened_w(Ps, [v for _, v in sys_], out=Ps)
    gw.check()
    for a, b in zip(Ps, W):
        assert torch.equal(a, b)


def test_not_positive_definite_and_not_finite(gw):
    P, v = system(300, 1, 3)
    gw.screened_w([-P], [v])
    with pytest.raises(gw.GWError) as e:
        gw.check()
    assert e.value.code == gw.GW_ENOTHPD
    for i, j in ((5, 200), (200, 5)):            # both triangles are checked
        Q = P.clone()
        Q[0, i, j] = complex(float("nan"), 0.0)
        gw.screened_w([Q], [v])
        with pytest.raises(gw.GWError) as e:
            gw.check()
        assert e.value.code in (gw.GW_ENONFINITE, gw.GW_ENOTHPD)
    W = gw.screened_w([P], [v])[0]
    gw.check()
    assert err(W, solve(P, v)) <= 1e-12
