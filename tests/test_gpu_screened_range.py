"""The screened interaction outside the range of well-behaved matrices: an eps that is not positive
definite is an error wherever its large entries stand.

An indefinite eps: the identity but for a pair of off-diagonal entries of magnitude above 1, in a
32-block, a 128-block or a panel other than the pivot's. The factor's entry passes the bound
sqrt(eps_ii) of a positive definite matrix, and the pivot 1 - |x|^2 is negative.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    import paper_1003_0316_gb300 as g
    return g


def w_of(gw, eps, real=False):
    """W^c for v = 1 of the given eps (P = 1 - eps)."""
    n = eps.shape[0]
    P = torch.eye(n, dtype=torch.complex128, device="cuda") - eps
    return gw.screened_w([P[None].contiguous()], [torch.ones(n, dtype=torch.float64, device="cuda")],
                         real=real)[0][0]


@pytest.mark.parametrize("n,i,j,real", [(257, 256, 0, False), (300, 280, 130, False), (700, 513, 255, False),
                                        (300, 127, 3, False), (449, 448, 5, True), (640, 390, 127, True),
                                        (200, 150, 10, False)])
@pytest.mark.parametrize("x", [1.01, 4.0, 7.6, 8.0, 10.0, 16.0, 1e3, 1e39])
def test_indefinite_is_an_error(gw, n, i, j, real, x):
    eps = torch.eye(n, dtype=torch.complex128, device="cuda")
    z = complex(x, 0.0) if real or n % 2 else complex(0.0, x)
    eps[i, j], eps[j, i] = z, z.conjugate()
    w_of(gw, eps, real)
    with pytest.raises(gw.GWError) as e:
        gw.check()
    assert e.value.code == gw.GW_ENOTHPD
    eps[i, j], eps[j, i] = 0.9 * z / x, 0.9 * z.conjugate() / x        # positive definite
    W = w_of(gw, eps, real)
    gw.check()
    ref = torch.linalg.inv(eps) - torch.eye(n, dtype=torch.complex128, device="cuda")
    assert float((W - ref).abs().max()) <= 1e-12


@pytest.mark.parametrize("n,real", [(300, False), (513, True), (700, False)])
def test_indefinite_random_is_an_error(gw, n, real):
    """Unit diagonal, Hermitian off-diagonal entries of every size from 0 to 12."""
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, n, 2), generator=g, dtype=torch.float64, device="cuda") * 3.0
    x = x[..., 0].to(torch.complex128) if real else torch.view_as_complex(x)
    eps = torch.tril(x, -1)
    eps = eps + eps.mH + torch.eye(n, dtype=torch.complex128, device="cuda")
    w_of(gw, eps, real)
    with pytest.raises(gw.GWError) as e:
        gw.check()
    assert e.value.code == gw.GW_ENOTHPD

