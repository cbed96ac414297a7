"""The screened interaction outside the range of well-behaved matrices. An eps that is not positive
definite is an error wherever its large entries stand; an eps whose diagonal spans many decades is as
exact as one with a unit diagonal; a spectrum of many decades costs no more than the float-float
storage does; below 257 basis functions small entries of eps keep their own relative precision.

An indefinite eps: the identity but for a pair of off-diagonal entries of magnitude above 1, in a
32-block, a 128-block or a panel other than the pivot's. The factor's entry passes the bound
sqrt(eps_ii) of a positive definite matrix, and the pivot 1 - |x|^2 is negative.

Scales: for eps = S B S with S diagonal, eps^-1 = S^-1 B^-1 S^-1, and Cholesky, inverse and product
keep the errors relative to S, |d eps^-1_IJ| <= c sqrt(eps^-1_II eps^-1_JJ) with c of the order of
2^-48 times N and the condition number of B. With B within 1 of the identity by 0.5 (condition 3) and
N <= 700: 1e-11 would be generous, 2e-12 is asked for; the FP64 inverse that it is compared with is
scaled the same way.

Spectra: eps = H diag(lambda) H^T / N with a Hadamard matrix and powers of two from 1 to kappa is exact
in FP64, and so is its inverse. Float-float rounds every entry of eps and of the panels' updates by
2^-49 at most; entries are sqrt(N) below the largest eigenvalue, so the rounding errors (rms 0.3 of
their bound, the 2-norm of N x N of them 2 sqrt(N) rms) disturb eps by 0.1 to 0.2 of 2^-48 kappa for
the few updates of an entry: 0.4 2^-48 kappa of eps^-1 in the Frobenius norm.
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



@pytest.mark.parametrize("n,real", [(200, False), (300, False), (513, True), (640, False)])
@pytest.mark.parametrize("lo,hi", [(-2, 2), (-3, 3), (0, 6)])
def test_scaled_diagonal(gw, n, real, lo, hi):
    g = torch.Generator(device="cuda").manual_seed(n + hi)
    x = torch.randn((n, n, 2), generator=g, dtype=torch.float64, device="cuda")
    x = x[..., 0].to(torch.complex128) if real else torch.view_as_complex(x)
    x = x + x.mH
    B = torch.eye(n, dtype=torch.complex128, device="cuda") + 0.5 * x / torch.linalg.matrix_norm(x, 2)
    u = torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
    s = 2.0 ** torch.round(3.3219 * (lo + (hi - lo) * u))
    eps = s[:, None] * B * s[None, :]
    W = w_of(gw, eps, real)
    gw.check()
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    inv = torch.linalg.inv((eye - (eye - eps)) / (s[:, None] * s[None, :]))     # of the P passed in
    off = ~eye.bool()
    assert float(((W * s[:, None] * s[None, :] - inv).abs())[off].max()) <= 2e-12


def hadamard_system(n, decades, real, seed):
    """eps = H diag(lambda) H^T / n with powers of two up to 2^decades (and phases), and its inverse."""
    H = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    while H.shape[0] < n:
        H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)], 0)
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.arange(n, device="cuda") * (decades + 1) // n
    lam = 2.0 ** k[torch.randperm(n, generator=g, device="cuda")].double()
    sign = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, -1.0, 1.0).double()
    H = H * sign[:, None]                               # not the Sylvester matrix itself: its factors are special
    eps, inv = ((H * d[None, :] / n) @ H.T for d in (lam, 1.0 / lam))
    ph = torch.ones(n, dtype=torch.complex128, device="cuda")
    if not real:
        ph = torch.exp(0.5j * torch.pi * torch.randint(4, (n,), generator=g, device="cuda"))
        ph = torch.complex(ph.real.round(), ph.imag.round())
    return [ph[:, None] * x * ph.conj()[None, :] for x in (eps, inv)]


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("decades", [10, 20])
def test_wide_spectrum(gw, real, decades):
    n = 1024
    eps, inv = hadamard_system(n, decades, real, decades)
    W = w_of(gw, eps, real)
    gw.check()
    ref = inv - torch.eye(n, dtype=torch.complex128, device="cuda")
    assert float((W - ref).norm() / inv.norm()) <= 0.4 * 2.0 ** (decades - 48)


@pytest.mark.parametrize("lo", [-20, -26])
@pytest.mark.parametrize("real", [False, True])
def test_small_entries_keep_their_precision(gw, lo, real):
    n = 70
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((n, n, 2), generator=g, dtype=torch.float64, device="cuda")
    x = x[..., 0].to(torch.complex128) if real else torch.view_as_complex(x)
    x = torch.tril(x, -1) * 10.0 ** lo
    x = x + x.mH
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    W = gw.screened_w([-x[None].contiguous()], [torch.ones(n, dtype=torch.float64, device="cuda")],
                      real=real)[0][0]
    gw.check()
    off = ~eye.bool()
    assert float(((W + x).abs() / x.abs().clamp(min=1e-300))[off].max()) <= 1e-12


def test_wide_spectrum_of_small_systems(gw):
    """Two panels, condition 2^30, general phases: the geometric mean over 16 matrices of the error above.
    Complex entries round twice and a product of two takes four real ones: 1.4 to 2 times the 0.1 to 0.2
    of 2^-48 kappa, in the middle 0.25 (and 2^-53 kappa of the phases' own rounding, 0.03). A panel by
    the explicit inverse of the whole 32 x 32 diagonal block adds that block's condition: 0.34."""
    logs = []
    for seed in range(16):
        eps, inv = hadamard_system(64, 30, True, 50 + seed)
        g = torch.Generator(device="cuda").manual_seed(seed)
        ph = torch.exp(2j * torch.pi * torch.rand(64, generator=g, dtype=torch.float64, device="cuda"))
        eps, inv = (ph[:, None] * x * ph.conj()[None, :] for x in (eps, inv))
        W = w_of(gw, eps)
        gw.check()
        ref = inv - torch.eye(64, dtype=torch.complex128, device="cuda")
        logs.append(float(((W - ref).norm() / inv.norm()).log()))
    assert float(torch.tensor(logs).mean().exp()) <= 0.25 * 2.0 ** (30 - 48)
