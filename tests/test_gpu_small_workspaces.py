"""Workspaces without room for the digit slices: a call takes what its FP64 (or float-float) arithmetic
needs by itself and gives the same results within the bounds of the two (1e-12 of the Frobenius norm);
one byte less is an error."""
import pytest

import synth_inputs as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    import paper_1003_0316_gb300 as g
    return g


def buf(n):
    return torch.empty(int(n), dtype=torch.uint8, device="cuda")


def randn(g, *shape):
    return torch.view_as_complex(torch.randn((*shape, 2), generator=g, dtype=torch.float64, device="cuda"))


def err(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("real", [False, True])
def test_screened_w(gw, real):
    """The size in gw.h: 16 (8 for real systems) x (2 N^2 + 1024 ceil(N / 32)) per system."""
    ns, nw = [300, 40, 520, 600], 2
    g = torch.Generator(device="cuda").manual_seed(2)
    Ps, vs = [], []
    for n in ns:
        X = randn(g, nw, n, 2 * n) / (1.0 + torch.arange(n, device="cuda", dtype=torch.float64)[:, None] / 16.0)
        if real:
            X = X.real.to(torch.complex128)
        P = -(X @ X.mH) / n
        Ps.append(0.5 * (P + P.mH))
        vs.append(torch.as_tensor(S.coulomb_eigenvalues(n), device="cuda"))
    ref = gw.screened_w(Ps, vs, real=real)
    gw.check()
    least = sum(nw * -(-(8 if real else 16) * (2 * n * n + 1024 * -(-n // 32)) // 256) * 256 for n in ns)
    for more in (0, 3 << 20, 30 << 20, 60 << 20, 150 << 20, 400 << 20):
        W = gw.screened_w(Ps, vs, ws=buf(least + more), real=real)
        gw.check()
        assert max(err(a, b) for a, b in zip(W, ref)) <= 1e-12
    with pytest.raises(gw.GWError) as e:
        gw.screened_w(Ps, vs, ws=buf(least - 1), real=real)
    assert e.value.code == gw.GW_EWORKSPACE


def test_polarization(gw):
    """64 KB per 64 x 64 tile of P, frequency and split of K hold the FP64 kernel's partial sums; at most
    K / 512 splits."""
    sizes, om = [(3000, 100), (20, 30), (1500, 64), (500, 200)], S.omega_mesh(4)[:2]
    g = torch.Generator(device="cuda").manual_seed(3)
    Ms = [randn(g, K, nb) for K, nb in sizes]
    ds = [0.05 + 2.0 * torch.rand(K, generator=g, dtype=torch.float64, device="cuda") for K, _ in sizes]
    ref = gw.polarization(Ms, ds, om, 0.25, "fp64")
    gw.check()
    least = 0
    for K, nb in sizes:
        t = -(-nb // 64)
        least += t * (t + 1) // 2 * len(om) * max(1, K // 512) * 65536
    full = gw.polarization_workspace([K for K, _ in sizes], [nb for _, nb in sizes], len(om), "fp64")
    assert least < full
    P = gw.polarization(Ms, ds, om, 0.25, "fp64", ws=buf(least))
    gw.check()
    assert max(err(a, b) for a, b in zip(P, ref)) <= 1e-12
    with pytest.raises(gw.GWError) as e:
        gw.polarization(Ms, ds, om, 0.25, "fp64", ws=buf(65536))
    assert e.value.code == gw.GW_EWORKSPACE


def test_sigma(gw):
    """The FP64 kernel's partial sums: 8 nw npair ceil(N_b / 64) bytes, rounded up to 256."""
    sizes, nw = [(500, 100), (130, 64), (0, 20), (77, 300)], 5
    om = S.omega_mesh(nw)
    g = torch.Generator(device="cuda").manual_seed(4)
    Ms = [randn(g, n, nb) for n, nb in sizes]
    Ws = []
    for _, nb in sizes:
        X = randn(g, nw, nb, 2 * nb)
        Ws.append(-(X @ X.mH))
    es = [torch.rand(n, generator=g, dtype=torch.float64, device="cuda") + 0.1 for n, _ in sizes]
    ps = [torch.arange(n, dtype=torch.int32, device="cuda") % 7 for n, _ in sizes]
    args = ([0.25] * 4, Ms, ps, es, Ws, om, om, 7)
    ref = gw.sigma_c(*args)
    gw.check()
    up = lambda b: -(-b // 256) * 256
    c = sum(up(8 * nw * n) for n, _ in sizes)
    part = up(sum(8 * nw * n * -(-nb // 64) for n, nb in sizes))
    conv = gw._lib.gw_sigma_convolve_workspace(4, gw._arr(gw._i64, [n for n, _ in sizes]))
    least = c + max(part, conv)
    assert least < gw.sigma_workspace([n for n, _ in sizes], [nb for _, nb in sizes], nw, "fp64")
    sig = gw.sigma_c(*args, ws=buf(least))
    gw.check()
    assert err(sig, ref) <= 1e-12
    with pytest.raises(gw.GWError) as e:
        gw.sigma_c(*args, ws=buf(least - 1))
    assert e.value.code == gw.GW_EWORKSPACE
