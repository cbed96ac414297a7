"""FP64 results of operands whose entries differ by many orders of magnitude, against sums of FP64
terms: where the digit slices of the tensor-core path would lose what FP64 keeps, the call has to
notice it.

Bound of the pair coefficients: 1e-14 of the sum of the magnitudes of the terms (the bound of the
digit slices for well-scaled operands; a change of scales s of the basis, x_I -> s_I x_I and W_IJ ->
W_IJ / (s_I s_J), by powers of two changes neither the terms nor their sum).
"""
import pytest

import synth_inputs as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    import paper_1003_0316_gb300 as g
    return g


def randn(g, *shape):
    return torch.view_as_complex(torch.randn((*shape, 2), generator=g, dtype=torch.float64, device="cuda"))


def pairs(npair, nb, nw, seed, kind):
    """Projections and W: negative definite, Hermitian without a diagonal, or general."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    M = randn(g, npair, nb)
    if kind == "definite":
        X = randn(g, nw, nb, 2 * nb)
        W = -(X @ X.mH)
        W = 0.5 * (W + W.mH)
    else:
        W = randn(g, nw, nb, nb)
        if kind == "hollow":
            W = W + W.mH
            W.diagonal(dim1=1, dim2=2).zero_()
    return M, W, g


def check_pairs(gw, M, W):
    c = gw.sigma_pair_coeffs([M], [W])[0]
    gw.check()
    r = torch.stack([((M @ w.T) * M.conj()).sum(1).real for w in W])
    a = torch.stack([((M.abs() @ w.abs().T) * M.abs()).sum(1) for w in W])
    assert float(((c - r).abs() / a).max()) <= 1e-14


@pytest.mark.parametrize("kind", ["definite", "hollow", "general"])
@pytest.mark.parametrize("npair,nb,nw,decades", [(130, 48, 4, 2), (64, 48, 4, 8), (200, 129, 4, 4),
                                                 (90, 300, 4, 12), (300, 70, 9, 14)])
def test_pair_coefficients_of_scaled_basis(gw, npair, nb, nw, decades, kind):
    M, W, g = pairs(npair, nb, nw, nb + decades, kind)
    s = 2.0 ** torch.round(3.3219 * decades * (2.0 * torch.rand(nb, generator=g, dtype=torch.float64,
                                                               device="cuda") - 1.0))
    check_pairs(gw, M * s, W / (s[:, None] * s[None, :]))


@pytest.mark.parametrize("kind", ["definite", "hollow"])
def test_pair_coefficients_of_frequencies_of_different_shape(gw, kind):
    """The diagonal of W falls off with the frequency by a different power for every basis function."""
    M, W, g = pairs(150, 60, 6, 11, kind)
    p = 3.0 * torch.rand(60, generator=g, dtype=torch.float64, device="cuda")
    for j in range(6):
        d = (1.0 + 4.0 * j) ** -p
        W[j] = d[:, None] * W[j] * d[None, :]
    check_pairs(gw, M, W)


@pytest.mark.parametrize("big", [1e3, 1e6, 1e12])
def test_pair_coefficients_of_rows_and_columns_with_one_large_entry(gw, big):
    """A row of M and a column of W whose largest entries meet small ones."""
    M, W, _ = pairs(140, 66, 4, 21, "general")
    M[::3, 5] *= big
    W[:, 5, :] *= 1e-3 / big
    W[:, :, 5] *= 1e-3 / big
    W[1, 7, 9] *= big
    W[2, 11, 11] *= big
    check_pairs(gw, M, W)


@pytest.mark.parametrize("m,f", [(1e-20, 1e-40), (1e-25, 1.0), (1e-12, 1e-60), (1e20, 1e-60)])
def test_polarization_of_small_weights(gw, m, f):
    """Products of M and the weights below the FP32 range: the sum over 200 transitions against the
    sum of magnitudes (FP64 sums, 2^-53 per term)."""
    g = torch.Generator(device="cuda").manual_seed(4)
    K, nb, om = 200, 40, S.omega_mesh(4)[:2]
    M = randn(g, K, nb) * m
    d = 0.05 + 2.0 * torch.rand(K, generator=g, dtype=torch.float64, device="cuda")
    ft = torch.full((K,), f, dtype=torch.float64, device="cuda")
    P = gw.polarization([M], [d], om, 0.25, "fp64", fs=[ft])[0]
    gw.check()
    for j, w in enumerate(om):
        s = -0.5 * f * d / (d * d + float(w) ** 2)
        r = (M * s[:, None]).T @ M.conj()
        a = ((M.abs() * s.abs()[:, None]).T @ M.abs())
        assert float(((P[j] - r).abs() / a).max()) <= 3e-14


@pytest.mark.parametrize("K", [300, 700, 5000])
@pytest.mark.parametrize("kind,f", [("spike", 20.0), ("spike", 200.0), ("spike", 600.0), ("gap", 1e-2),
                                    ("gap", 1e-3), ("half", 1e-6)])
def test_polarization_of_uneven_columns(gw, K, kind, f):
    """A few large entries per column, in the same rows for pairs of columns; small gaps; columns that are
    large in one half of the rows. Root mean square error relative to sqrt(P_II P_JJ): the FP64 kernel's
    sums of K terms, about 2^-53 (1.1e-16) per partial sum, give at most 3e-16 for any of these; digits
    with a share of that from every term would give more."""
    g = torch.Generator(device="cuda").manual_seed(K)
    nb = 70
    M = randn(g, K, nb)
    d = 0.05 + 2.0 * torch.rand(K, generator=g, dtype=torch.float64, device="cuda")
    col = torch.arange(nb, device="cuda")
    if kind == "spike":
        rows = torch.randint(K, (nb // 2 + 1,), generator=g, device="cuda")[col // 2]
        M[rows, col] *= f
    elif kind == "gap":
        d = d - 0.05 + f
        d[3], d[K // 2] = f, 1.1 * f
    else:
        M[: K // 2, ::2] *= f
        M[K // 2:, 1::2] *= f
    P = gw.polarization([M], [d], [0.0, 1.0], 0.25, "fp64")[0]
    gw.check()
    for j, w in enumerate((0.0, 1.0)):
        s = -0.5 * d / (d * d + w * w)
        hi = torch.zeros((nb, nb, 2), dtype=torch.float64, device="cuda")
        lo = hi.clone()
        for t in range(0, K, 32):                    # FP64 sums of 32 terms, added without rounding
            m = M[t:t + 32]
            x = torch.view_as_real(((m * s[t:t + 32, None]).T @ m.conj()).contiguous())
            a = hi + x
            b = a - hi
            lo += (hi - (a - b)) + (x - b)
            hi = a
        R = torch.view_as_complex(hi + lo)
        dg = R.diagonal().real.abs().sqrt()
        assert float(((P[j] - R).abs() / (dg[:, None] * dg)).square().mean().sqrt()) <= 3e-16
