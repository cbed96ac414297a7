"""The FP64 polarization on the tensor cores (digit slices) against a complex128 reference.

Sizes at the edges of its tiles (128 basis functions), stages (32 rows), superblocks and splits, q
points of unequal size in one call, accumulation, the extrapolar weights' signs, and inputs that
must fall back to the FP64 kernel. Bound: |dP_IJ| <= 1e-14 sqrt(P_II P_JJ). The digits leave
errors below 2^-53 of the largest products; those are at most about 2^6 times the mean square
product here and average over K >= 32 terms (below 1e-15), and the reference's own FP64 sums
stay near 1e-15.
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


def inputs(K, nb, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((K, nb, 2), generator=g, dtype=torch.float64, device="cuda")
    x /= 1.0 + torch.arange(nb, device="cuda", dtype=torch.float64)[:, None] / 16.0
    d = 0.05 + 2.4 * torch.rand(K, generator=g, dtype=torch.float64, device="cuda")
    return torch.view_as_complex(x), d


def reference(M, d, om, pref, dbar=None):
    out = []
    for w in om:
        s = -2.0 * pref * d / (d * d + w * w)
        if dbar is not None:
            s = s + 2.0 * pref * dbar / (dbar * dbar + w * w)
        out.append((M * s[:, None]).T @ M.conj())
    return torch.stack(out)


def scaled_error(P, R, scale=None):
    dg = torch.diagonal(R if scale is None else scale, dim1=1, dim2=2).real.abs().sqrt()
    return float(((P - R).abs() / (dg[:, :, None] * dg[:, None, :])).max())


@pytest.mark.parametrize("K,nb,nw", [(31, 20, 3), (32, 1, 2), (33, 129, 1), (64, 128, 3), (255, 127, 4),
                                     (256, 130, 5), (257, 64, 9), (2053, 257, 2), (8193, 40, 2),
                                     (40001, 97, 1)])
def test_polarization_edges(gw, K, nb, nw):
    M, d = inputs(K, nb, K + nb)
    om = S.omega_mesh(max(nw, 4))[:nw]
    P = gw.polarization([M], [d], om, 0.25, "fp64")[0]
    gw.check()
    R = reference(M, d, om, 0.25)
    assert scaled_error(P, R) <= 1e-14
    assert torch.equal(P, P.mH) and torch.count_nonzero(torch.diagonal(P, dim1=1, dim2=2).imag) == 0
    # the same sum in two accumulated parts (unequal, not whole stages)
    h = K // 3
    Q = gw.polarization([M[:h]], [d[:h]], om, 0.25, "fp64")
    gw.polarization([M[h:]], [d[h:]], om, 0.25, "fp64", out=Q, options={"accumulate": True})
    gw.check()
    assert scaled_error(Q[0], R) <= 1e-14


def test_polarization_uneven_batch(gw):
    sizes = [(500, 33), (20, 50), (3000, 200), (97, 8)] + [(64 + 7 * i, 20 + 3 * i) for i in range(20)]
    om = S.omega_mesh(5)
    ins = [inputs(K, nb, 100 + i) for i, (K, nb) in enumerate(sizes)]
    P = gw.polarization([m for m, _ in ins], [d for _, d in ins], om, 0.5, "fp64")
    gw.check()
    for (M, d), p in zip(ins, P):
        assert scaled_error(p, reference(M, d, om, 0.5)) <= 1e-14


def test_extrapolar_weights_of_both_signs(gw):
    K, nb, nkn = 700, 60, 10
    M, d = inputs(K, nb, 5)
    om = S.omega_mesh(6)
    dbar = torch.full((K,), 0.8, dtype=torch.float64, device="cuda")
    C = torch.zeros((nkn, nb, nb), dtype=torch.complex128, device="cuda")
    dk = torch.full((nkn,), 9.0, dtype=torch.float64, device="cuda")
    P = gw.polarization_extrapolar([M], [d], [dbar], [C], [dk], om, 0.25, "fp64")[0]
    gw.check()
    R = reference(M, d, om, 0.25, dbar)
    size = reference(M, d, om, 0.25).abs() + reference(M, dbar, om, 0.25).abs()
    assert scaled_error(P, R, size) <= 1e-14


@pytest.mark.parametrize("what", ["spike", "tiny", "huge", "nan", "inf"])
def test_inputs_outside_the_digits_range_take_the_fp64_kernel(gw, what):
    """One q of two is bad: it gets what FP64 arithmetic gives, the other is unaffected."""
    K, nb = 4096, 70
    M, d = inputs(K, nb, 9)
    M2, d2 = inputs(K, nb, 10)
    bad = M2.clone()
    if what == "spike":
        bad[7, 3] = 1e9
    elif what == "tiny":
        bad[:, 3] *= 1e-120
    elif what == "huge":
        bad[:, 3] *= 1e120
    else:
        bad[7, 3] = complex(float(what), 0.0)
    om = S.omega_mesh(4)[1:3]
    P, Pb = gw.polarization([M, bad], [d, d2], om, 0.25, "fp64")
    gw.check()
    assert scaled_error(P, reference(M, d, om, 0.25)) <= 1e-14
    R = reference(bad, d2, om, 0.25)
    rest = [i for i in range(nb) if i != 3]
    sub = lambda X: X[:, rest][:, :, rest]
    assert scaled_error(sub(Pb), sub(R)) <= 1e-14
    if what in ("nan", "inf"):
        assert not torch.isfinite(Pb[:, 3]).any() and not torch.isfinite(Pb[:, :, 3]).any()
    else:
        # entry by entry against the sum of magnitudes, which fixed-point digits would miss
        mag = reference(bad.abs().to(torch.complex128), d2, om, 0.25).abs()
        assert float(((Pb - R).abs() / mag).max()) <= 1e-14


# ---------------------------------------------------------------- pair coefficients
def pair_inputs(npair, nb, nw, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    M, _ = inputs(npair, nb, seed)
    W = torch.view_as_complex(torch.randn((nw, nb, nb, 2), generator=g, dtype=torch.float64, device="cuda"))
    dec = 1.0 / (1.0 + torch.arange(nb, device="cuda", dtype=torch.float64))
    return M, W * (dec[:, None] * dec[None, :]).sqrt()


def pair_reference(M, W):
    """c and the sum of the magnitudes of its terms (no assumption on W's symmetry)."""
    c = torch.stack([((M @ w.T) * M.conj()).sum(1).real for w in W])
    a = torch.stack([((M.abs() @ w.abs().T) * M.abs()).sum(1) for w in W])
    return c, a


@pytest.mark.parametrize("npair,nb,nw", [(1, 1, 4), (127, 15, 4), (128, 64, 5), (129, 65, 4), (300, 200, 3),
                                         (1000, 97, 17)])
def test_pair_coefficients_edges(gw, npair, nb, nw):
    """|dc| <= 1e-14 of the sum of the magnitudes of the terms (the digits' bound of the module
    docstring; the largest entry of a column of W is below 2^6 times its mean square here)."""
    M, W = pair_inputs(npair, nb, nw, npair + nb)
    c = gw.sigma_pair_coeffs([M], [W])[0]
    gw.check()
    r, a = pair_reference(M, W)
    assert float(((c - r).abs() / a).max()) <= 1e-14


def test_pair_coefficients_batch_and_scales(gw):
    """q points of unequal size (one empty) and of very different scales in one call."""
    ins = [pair_inputs(n, nb, 4, 50 + i) for i, (n, nb) in enumerate([(40, 30), (0, 8), (700, 70), (5, 129)])]
    ins[2] = (ins[2][0] * 1e-25, ins[2][1] * 1e-25)
    ins[3] = (ins[3][0] * 1e25, ins[3][1])
    cs = gw.sigma_pair_coeffs([m for m, _ in ins], [w for _, w in ins])
    gw.check()
    for (M, W), c in zip(ins, cs):
        if M.shape[0]:
            r, a = pair_reference(M, W)
            assert float(((c - r).abs() / a).max()) <= 1e-14


@pytest.mark.parametrize("what", ["nan", "huge"])
def test_pair_coefficients_fall_back(gw, what):
    M, W = pair_inputs(200, 40, 4, 3)
    M2, W2 = M.clone(), W.clone()
    if what == "nan":
        W2[1, 3, 5] = float("nan")
    else:
        M2 *= 1e40
    c, c2 = gw.sigma_pair_coeffs([M, M2], [W, W2])
    gw.check()
    r, a = pair_reference(M, W)
    assert float(((c - r).abs() / a).max()) <= 1e-14
    r2, a2 = pair_reference(M2, W2)
    assert torch.equal(torch.isfinite(c2), torch.isfinite(r2))
    ok = torch.isfinite(r2)
    assert float(((c2 - r2).abs() / a2)[ok].max()) <= 1e-14
