"""Convolution weights over the whole range of energies: the closed-form moments change from a
series to a logarithm where the integration variable passes the pole's distance, and each of the
energies is compared by itself.

Bound 1e-11 of a state's largest value: the recursions of the moments amplify the rounding of
their start (2e-16) at most by 1 / 0.3^3 = 37 in each of three steps' sums, the spline's
coefficients by about 10, and the oracle's quadrature is converged to 1e-13."""
import numpy as np
import pytest

import synth_inputs as S
from oracle import selfenergy as OE

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw,nq", [(4, 1), (12, 3), (33, 2)])
def test_convolution_energy_range(nw, nq):
    import paper_1003_0316_gb300 as gw
    rng = np.random.default_rng(nw)
    om = S.omega_mesh(nw)
    om_out = np.concatenate([S.omega_mesh(16), [-0.7]])          # two blocks of output frequencies
    mag = np.logspace(-3, 3, 7 + nq)
    cs, sts, es, nsig = [], [], [], 0
    for q in range(nq):
        e = rng.permutation(np.concatenate([-mag, mag])[q:])
        cs.append(-rng.uniform(0.1, 2.0, (nw, len(e))) / (1.0 + om[:, None] ** 2))
        es.append(e)
        sts.append((nsig + np.arange(len(e))).astype(np.int32))   # every pair its own state
        nsig += len(e)
    wq = list(rng.uniform(0.2, 1.0, nq))
    T = lambda a: torch.as_tensor(a, device="cuda")
    got = gw.sigma_convolve(wq, [T(c) for c in cs], [T(x) for x in sts], [T(e) for e in es], om,
                            om_out, nsig).cpu().numpy()
    gw.check()
    ref = OE.sigma_c(om, om_out, wq, cs, sts, es, nsig)
    err = np.abs(got - ref).max(axis=1) / np.abs(ref).max(axis=1)
    assert err.max() <= 1e-11
