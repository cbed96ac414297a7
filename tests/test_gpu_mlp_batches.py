"""Loss and gradient of one training pass at the edges of its distribution: passes of four curves,
one pass per SM before the first CTA takes a second one, ragged ends, and parameters and gradient
that are not 16-byte aligned. FP32 sums of at most 128 terms per layer against the FP64 oracle:
2e-6 per layer, amplified by the poles of the loss; 1e-5 of the loss and 1e-4 of the gradient."""
import numpy as np
import pytest

import synth_inputs as S
from oracle import mlp as OM

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,off", [(1, 0), (3, 1), (4, 0), (5, 2), (607, 0), (611, 3), (1301, 0)])
def test_batches(n, off):
    import paper_1003_0316_gb300 as gw
    om = S.omega_mesh(24)
    y, _ = S.model_sigma_curves(S.SEED_BASE + 100, n, om, first=31)
    w0 = gw.mlp_init(11)
    npar = gw.mlp_param_count()
    w = torch.empty(npar + 4, device="cuda")[off:off + npar]
    grad = torch.full((npar + 4,), 7.0, device="cuda")
    w.copy_(w0)
    loss = torch.full((1,), 3.0, device="cuda")
    gw.mlp_train_step(torch.as_tensor(y, device="cuda"), om, w, grad[off:off + npar], None, None, 0.0, 1,
                      loss)
    gw.check()
    L, g = OM.loss_and_grads(OM.unpack(w0.cpu().numpy().astype(np.float64)), om, y)
    g = OM.pack(g)
    got = grad.cpu().numpy().astype(np.float64)
    assert abs(float(loss) - L) <= 1e-5 * abs(L)
    assert np.linalg.norm(got[off:off + npar] - g) <= 1e-4 * np.linalg.norm(g)
    assert np.all(got[:off] == 7.0) and np.all(got[off + npar:] == 7.0)
