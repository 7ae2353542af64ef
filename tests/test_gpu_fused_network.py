"""The fused network (widths up to 256) at the edges of its tiles: row counts
around one 128-row tile and beyond one tile per SM (a CTA then adds several
tiles into its slot), widths around the 128-column block and the widest it
takes, and the first width past it (the separate kernels).  Against the FP64
reference with the same BF16 roundings; the bounds of test_gpu_warmstart.py."""
import numpy as np
import pytest

from oracle import mlp
from test_gpu_warmstart import ws_with_random_params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("H,n", [(128, 1), (128, 127), (128, 129), (120, 20_000), (128, 40_001), (144, 128),
                                 (248, 20_000), (256, 129), (264, 300)])
def test_fused_network_matches_reference(dlm_lib, H, n):
    ws, P, X, y, mu, sd = ws_with_random_params(dlm_lib, H=H, seed=17, n=max(n, 50))
    X, y = X[:n], y[:n]
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    out = ws.predict(Xd).cpu().numpy().astype(np.float64)
    ref = mlp.predict(P, X.astype(np.float64), mu, sd, bf16_round=True)
    assert (np.abs(out - ref) <= 5e-3 * (np.abs(ref) + 0.1)).all()
    loss, g = ws.loss_grad(Xd, yd)
    rl, rg = mlp.loss_and_grad(P, X.astype(np.float64), y.astype(np.float64), mu, sd, bf16_round=True)
    assert abs(loss - rl) <= 1e-4 * rl + 1e-12
    G = ws.unpack(g)
    for k in rg:
        d = np.linalg.norm(G[k].astype(np.float64) - rg[k])
        assert d <= 1e-2 * np.linalg.norm(rg[k]) + 1e-9, (k, d / np.linalg.norm(rg[k]))
    # the same bits on a second call
    loss2, g2 = ws.loss_grad(Xd, yd)
    assert loss2 == loss and np.array_equal(g, g2)
    ws.close()
