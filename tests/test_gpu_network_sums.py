"""The fused network's bias and w3 gradients keep FP64's bits over the rows.  All
rows have the same features, so a row's term is its error times one factor:
errors of 2^30 and 2^6 of both signs cancel exactly and leave the small ones, whose
sum must be their number times the term that a call with small errors only
gives -- to n 2^-53 of the largest partial sum, half of it here (48 bits leave none)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("H", [64, 128, 200, 256])
def test_column_sums_keep_small_terms(dlm_lib, H):
    n = 128
    rng = np.random.default_rng(H)
    ws = dlm_lib.WarmStart(H, 3)
    W = [rng.normal(0, 0.3, 7 * H), np.full(H, 0.2), rng.normal(0, 0.05, H * H), np.full(H, 0.2),
         rng.normal(0, 0.01, H), np.zeros(1)]
    ws.set_params(np.concatenate(W), np.zeros(7), np.ones(7))
    X = torch.from_numpy(np.tile(rng.uniform(0, 1, 7).astype(np.float32), (n, 1))).cuda()
    X[:, 4] = 0.0  # the floor: an output of about 1e-6
    out = ws.predict(X).cpu().numpy()
    assert (out == out[0]).all() and 2e-7 < out[0] < 3e-6
    y = np.zeros(n, np.float32)
    _, small = ws.loss_grad(X, torch.from_numpy(y).cuda())
    for half in (0, 64):  # the rows of a thread's column
        y[half], y[half + 63] = -2.0 ** 30, 2.0 ** 30
        y[half + 1], y[half + 62] = -2.0 ** 6, 2.0 ** 6
    big = out[0] - y
    assert (big[y != 0] == -y[y != 0]).all()
    _, mixed = ws.loss_grad(X, torch.from_numpy(y).cuda())
    small, mixed = ws.unpack(small.astype(np.float64)), ws.unpack(mixed.astype(np.float64))
    bound = n * 2.0 ** -53 * 4 * 2.0 ** 30 / out[0] / 120
    for k in ("w3", "b2", "b1"):
        want = small[k] * 120 / n
        on = np.abs(small[k]) > 0
        assert on.any()
        err = np.abs(mixed[k] - want)[on] / np.abs(want)[on]
        assert err.max() <= bound, (k, err.max(), bound)
    ws.close()
