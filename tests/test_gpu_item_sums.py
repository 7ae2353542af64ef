"""A shard's fixed-point item sums on each side of what shared memory holds (both
sums, one, none): the exact integers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("J", [50, 14_000, 15_000, 28_000, 30_000, 65_536])
def test_shard_item_sums_are_exact(dlm_lib, J, bf16):
    rng = np.random.default_rng(J)
    I, d = 4001, 9
    rp = d * np.arange(I + 1, dtype=np.int64)
    start = (rng.integers(0, J, size=I) ** 2 // J)[:, None]  # popular items among the first
    col = ((start + np.arange(d) * (J // d)) % J).reshape(-1).astype(np.int32)
    a = torch.from_numpy(rng.uniform(-1.5, 1.5, I * d).astype(np.float32)).cuda()
    a = a.bfloat16() if bf16 else a
    args = (torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), a, a, torch.ones(J, dtype=torch.float64).cuda())
    loc, deg = dlm_lib.shard_local(*args, J)
    assert np.array_equal(deg, np.bincount(col, minlength=J))
    g = dlm_lib.shard_combine([loc], [deg])
    sq, s1 = dlm_lib.shard_item_sums(*args, g, J)
    v = a.float().cpu().numpy()

    def shift(bound):
        return min(int(np.floor(61.0 - np.log2(bound))), 100)

    big = g["max_abs_a"]
    f = lambda x, s: np.rint((x * np.float32(2.0 ** s)).astype(np.float64)).astype(np.int64)  # noqa: E731
    want_sq, want_s1 = np.zeros(J, np.int64), np.zeros(J, np.int64)
    np.add.at(want_sq, col, f(v * v, shift(g["max_item_degree"] * big * big)))
    np.add.at(want_s1, col, f(v, shift(g["max_item_degree"] * big)))
    assert np.array_equal(sq, want_sq) and np.array_equal(s1, want_s1)
