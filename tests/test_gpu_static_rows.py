"""The allocation-free evaluation at the edges of its row classes and of its
item storage: rows around the 64 edges a group of eight lanes holds in
registers and around the 32 lanes of the wide path, empty rows, row counts
that leave a group of four rows ragged, arrays that start off a 16-byte
boundary, and item counts on both sides of what shared memory holds (two
blocks an SM, one, none).  Against the oracle's FP64 sweep with the bounds of
test_zz_no_alloc.py."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, x_error_report

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DEGREES = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 56, 57, 63, 64, 65, 66, 96, 97, 200]


def instance(J, I, seed):
    rng = np.random.default_rng(seed)
    deg = rng.choice([d for d in DEGREES if d <= J], size=I)
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = -rng.lognormal(0, 0.5, rp[-1]).astype(np.float32)
    a = rng.uniform(0.5, 1.5, rp[-1]).astype(np.float32)
    b = 0.05 * np.bincount(col, weights=a, minlength=J)
    return synth.Instance(rp, col, c, a, b, J)


def off_boundary(v, by):
    """The array on the device, starting `by` elements past an aligned address."""
    t = torch.empty(len(v) + by, dtype=torch.from_numpy(v).dtype, device="cuda")
    t[by:] = torch.from_numpy(v).cuda()
    return t[by:]


@pytest.mark.parametrize("J,I,kind,by", [(210, 1, oracle.SIMPLEX_LE, 0), (210, 1003, oracle.SIMPLEX_LE, 1),
                                         (210, 1001, oracle.SIMPLEX_EQ, 2), (210, 1002, oracle.BOX, 3),
                                         (8533, 700, oracle.SIMPLEX_LE, 0), (8600, 700, oracle.SIMPLEX_LE, 1),
                                         (18_900, 700, oracle.SIMPLEX_EQ, 0), (65_536, 700, oracle.SIMPLEX_LE, 3)])
def test_static_rows_match_the_oracle(dlm_lib, J, I, kind, by):
    inst = instance(J, I, 41 + I)
    p = oracle_problem(inst, kind, 1.0)
    rng = np.random.default_rng(7)
    rp = torch.from_numpy(inst.row_ptr).cuda()
    col, c, a = (off_boundary(v, by) for v in (inst.col, inst.c, inst.a))
    b = torch.from_numpy(inst.b).cuda()
    g = torch.zeros(1, dtype=torch.float64, device="cuda")
    for gamma in (1e-1, 1e-3):
        lam32 = rng.uniform(0, 1.2, J).astype(np.float32)
        lam = torch.from_numpy(lam32).cuda()
        grad = torch.empty(J, dtype=torch.float32, device="cuda")
        x = off_boundary(np.full(inst.nnz, np.nan, np.float32), by)
        dlm_lib.dlm_calculate_static(inst.I, J, inst.nnz, rp, col, c, a, b, kind, 1.0, lam, gamma, g, grad, x, None)
        torch.cuda.synchronize()
        lam64 = lam32.astype(np.float64)
        ref = oracle.sweep(p, lam64, gamma)
        dx, tol = x_error_report(x.cpu().numpy(), ref["x"], p, lam64, gamma)
        assert (dx <= tol).all(), dx.max()
        scale = np.bincount(p.col, weights=p.a * ref["x"], minlength=J) + np.abs(p.b)
        allow = np.bincount(p.col, weights=p.a * np.maximum(tol - 2e-6, 0), minlength=J)
        dg = np.abs(grad.cpu().numpy().astype(np.float64) - ref["grad"])
        assert (dg <= 2e-6 * scale + allow + 1e-6).all(), dg.max()
        assert abs(g.item() - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"])), (g.item(), ref["g"])
