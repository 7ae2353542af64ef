"""The allocation-free evaluation at large magnitudes: item terms |a| x on both
sides of 2^55, where the exponent of the fixed-point item sums reaches its lower
end (the sums themselves stay below 2^63), and an objective whose sum is past the
largest float.  Against the oracle's FP64 sweep with the bounds of test_gpu_static_rows.py."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, x_error_report

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def evaluate(dlm_lib, inst, kind, lam32, gamma):
    t = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    g = torch.zeros(1, dtype=torch.float64, device="cuda")
    grad = torch.empty(inst.J, dtype=torch.float32, device="cuda")
    x = torch.empty(inst.nnz, dtype=torch.float32, device="cuda")
    dlm_lib.dlm_calculate_static(inst.I, inst.J, inst.nnz, t(inst.row_ptr), t(inst.col), t(inst.c), t(inst.a),
                                 t(inst.b), kind, 1.0, t(lam32), gamma, g, grad, x, None)
    torch.cuda.synchronize()
    return g.item(), grad.cpu().numpy(), x.cpu().numpy()


@pytest.mark.parametrize("kind", [oracle.SIMPLEX_LE, oracle.SIMPLEX_EQ, oracle.BOX])
@pytest.mark.parametrize("I,degrees", [(5, [1, 2, 3]), (100, [1, 2, 7, 8, 9, 33, 40]), (60, [65, 70])])
@pytest.mark.parametrize("exp", [50, 54, 55, 57])
def test_terms_around_2_to_55(dlm_lib, exp, I, degrees, kind):
    J = 80
    rng = np.random.default_rng(exp + I)
    deg = rng.choice(degrees, size=I)
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = -rng.lognormal(0, 0.5, rp[-1]).astype(np.float32)
    a = np.ldexp(rng.uniform(0.5, 1.5, rp[-1]), exp).astype(np.float32)
    inst = synth.Instance(rp, col, c, a, 0.05 * np.bincount(col, weights=a.astype(np.float64), minlength=J), J)
    p = oracle_problem(inst, kind, 1.0)
    gamma = 1e-1 if kind != oracle.BOX else 10.0  # (a box takes x = u / gamma < 1 here: the sums stay below 2^63)
    lam32 = np.ldexp(rng.uniform(0, 0.5, J), -exp).astype(np.float32)
    lam64 = lam32.astype(np.float64)
    ref = oracle.sweep(p, lam64, gamma)
    total = np.bincount(p.col, weights=p.a * ref["x"], minlength=J)
    assert total.max() < 2.0 ** 63
    g, grad, x = evaluate(dlm_lib, inst, kind, lam32, gamma)
    dx, tol = x_error_report(x, ref["x"], p, lam64, gamma)
    assert (dx <= tol).all(), dx.max()
    scale = total + np.abs(p.b)
    allow = np.bincount(p.col, weights=p.a * np.maximum(tol - 2e-6, 0), minlength=J)
    dg = np.abs(grad.astype(np.float64) - ref["grad"])
    assert (dg <= 2e-6 * scale + allow + 1e-6).all(), (dg / scale).max()
    assert abs(g - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"])), (g, ref["g"])


def test_objective_past_the_largest_float(dlm_lib):
    I, J = 200_000, 50  # ten rows a lane, some 5e37 each
    rng = np.random.default_rng(9)
    rp = 2 * np.arange(I + 1, dtype=np.int64)
    first = rng.integers(0, J, size=I)
    col = np.stack([first, (first + rng.integers(1, J, size=I)) % J], 1).reshape(-1).astype(np.int32)
    c = (-1e37 * rng.uniform(4, 8, 2 * I)).astype(np.float32)
    a = rng.uniform(0.5, 1.5, 2 * I).astype(np.float32)
    inst = synth.Instance(rp, col, c, a, np.ones(J), J)
    p = oracle_problem(inst, oracle.SIMPLEX_LE, 1.0)
    lam32 = (1e36 * rng.uniform(0, 1, J)).astype(np.float32)
    gamma = 1e36
    ref = oracle.sweep(p, lam32.astype(np.float64), gamma)
    g, _, _ = evaluate(dlm_lib, inst, oracle.SIMPLEX_LE, lam32, gamma)
    assert abs(g - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"])), (g, ref["g"])
