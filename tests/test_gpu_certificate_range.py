"""The certificate's objective keeps FP64's range whatever the magnitudes are:
ridges far above the costs (x = u / gamma, so that a row's part is (gamma z / u)^2
below the largest it could be), costs far below one, a slack box, and one outlying
cost that is never taken.  b is 0, so nothing hides the objective in g.  The bound is the
one of the other objective tests; repeated evaluations give the same bits."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DEGREES = [1, 2, 5, 9, 24, 33, 59, 64, 70, 150]


def instance(I, J=200, c_scale=1.0, outlier=0.0, bf16=False):
    rng = np.random.default_rng(I)
    deg = rng.choice(DEGREES, size=I, p=[0.25, 0.25, 0.2, 0.1, 0.1, 0.05, 0.02, 0.01, 0.01, 0.01])
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = (-c_scale * rng.lognormal(0, 0.5, rp[-1])).astype(np.float32)
    if outlier:
        c[len(c) // 2] = outlier
    a = rng.uniform(0.5, 1.5, rp[-1]).astype(np.float32)
    return synth.Instance(rp, col, c, a, np.zeros(J), J)


def check(dlm_lib, inst, kind, z, gamma, lam_scale, bf16):
    p = oracle_problem(inst, kind, z, bf16)
    lam = (lam_scale * np.random.default_rng(1).uniform(0, 0.4, inst.J)).astype(np.float32)
    ref = oracle.sweep(p, lam.astype(np.float64), gamma)
    bound = 2e-6 * (abs(ref["g"]) + abs(ref["obj"]))
    s = dlm_lib.Solver(*to_device(inst, torch, bf16), inst.J, kind=kind, z=z, bf16=bf16)
    got = [s.calculate(torch.from_numpy(lam).cuda(), gamma)[0] for _ in range(4)]
    assert abs(got[0] - ref["g"]) <= bound, (got[0], ref["g"])
    s.set_schedule(gamma)
    s.set_lambda(torch.from_numpy(lam).cuda())
    got.append(s.stats().dual_obj)
    assert len(set(got)) == 1, got
    s.close()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("kind", [oracle.SIMPLEX_LE, oracle.BOX])
@pytest.mark.parametrize("I", [40, 20_000])
@pytest.mark.parametrize("ratio", [1e5, 1e7, 1e9])
def test_ridge_far_above_the_costs(dlm_lib, ratio, I, kind, bf16):
    check(dlm_lib, instance(I), kind, 1.0, ratio, 1.0, bf16)


def test_small_costs_and_a_slack_box(dlm_lib):
    check(dlm_lib, instance(5_000, c_scale=1e-6), oracle.SIMPLEX_LE, 1.0, 10.0, 1e-6, False)
    check(dlm_lib, instance(5_000), oracle.BOX, 1e6, 10.0, 1.0, False)


@pytest.mark.parametrize("kind", [oracle.SIMPLEX_LE, oracle.SIMPLEX_EQ, oracle.BOX])
def test_one_outlying_cost(dlm_lib, kind):
    check(dlm_lib, instance(20_000, outlier=1e13), kind, 1.0, 1e-2, 1.0, False)
