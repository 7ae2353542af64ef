"""The certificate sweep's objective is summed in fixed point at a scale chosen
from gamma and the bounds of the data, in FP64 where no normal float is that
scale.  Scaling c, lam and gamma by a power of two scales g by it and leaves x
alone, so one oracle value serves for magnitudes on each side of the range, for
gammas far above and below the schedule's, and for one warp's worth of rows
and many."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind,z", [(oracle.SIMPLEX_LE, 1.0), (oracle.SIMPLEX_EQ, 0.7), (oracle.BOX, 0.6)])
@pytest.mark.parametrize("I", [9, 6000])
def test_objective_at_any_scale(dlm_lib, kind, z, I):
    J = 200
    rng = np.random.default_rng(I)
    deg = rng.integers(1, 60, size=I)
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = -rng.lognormal(0, 0.5, rp[-1]).astype(np.float32)
    a = rng.uniform(0.5, 1.5, rp[-1]).astype(np.float32)
    b = 0.05 * np.bincount(col, weights=a, minlength=J) + 0.1
    lam = rng.uniform(0, 1.0, J).astype(np.float32)
    p = oracle_problem(synth.Instance(rp, col, c, a, b, J), kind, z)
    for scale in (2.0 ** -80, 1.0, 2.0 ** 30):
        inst = synth.Instance(rp, col, (c * np.float32(scale)).astype(np.float32), a, b, J)
        s = dlm_lib.Solver(*to_device(inst, torch, False), J, kind=kind, z=z)
        for gamma in (1e3, 1e-2, 1e-5):
            ref = oracle.sweep(p, lam.astype(np.float64), gamma)
            g, _, _ = s.calculate(torch.from_numpy(lam * np.float32(scale)).cuda(), gamma * scale)
            assert abs(g / scale - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"])), (scale, gamma)
        s.close()
