"""Slices taken in quarters at the default cooperative threshold (their rows'
threshold iteration is then the whole warp's) and under a count constraint: against the
FP64 oracle, and bit for bit across mappings, CTA sizes and batches."""
import numpy as np
import pytest

import oracle
from gpu_cases import oracle_problem, to_device
from test_gpu_wide_slices import instance

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def solver(dlm_lib, inst, kind, limit, **opt):
    s = dlm_lib.Solver(*to_device(inst, torch), inst.J, kind=kind)
    s.set_schedule(1e-1, 1e-3, 0.3, 10)
    if limit:
        s.set_count_limit(limit)
    s.set_options(precondition=True, **opt)
    return s


@pytest.mark.parametrize("limit", [None, 300.0])
@pytest.mark.parametrize("kind", [oracle.SIMPLEX_LE, oracle.SIMPLEX_EQ])
def test_quarters_agree_bit_for_bit(dlm_lib, kind, limit):
    inst = instance(21)

    def state(s, n=60):
        lam, y, _ = s.get_state()
        return lam.cpu().numpy(), y.cpu().numpy(), s.trajectory(0, n)

    s = solver(dlm_lib, inst, kind, limit)
    s.step(60)
    want = state(s)
    dual = s.stats().dual_obj
    assert dual == s.stats().dual_obj
    s.close()
    for opt in ({"mapping": 2}, {"mapping": 3}, {"block_threads": 512}, {"block_threads": 1024}):
        s = solver(dlm_lib, inst, kind, limit, **opt)
        s.step(60)
        for got, ref in zip(state(s), want):
            assert np.array_equal(got.view(np.uint64), ref.view(np.uint64)), opt
        assert abs(s.stats().dual_obj - dual) <= 1e-12 * abs(dual)  # (FP64 parts added in another order)
        s.close()
    members = [solver(dlm_lib, inst, kind, limit) for _ in range(3)]
    bt = dlm_lib.Batch(members)
    bt.step(60)
    for m in members:
        for got, ref in zip(state(m), want):
            assert np.array_equal(got.view(np.uint64), ref.view(np.uint64))
    bt.close()
    for m in members:
        m.close()


@pytest.mark.parametrize("kind", [oracle.SIMPLEX_LE, oracle.SIMPLEX_EQ])
def test_counted_quarters_match_the_oracle(dlm_lib, kind):
    inst = instance(22)
    p = oracle_problem(inst, kind)
    # the count dual acts as one more item in every row: u = -(c + a y) - mu
    mu = 0.3
    s = dlm_lib.Solver(*to_device(inst, torch), inst.J, kind=kind)
    s.set_count_limit(500.0)
    rng = np.random.default_rng(4)
    for gamma in (1e-1, 1e-2, 1e-3):
        y = np.append(rng.uniform(0, 1.0, inst.J), mu).astype(np.float32)
        g, grad, x = s.calculate(torch.from_numpy(y).cuda(), gamma)
        shifted = oracle.Problem(p.row_ptr, p.col, p.c + float(np.float32(mu)), p.a, p.b, p.J, kind, 1.0)
        ref = oracle.sweep(shifted, y[:-1].astype(np.float64), gamma)
        total = ref["x"].sum()
        assert abs(float(grad[inst.J]) - (total - 500.0)) <= 1e-5 * (total + 500.0)
        want = ref["g"] - float(np.float32(mu)) * 500.0
        assert abs(g - want) <= 2e-6 * (abs(want) + abs(ref["obj"]) + mu * total)
    s.close()
