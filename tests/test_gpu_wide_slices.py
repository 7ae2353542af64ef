"""The one-family sweep's wide slices, taken in quarters by four lanes a row.
Small instances whose widest rows lie around the width from which slices are
cut (64 edges) and well above it, tails of every length, values tied across the
four lanes' shares, and ridges at which rows have one to dozens of active
edges: against the FP64 oracle, and bit for bit across mappings and batches."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, to_device, x_error_report

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DEGREES = [1, 3, 4, 5, 11, 25, 33, 62, 63, 64, 65, 66, 67, 68, 127, 130, 257, 499, 500]


def instance(seed, I=1500, J=600, ties=False):
    rng = np.random.default_rng(seed)
    deg = rng.choice(DEGREES, size=I)
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = -rng.choice([0.5, 0.75, 1.0], size=rp[-1]) if ties else -rng.lognormal(0, 0.5, rp[-1])
    a = np.ones(rp[-1]) if ties else rng.uniform(0.5, 1.5, rp[-1])
    b = 0.05 * np.bincount(col, weights=a, minlength=J)
    return synth.Instance(rp, col, c.astype(np.float32), a.astype(np.float32), b, J)


@pytest.mark.parametrize("kind,z,bf16", [(oracle.SIMPLEX_LE, 1.0, False), (oracle.SIMPLEX_LE, 1.0, True),
                                         (oracle.SIMPLEX_EQ, 0.7, False), (oracle.BOX, 0.6, True)])
def test_wide_slices_match_the_oracle(dlm_lib, kind, z, bf16):
    inst = instance(11)
    s = dlm_lib.Solver(*to_device(inst, torch, bf16), inst.J, kind=kind, z=z, bf16=bf16)
    p = oracle_problem(inst, kind, z, bf16)
    rng = np.random.default_rng(3)
    for gamma in (1e-1, 1e-2, 1e-3):
        lam32 = rng.uniform(0, 1.0, inst.J).astype(np.float32)
        g, grad, x = s.calculate(torch.from_numpy(lam32).cuda(), gamma)
        ref = oracle.sweep(p, lam32.astype(np.float64), gamma)
        dx, tol = x_error_report(x.cpu().numpy(), ref["x"], p, lam32.astype(np.float64), gamma)
        assert (dx <= tol).all(), dx.max()
        assert abs(g - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"]))
    s.set_schedule(1e-1, 1e-3, 0.3, 15)
    s.set_options(precondition=True)
    s.step(90)
    ref = oracle.fista(p, 90, 1e-1, 1e-3, 0.3, 15, precondition=True, trajectory=False)["lam"]
    err = np.abs(s.lam().cpu().numpy().astype(np.float64) - ref).max()
    assert err <= 1e-5 * max(np.abs(ref).max(), 1e-6), err
    s.close()


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("kind", [oracle.SIMPLEX_LE, oracle.SIMPLEX_EQ, oracle.BOX])
def test_mappings_and_batches_agree_bit_for_bit(dlm_lib, kind, ties):
    inst = instance(12, ties=ties)
    arrays = to_device(inst, torch)

    def solver(**opt):
        s = dlm_lib.Solver(*arrays, inst.J, kind=kind)
        s.set_schedule(1e-1, 1e-3, 0.3, 10)
        s.set_options(precondition=True, coop_max=1, **opt)
        return s

    def state(s):
        lam, y, _ = s.get_state()
        out = lam.cpu().numpy(), y.cpu().numpy(), s.trajectory(0, 60)
        s.close()
        return out

    first = solver()
    first.step(60)
    want = state(first)
    for opt in ({"mapping": 2}, {"mapping": 3}, {"block_threads": 512}):
        s = solver(**opt)
        s.step(60)
        for got, ref in zip(state(s), want):
            assert np.array_equal(got.view(np.uint64), ref.view(np.uint64)), opt
    members = [solver(), solver()]
    for mapping in (1, 3):
        for m in members:
            m.set_schedule(1e-1, 1e-3, 0.3, 10)
            m.set_lambda(torch.zeros(inst.J, dtype=torch.float32, device="cuda"))
        bt = dlm_lib.Batch(members)
        bt.set_options(mapping=mapping, coop_max=1)
        bt.step(60)
        for m in members:
            lam, y, _ = m.get_state()
            assert np.array_equal(lam.cpu().numpy().view(np.uint64), want[0].view(np.uint64))
            assert np.array_equal(m.trajectory(0, 60).view(np.uint64), want[2].view(np.uint64))
        bt.close()
    for m in members:
        m.close()
