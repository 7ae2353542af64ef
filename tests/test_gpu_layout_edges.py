"""The slice layout at the edges of its set-up kernels: rows around the 32
edges that one pass of a warp reads and around the four-edge groups, ties in
cost at the lead edges' boundary, fewer rows than a slice, arrays that start
off a 16-byte boundary, item counts on each side of the shared memory that
holds the item sums (both sums, one, none), and items of degree under 64
(their fixed-point terms exceed 2^55).  x comes back in the caller's order and
the preconditioned iterate depends on every item's sum a^2, so both are
checked against the oracle; a repeated item is found in short and long rows."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, x_error_report
from test_gpu_static_rows import off_boundary

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DEGREES = [0, 1, 2, 3, 4, 5, 7, 8, 9, 28, 31, 32, 33, 34, 35, 36, 37, 60, 63, 64, 65, 67, 130]


def instance(J, I, seed, negative=False):
    rng = np.random.default_rng(seed)
    deg = rng.choice(DEGREES, size=I)
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    nnz = int(rp[-1])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = -rng.choice([0.25, 0.5, 1.0, 1.5], size=nnz)  # ties among a row's lowest costs
    c = np.where(rng.uniform(size=nnz) < 0.7, -rng.lognormal(0, 0.5, nnz), c)
    c[rng.uniform(size=nnz) < 0.02] = 0.0
    c[rng.uniform(size=nnz) < 0.02] = -0.0
    a = rng.uniform(0.5, 1.5, nnz)
    b = 0.05 * np.bincount(col, weights=a, minlength=J) + 0.1
    return synth.Instance(rp, col, c.astype(np.float32), a.astype(np.float32), b, J)


@pytest.mark.parametrize("J,I,bf16,by", [(140, 3, False, 0), (140, 2000, False, 1), (140, 2000, True, 1),
                                         (140, 2001, True, 0), (9000, 1500, False, 2), (15_000, 1500, True, 3),
                                         (18_900, 1500, False, 0)])
def test_layout_matches_the_oracle(dlm_lib, J, I, bf16, by):
    inst = instance(J, I, 3 + I + J)
    if bf16:
        inst.c = synth.bf16_to_f32(synth.round_bf16(inst.c))
        inst.a = synth.bf16_to_f32(synth.round_bf16(inst.a))
    p = oracle_problem(inst)
    rp = torch.from_numpy(inst.row_ptr).cuda()
    col, c, a = (off_boundary(v, by) for v in (inst.col, inst.c, inst.a))
    if bf16:
        c, a = (off_boundary(synth.round_bf16(v).view(np.int16), by).view(torch.bfloat16) for v in (inst.c, inst.a))
    s = dlm_lib.Solver(rp, col, c, a, torch.from_numpy(inst.b).cuda(), J, bf16=bf16)
    rng = np.random.default_rng(5)
    for gamma in (1e-1, 1e-3):
        lam32 = rng.uniform(0, 1.0, J).astype(np.float32)
        g, grad, x = s.calculate(torch.from_numpy(lam32).cuda(), gamma)
        lam64 = lam32.astype(np.float64)
        ref = oracle.sweep(p, lam64, gamma)
        dx, tol = x_error_report(x.cpu().numpy(), ref["x"], p, lam64, gamma)
        assert (dx <= tol).all(), dx.max()
        assert abs(g - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"]))
    s.set_schedule(1e-2)
    s.set_options(precondition=True)
    s.step(30)
    ref = oracle.fista(p, 30, 1e-2, precondition=True, trajectory=False)["lam"]
    err = np.abs(s.lam().cpu().numpy().astype(np.float64) - ref).max()
    assert err <= 1e-5 * max(np.abs(ref).max(), 1e-6), err
    s.close()


@pytest.mark.parametrize("d", [2, 31, 32, 33, 64, 130, 141])
def test_repeated_items_are_found(dlm_lib, d):
    J = 140
    rng = np.random.default_rng(d)
    rows = [rng.choice(J, size=20, replace=False) for _ in range(50)]
    bad = np.concatenate([rng.choice(J, size=min(d, J) - 1, replace=False), [0] * (d - min(d, J) + 1)])
    bad[-1] = bad[0]
    rows.insert(17, bad)
    rp = np.zeros(len(rows) + 1, np.int64)
    np.cumsum([len(r) for r in rows], out=rp[1:])
    col = np.concatenate(rows).astype(np.int32)
    t = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    c = t(-rng.uniform(0.1, 1, len(col)).astype(np.float32))
    with pytest.raises(dlm_lib.DlmError) as e:
        dlm_lib.Solver(t(rp), t(col), c, -c, t(np.ones(J)), J)
    assert e.value.status == dlm_lib.DLM_ERR_INVALID_ARG and "twice" in str(e.value)
