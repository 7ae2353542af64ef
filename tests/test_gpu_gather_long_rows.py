"""The layout's gather of rows longer than a warp stages (1,024 edges), whose slices
a block takes with all of its warps: several such slices, then shorter ones and a ragged end,
widths on each side of a strip and of a group of four.  x comes back in the caller's
order, so every edge's place is checked against the oracle; a repeated item
is found in whichever warp's row it is, near its start or its end."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, x_error_report

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("w", [1025, 1056, 1058, 1279, 1280, 2051, 5000])
def test_long_rows(dlm_lib, w, bf16):
    J = 5200
    rng = np.random.default_rng(w)
    deg = np.concatenate([np.full(33, w), rng.integers(1025, w + 1, size=50), rng.integers(1, 1025, size=70)])
    deg = rng.permutation(deg)
    rp = np.zeros(len(deg) + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    nnz = int(rp[-1])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = (-rng.choice([0.25, 0.5, 1.0, 1.5], size=nnz)).astype(np.float32)  # ties at the lead edges' boundary
    a = synth.bf16_to_f32(synth.round_bf16(rng.uniform(0.5, 1.5, nnz).astype(np.float32)))
    b = 0.05 * np.bincount(col, weights=a, minlength=J) + 0.1
    p = oracle_problem(synth.Instance(rp, col, c, a, b, J))
    t = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    tc, ta = (t(v).bfloat16() if bf16 else t(v) for v in (c, a))
    s = dlm_lib.Solver(t(rp), t(col), tc, ta, t(b), J, bf16=bf16)
    lam = rng.uniform(0, 1.0, J).astype(np.float32)
    for gamma in (1.0, 1e-2):  # many active edges a row, and few
        g, grad, x = s.calculate(t(lam), gamma)
        ref = oracle.sweep(p, lam.astype(np.float64), gamma)
        dx, tol = x_error_report(x.cpu().numpy(), ref["x"], p, lam.astype(np.float64), gamma)
        assert (dx <= tol).all(), dx.max()
        assert abs(g - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"]))
    s.close()
    long = np.nonzero(deg > 1024)[0]
    for row in long[:: max(1, len(long) // 12)]:
        for at in (rp[row], rp[row + 1] - 2):
            bad = col.copy()
            bad[at + 1] = bad[rp[row]] if at > rp[row] else bad[at]
            with pytest.raises(dlm_lib.DlmError) as e:
                dlm_lib.Solver(t(rp), t(bad), tc, ta, t(b), J, bf16=bf16)
            assert e.value.status == dlm_lib.DLM_ERR_INVALID_ARG and "twice" in str(e.value)
