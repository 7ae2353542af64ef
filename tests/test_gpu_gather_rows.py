"""The layout's gather at the edges of its row batches: 32 rows at a time to one
by width, the longest rows it stages (1,024 edges) and the first past them, widths on each side of a group of four, and ragged last slices.  x comes back
in the caller's order, so every edge's place is checked against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_cases import oracle_problem, x_error_report

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("w", [31, 32, 33, 64, 65, 97, 127, 128, 129, 255, 257, 511, 513, 1021, 1024, 1027])
def test_rows_of_one_width(dlm_lib, w, bf16):
    J, I = 1100, 70  # two whole slices and a ragged one
    rng = np.random.default_rng(w)
    deg = np.where(rng.uniform(size=I) < 0.5, w, rng.integers(1, w + 1, size=I))
    rp = np.zeros(I + 1, np.int64)
    np.cumsum(deg, out=rp[1:])
    nnz = int(rp[-1])
    col = np.concatenate([rng.choice(J, size=d, replace=False) for d in deg]).astype(np.int32)
    c = (-rng.choice([0.25, 0.5, 1.0, 1.5], size=nnz)).astype(np.float32)  # ties at the lead edges' boundary
    a = synth.bf16_to_f32(synth.round_bf16(rng.uniform(0.5, 1.5, nnz).astype(np.float32)))
    b = 0.05 * np.bincount(col, weights=a, minlength=J) + 0.1
    inst = synth.Instance(rp, col, c, a, b, J)
    p = oracle_problem(inst)
    tc, ta = (torch.from_numpy(v).cuda() for v in (c, a))
    if bf16:
        tc, ta = tc.bfloat16(), ta.bfloat16()
    s = dlm_lib.Solver(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), tc, ta, torch.from_numpy(b).cuda(), J,
                       bf16=bf16)
    lam = rng.uniform(0, 1.0, J).astype(np.float32)
    for gamma in (1.0, 1e-2):  # many active edges a row, and few
        g, grad, x = s.calculate(torch.from_numpy(lam).cuda(), gamma)
        ref = oracle.sweep(p, lam.astype(np.float64), gamma)
        dx, tol = x_error_report(x.cpu().numpy(), ref["x"], p, lam.astype(np.float64), gamma)
        assert (dx <= tol).all(), dx.max()
        assert abs(g - ref["g"]) <= 2e-6 * (abs(ref["g"]) + abs(ref["obj"]))
    s.close()
    bad = col.copy()
    at = int(rp[:-1][deg >= 2][-1])  # a repeated item in the last such row
    bad[at + 1] = bad[at]
    with pytest.raises(dlm_lib.DlmError) as e:
        dlm_lib.Solver(torch.from_numpy(rp).cuda(), torch.from_numpy(bad).cuda(), tc, ta, torch.from_numpy(b).cuda(), J,
                       bf16=bf16)
    assert e.value.status == dlm_lib.DLM_ERR_INVALID_ARG and "twice" in str(e.value)
