"""A handle on a stream of its own that does not synchronize with the default
one: what a call leaves behind is in order on that stream, also while the default
stream is busy."""
import numpy as np
import pytest

import synth
from gpu_cases import to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def state(s):
    lam, y, _ = s.get_state()
    return lam.cpu().numpy(), y.cpu().numpy()


def run(dlm_lib, arrays, J, users, stream, busy):
    s = dlm_lib.Solver(*arrays, J, stream=stream)
    s.set_schedule(1e-2)
    s.set_options(precondition=True)
    s.set_count_limit(0.1 * users)
    s.step(30)
    lam = np.empty(J + 1, np.float32)
    dlm_lib.dlm_get_lambda(s.h, lam, dlm_lib.DLM_MEM_HOST)
    assert lam[J] > 0  # the count binds
    if busy:
        torch.cuda._sleep(400_000_000)  # some 0.2 s of the default stream
    s.set_count_limit(0.2 * users)
    after = np.empty(J + 1, np.float32)
    dlm_lib.dlm_get_lambda(s.h, after, dlm_lib.DLM_MEM_HOST)
    s.step(20)
    torch.cuda.synchronize()
    s.step(1)
    torch.cuda.synchronize()
    out = after, *state(s)
    s.close()
    return out


def test_count_limit_is_in_order_on_a_side_stream(dlm_lib):
    inst = synth.generate(synth.recipe_tiny())
    arrays = to_device(inst, torch)
    torch.cuda.synchronize()
    want = run(dlm_lib, arrays, inst.J, inst.I, None, False)
    got = run(dlm_lib, arrays, inst.J, inst.I, torch.cuda.Stream(), True)
    assert want[0][inst.J] == 0.0 and got[0][inst.J] == 0.0
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
