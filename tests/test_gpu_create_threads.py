"""Handles of different item counts created by two host threads at the same time:
the set-up kernels' shared memory differs, and neither thread's creation may fail
or change the other's handle."""
import threading

import numpy as np
import pytest

import synth
from gpu_cases import to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def instance(J, seed):
    rng = np.random.default_rng(seed)
    I = 64
    rp = 5 * np.arange(I + 1, dtype=np.int64)
    col = np.concatenate([rng.choice(J, size=5, replace=False) for _ in range(I)]).astype(np.int32)
    c = -rng.uniform(0.1, 1, 5 * I).astype(np.float32)
    a = rng.uniform(0.5, 1.5, 5 * I).astype(np.float32)
    return synth.Instance(rp, col, c, a, 0.05 * np.bincount(col, weights=a, minlength=J), J)


def test_two_threads_create_handles(dlm_lib):
    insts = [instance(60, 1), instance(18_000, 2)]
    arrays = [to_device(i, torch) for i in insts]
    streams = [torch.cuda.Stream() for _ in insts]
    torch.cuda.synchronize()

    def once(k):
        s = dlm_lib.Solver(*arrays[k], insts[k].J, stream=streams[k])
        s.set_schedule(1e-2)
        s.step(3)
        lam = np.empty(insts[k].J, np.float32)
        dlm_lib.dlm_get_lambda(s.h, lam, dlm_lib.DLM_MEM_HOST)
        s.close()
        return lam

    want = [once(0), once(1)]
    errors = []

    def work(k):
        try:
            for _ in range(400):
                assert np.array_equal(once(k), want[k])
        except BaseException as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
