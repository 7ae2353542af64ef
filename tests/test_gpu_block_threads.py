"""block_threads: the launched sweeps have the CTA size that the options name,
on an instance small enough that the default takes fewer, and the iterate does
not depend on it (nor on whether the launches are chained)."""
import json

import numpy as np
import pytest

import synth
from gpu_cases import to_device

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def sweep_blocks(run, path):
    from torch.profiler import ProfilerActivity, profile

    for _ in range(3):  # (a process's first session may start too late to see a launch)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            torch.zeros(1, device="cuda")
            run()
            torch.cuda.synchronize()
        prof.export_chrome_trace(str(path))
        kernels = [e for e in json.loads(path.read_text())["traceEvents"] if e.get("cat") == "kernel"]
        if kernels:
            return {e["args"]["block"][0] for e in kernels if "sweep" in e["name"]}
    pytest.skip("the profiler shows no kernels here")


def solver(dlm_lib, inst, **opt):
    s = dlm_lib.Solver(*to_device(inst, torch), inst.J)
    s.set_schedule(1e-1, 1e-3, 0.3, 10)
    s.set_options(precondition=True, **opt)
    return s


def test_block_threads_are_those_asked_for(dlm_lib, tmp_path):
    inst = synth.generate(synth.recipe_tiny())
    lam = {}
    for threads in (0, 512, 1024):
        s = solver(dlm_lib, inst, block_threads=threads)
        got = sweep_blocks(lambda: s.step(3), tmp_path / f"{threads}.json")
        assert got == {threads} if threads else max(got) < 1024, (threads, got)
        s.set_schedule(1e-1, 1e-3, 0.3, 10)  # from the start again
        s.set_lambda(torch.zeros(inst.J, device="cuda"))
        s.step(60)
        lam[threads] = s.get_state()[0].cpu().numpy()
        s.close()
    s = solver(dlm_lib, inst)  # launched one by one, not chained
    s.step_timed(60)
    lam["timed"] = s.get_state()[0].cpu().numpy()
    s.close()
    for v in lam.values():
        assert np.array_equal(v.view(np.uint64), lam[1024].view(np.uint64))


def test_autotune_reports_what_it_runs(dlm_lib, tmp_path):
    inst = synth.generate(synth.recipe_tiny())
    s = solver(dlm_lib, inst)
    chosen, ms = s.autotune(2)
    got = sweep_blocks(lambda: s.step(3), tmp_path / "tuned.json")
    assert ms > 0 and got == {chosen.block_threads}, (chosen.block_threads, got)
    s.close()
