"""Plan buffers and graph captures: a plan is made on one thread while another
thread captures a graph; neither disturbs the other."""
import threading

import pytest
import torch

import paper_2405_02603_gb300 as fsp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo,N", [("vg_dct", 32), ("he", 45)])
def test_plan_made_during_another_threads_capture(algo, N):
    rho = torch.randn(N, N, N, dtype=torch.float64, device="cuda")
    plan = fsp.Plan(N, 1.0, algo, "f64")
    want = plan.solve(rho)
    out = torch.zeros_like(rho)
    made, errors, side = [], [], torch.cuda.Stream()
    torch.cuda.synchronize()

    def make():
        try:
            with torch.cuda.stream(side):
                made.append(fsp.Plan(N, 1.0, algo, "f64"))
        except Exception as e:  # noqa: BLE001 -- reported below
            errors.append(e)

    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(st):
        g.capture_begin(capture_error_mode="thread_local")
        try:
            plan.solve_into(rho, out)
            t = threading.Thread(target=make)
            t.start()
            t.join()
        finally:
            g.capture_end()
    assert not errors, errors
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    assert torch.equal(made[0].solve(rho), want)
    made[0].close()
    plan.close()
