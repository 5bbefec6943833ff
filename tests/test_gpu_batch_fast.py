"""The persistent batched kernel on the specialised FP32 passes: every size it
serves, alone and mixed, against the plans' own solves; its bounded wait."""
import numpy as np
import pytest

import fsp_inputs as I
from conftest import f32_gate, to_dev

pytestmark = pytest.mark.gpu
SIZES = [32, 48, 64, 96, 128, 160, 192, 256]


@pytest.mark.parametrize("Ns", [[N] for N in SIZES] + [SIZES, [64, 32, 32, 160, 48, 96, 32]])
def test_against_single_solves(fsp, Ns):
    import torch
    plans = [fsp.Plan(N, 1.0, "vg_dct", "f32") for N in Ns]
    assert all(p.fast_path for p in plans)
    rhos = [to_dev(I.random_field(N, seed=i), "f32") for i, N in enumerate(Ns)]
    phis = [torch.full_like(r, float("nan")) for r in rhos]
    b = fsp.Batch(plans, rhos, phis)
    for rep in range(2):
        b.launch()
        assert b.wait() == fsp.FSP_OK
        for p, r, f in zip(plans, rhos, phis):
            a = p.solve(r)
            if p.N in (48, 64, 256):  # other schedules in the solve's own launches
                assert float((a - f).abs().max()) <= 2 * f32_gate(p.N) * float(a.abs().max())
            else:
                assert torch.equal(a, f), p.N
            f.fill_(float("nan"))
        for r in rhos:
            r.mul_(-0.5)
    b.close()


def test_timeout(fsp):
    import torch
    plans = [fsp.Plan(N, 1.0, "he", "f32") for N in (32, 96)]
    rhos = [to_dev(I.gaussian_mixture(N), "f32") for N in (32, 96)]
    phis = [torch.zeros_like(r) for r in rhos]
    b = fsp.Batch(plans, rhos, phis)
    b.set_timeout(50.0)
    b.inject_stall()
    b.launch()
    assert b.wait() == fsp.FSP_ETIMEOUT
    b.close()
    b = fsp.Batch(plans, rhos, phis)
    b.launch()
    assert b.wait() == fsp.FSP_OK
    assert torch.equal(phis[0], plans[0].solve(rhos[0]))
    b.close()
