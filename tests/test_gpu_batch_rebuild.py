"""Batches of different sizes alive at the same time, rebuilt in turn."""
import pytest

import fsp_inputs as I
from conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,Ns", [("f32", [[256, 160], [32], [96, 48]]), ("f64", [[75, 128], [16], [50]])])
def test_live_batches_of_different_sizes(fsp, dtype, Ns):
    import torch
    batches = []
    for k, ns in enumerate(Ns):
        plans = [fsp.Plan(N, 1.0, "he", dtype) for N in ns]
        rhos = [to_dev(I.random_field(N, seed=N), dtype) for N in ns]
        phis = [torch.zeros_like(r) for r in rhos]
        b = fsp.Batch(plans, rhos, phis)
        b.launch()
        assert b.wait() == fsp.FSP_OK
        batches.append((b, phis, [f.clone() for f in phis]))
    for b, phis, want in batches:
        for f in phis:
            f.zero_()
        b.set_timeout(900.0)
        b.launch()
        assert b.wait() == fsp.FSP_OK
        assert all(torch.equal(f, w) for f, w in zip(phis, want))
    for b, _, _ in batches:
        b.close()
