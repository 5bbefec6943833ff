"""Memory that the library keeps of destroyed plans goes back on request."""
import pytest

pytestmark = pytest.mark.gpu


def test_trim(fsp):
    import torch
    fsp.memory_trim()
    before = torch.cuda.mem_get_info()[0]
    p = fsp.Plan(96, 1.0, "vg_dct", "f64")  # 60 MB of workspace and spectrum, 100 MB while it is made
    rho = torch.randn(96, 96, 96, dtype=torch.float64, device="cuda")
    want = p.solve(rho)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    fsp.memory_trim()  # the live plan stays
    assert torch.equal(p.solve(rho), want)
    p.close()
    kept = torch.cuda.mem_get_info()[0]
    fsp.memory_trim()
    after = torch.cuda.mem_get_info()[0]
    assert held >= p_bytes() and after - kept >= p_bytes()


def p_bytes():
    return 3 * 96 * 96 * 112 * 16  # W1 and W2, rows of 97 rounded up to 112
