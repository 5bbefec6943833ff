"""FP64 solves in boxes and of sources of any size.  The spectrum scales with the
square of the box side (the field's with the side), the results with it and
with the source; powers of two scale every array exactly, so the reference is
the unit box and source."""
import numpy as np
import pytest

import fsp_inputs as I

pytestmark = pytest.mark.gpu

# 2-norm of the difference of two results, relative.  Each side stores five
# arrays, one rounding of at most 2^-53 each, and holds its transforms' values
# in units that are small against that: 2 * 5 * 2^-53 with the spectrum's own.
TOL = 10 * 2.0 ** -53


def sources(N):
    import torch
    yield torch.from_numpy(I.random_field(N, 2)).cuda()
    one = torch.zeros(N, N, N, dtype=torch.float64, device="cuda")
    one[N // 3, (3 * N) // 8, N // 5] = 1.7
    yield one


def check(got, want):
    err = float((got - want).norm() / want.norm())
    print("rel %.2e = %.2f * 2^-53" % (err, err * 2 ** 53))
    assert err <= TOL


@pytest.mark.parametrize("e", [-150, -45, 40, 66, 150])
@pytest.mark.parametrize("N", [8, 32, 64, 75, 96, 128, 135])
def test_solve(fsp, N, e):
    a, b = fsp.Plan(N, 1.0, "vg_dct", "f64"), fsp.Plan(N, 2.0 ** e, "vg_dct", "f64")
    for rho in sources(N):
        check(b.solve(rho), a.solve(rho) * 2.0 ** (2 * e))


@pytest.mark.parametrize("e", [-95, 105])
@pytest.mark.parametrize("N", [32, 75, 128])
def test_source(fsp, N, e):
    p = fsp.Plan(N, 1.0, "vg_dct", "f64")
    for rho in sources(N):
        check(p.solve(rho * 2.0 ** e), p.solve(rho) * 2.0 ** e)


@pytest.mark.parametrize("n3", [(64, 64, 128), (30, 45, 40)])
def test_box(fsp, n3):
    import torch
    L = [n / 64 for n in n3]
    a, b = fsp.Plan(n3, L, "vg_dct", "f64"), fsp.Plan(n3, [x * 2.0 ** 70 for x in L], "vg_dct", "f64")
    rho = torch.from_numpy(I.random_field3(n3, 4)).cuda()
    check(b.solve(rho), a.solve(rho) * 2.0 ** 140)


@pytest.mark.parametrize("n3", [(64, 64, 64), (75, 75, 75), (64, 64, 128), (30, 45, 40)])
@pytest.mark.parametrize("e", [-120, 120])
def test_field(fsp, n3, e):
    import torch
    L = [n / 64 for n in n3]
    a, b = (fsp.Plan(n3, [x * s for x in L], "vg_dct", "f64") for s in (1.0, 2.0 ** e))
    rho = torch.from_numpy(I.random_field3(n3, 4)).cuda()
    for c, (x, y) in enumerate(zip(a.solve_field(rho, with_phi=True), b.solve_field(rho, with_phi=True))):
        check(y, x * 2.0 ** (2 * e if c == 3 else e))


def test_largest_length(fsp):
    a, b = fsp.Plan(512, 1.0, "vg_dct", "f64"), fsp.Plan(512, 2.0 ** 66, "vg_dct", "f64")
    for rho in sources(512):
        check(b.solve(rho), a.solve(rho) * 2.0 ** 132)


@pytest.mark.parametrize("N", [32, 30])
def test_spectrum_batch_and_slabs(fsp, N):
    """The stored spectrum is the true one, restores the plan bit for bit, and
    serves a batch and the slab form; one of another order is taken as it is."""
    import torch
    L = 2.0 ** -60
    a, b = fsp.Plan(N, 1.0, "vg_dct", "f64"), fsp.Plan(N, L, "vg_dct", "f64")
    S = b.spectrum()
    assert np.max(np.abs(S - a.spectrum() * L ** 2)) <= 16 * 2.0 ** -53 * np.max(S)
    rho = next(sources(N))
    want = b.solve(rho)
    assert torch.equal(fsp.Plan.from_spectrum(N, L, "vg_dct", "f64", S).solve(rho), want)
    check(fsp.Plan.from_spectrum(N, 1.0, "vg_dct", "f64", S * 2.0 ** -200).solve(rho), want * 2.0 ** -200)
    phi = torch.empty_like(rho)
    for form in (0, 1):
        batch = fsp.Batch([b], [rho], [phi.zero_()])
        batch.set_form(form)
        batch.launch()
        assert batch.wait() == fsp.FSP_OK
        check(phi, want)
        batch.close()
    check(fsp.solve_noalloc(torch.from_numpy(S).cuda(), rho, phi), want)
    check(fsp.solve_distributed_local(N, rho, L, "vg_dct", "f64", 3), want)


@pytest.mark.parametrize("N", [32, 30])
def test_largest_sources(fsp, N):
    """What overflows is what overflowed: a source close to the range's end in a
    box whose spectrum is small."""
    import torch
    p = fsp.Plan(N, 2.0 ** -60, "vg_dct", "f64")
    rho = torch.full((N, N, N), 1.0, dtype=torch.float64, device="cuda")
    top = 2.0 ** (1023 - 2 * int(np.ceil(np.log2(N))))  # the second pass holds N^2 of it
    check(p.solve(rho * top) / top, p.solve(rho))  # (the 2-norm of the results overflows)
