"""rows_per_band is a request: desc reports it as asked for, also where the
pairing of rows or shared memory makes the plan run another value, and the
transforms do not depend on it (1e-6, as the other rows-per-band test). Shapes
on both sides of the rounding: few lattice rows (3 and 5 run as 2 and 4), many
(as 4 and 6), and rows so long that shared memory holds two pairs (6 runs as 4)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07651_gb300 as hr
    return hr


@pytest.mark.parametrize("Nt,Nx,Nq,more", [
    (256, 64, 64, {}),
    (1200, 1200, 50, {}),
    (512, 352, 20, dict(sigma=16.0, qmin=0.0, qmax=3.0)),
])
def test_requests_are_reported_and_do_not_change_results(hr, Nt, Nx, Nq, more):
    kw = dict(qmin=0.2, qmax=0.7)
    kw.update(more)
    gen = torch.Generator(device="cuda").manual_seed(3)
    f = torch.randn((Nx, Nt), device="cuda", generator=gen)
    g = torch.randn((Nq, Nt), device="cuda", generator=gen)
    want = None
    for R in (2, 1, 3, 5, 6):
        plan = hr.Plan(Nt=Nt, Nx=Nx, Ntau=Nt, Nq=Nq, dt=2.0 / (Nt - 1), dx=2.0 / (Nx - 1), rows_per_band=R, **kw)
        assert plan.desc.rows_per_band == R
        got = plan.forward(f), plan.adjoint(g)
        want = want or got
        for a, b in zip(got, want):
            assert float((a - b).norm()) <= 1e-6 * float(b.norm()), R
        plan.close()
