"""radon_fwd_noalloc at the limit of its static work area: the bytes that a
plan needs are those of its buffers without row padding and with the gridding
cut into runs of eight samples, whatever layout and cut the plan uses. Plans
within the limit are taken and give radon_fwd's result (on a second call too,
over the first one's leftovers), plans above it are refused."""
import ctypes

import pytest
import torch

import synth
from parity import assert_parity

pytestmark = pytest.mark.gpu

UNSUPPORTED = 4


@pytest.fixture(scope="module")
def hr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07651_gb300 as hr
    return hr


def _call(hr, plan, f, g):
    from paper_1604_07651_gb300 import _lib
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    return _lib.load().radon_fwd_noalloc(plan._handle, ctypes.c_void_p(f.data_ptr()), ctypes.c_void_p(g.data_ptr()), stream)


def _plan(hr, geo, **kw):
    return hr.Plan(geo.Nt, geo.Nx, geo.Ntau, geo.Nq, geo.dt, geo.dx, geo.qmin, geo.qmax, **kw)


@pytest.mark.parametrize("Nt,Nx,kw", [
    (600, 600, dict(n_qsplit=5)),                    # 28.2 MiB; 38.4 with runs of four samples
    (1024, 256, dict(n_qsplit=8)),                   # 24.6 MiB; 36.3
    (600, 600, dict(n_qsplit=3, sigma=1.783)),       # 2560 bytes below the limit: the row padding alone exceeds it
])
def test_plans_within_the_limit_are_taken(hr, Nt, Nx, kw):
    geo = synth.Geometry(Nt, Nx, Nt, Nx, 2.0 / (Nt - 1), 2.0 / (Nx - 1), 0.2, 0.7)
    plan = _plan(hr, geo, **kw)
    for tag in (61, 62):
        f = torch.tensor(synth.band_limited_gather(geo, tag, n_events=6, nu=10.0), dtype=torch.float32, device="cuda")
        want = plan.forward(f)
        g = torch.full_like(want, float("nan"))
        assert _call(hr, plan, f, g) == 0
        assert_parity(g.double().cpu().numpy(), want.double().cpu().numpy(), what=f"no-alloc call {tag}")
    plan.close()


def test_plan_above_the_limit_is_refused(hr):
    from paper_1604_07651_gb300 import _lib
    geo = synth.Geometry(600, 600, 600, 600, 2.0 / 599, 2.0 / 599, 0.2, 0.7)
    plan = _plan(hr, geo, n_qsplit=3, sigma=1.7842)  # 256 bytes above
    f = torch.zeros((600, 600), device="cuda")
    assert _call(hr, plan, f, torch.zeros_like(f)) == UNSUPPORTED
    assert "33554688 bytes" in _lib.load().radon_last_error().decode()
    plan.close()
