"""Every FFT schedule that a plan can produce, against the FP64 log-polar
oracle: lengths of two, three and four passes (16 R0, the radix-2, 4 and 8
middle passes, 256 R0, 4096, 5120, 6144) and those that are no multiple of 16,
with the padding below and above half of the row, bands of one, two and three
pairs of rows, cubic and quintic. Small gathers found on the host with
radon_geometry, whose lattices take these lengths together; the bounds are
those of tests/parity.py."""
import numpy as np
import pytest
import torch

import synth
from oracle.logpolar import Desc, LogPolar
from parity import assert_parity

pytestmark = pytest.mark.gpu

# Nt = Ntau, Nx = Nq, T (s), X (km), qmax, sigma, omega_c, B-spline degree
GEOMETRIES = [
    (24, 12, 0.5, 2.4, 0.7, 3.0, 0.25, 3),       # lengths below 32: 16, 18, 20, 24, 36
    (200, 8, 0.5, 2.4, 0.7, 1.25, 0.25, 3),
    (700, 8, 0.5, 1.0, 0.7, 1.25, 0.4, 3),
    (700, 8, 4.0, 1.0, 0.7, 1.25, 0.4, 5),
    (96, 8, 0.5, 0.3, 0.7, 1.25, 0.4, 3),
    (48, 8, 0.5, 2.4, 0.7, 2.0, 0.4, 3),
    (512, 8, 4.0, 1.0, 0.7, 2.5, 0.35, 3),       # rows (5, 4, 16)
    (700, 8, 2.0, 0.6, 0.7, 3.0, 0.25, 3),       # rows (9, 2, 16)
    (512, 128, 0.5, 2.4, 0.7, 2.5, 0.25, 3),     # columns (9, 8, 16)
    (700, 32, 4.0, 1.6, 0.7, 3.0, 0.35, 5),      # rows (9, 4, 16)
    (700, 64, 4.0, 2.4, 0.7, 3.0, 0.4, 5),       # rows (5, 8, 16)
    (200, 128, 0.5, 2.4, 0.7, 3.0, 0.35, 3),     # columns (6, 16, 16)
    (200, 200, 0.5, 1.0, 0.7, 1.5, 0.25, 3),     # rows (16, 16), padded by half
    (200, 200, 0.5, 1.0, 0.7, 3.0, 0.4, 5),      # rows (2, 16, 16)
    (16, 1024, 4.0, 2.4, 0.7, 1.1, 0.4, 3),      # columns 512, 256, 144
    (16, 512, 1.0, 0.3, 0.7, 1.25, 0.25, 3),     # 768
    (16, 1500, 4.0, 2.4, 0.5, 1.1, 0.35, 3),     # 1024, 384
    (16, 1500, 4.0, 1.6, 0.7, 1.5, 0.4, 3),      # 1280, 576
    (16, 3000, 1.0, 0.3, 0.7, 1.5, 0.25, 3),     # 2304, 1024, 640
    (32, 3000, 1.0, 0.3, 0.7, 1.1, 0.25, 5),     # 3072, 1536
    (16, 3000, 4.0, 1.0, 0.5, 1.1, 0.35, 3),     # 4096, 2048, 1152
    (16, 1500, 2.0, 0.6, 0.7, 3.0, 0.35, 3),     # 5120: four passes
    (32, 3000, 4.0, 1.6, 0.5, 2.0, 0.25, 3),     # 6144: four passes
    (3000, 8, 4.0, 0.6, 0.7, 1.1, 0.35, 3),      # rows 64, 192, 512
    (3000, 12, 2.0, 0.3, 0.5, 1.1, 0.25, 3),     # 144, 768
    (4096, 8, 2.0, 0.3, 0.5, 2.0, 0.35, 5),      # 1280
    (4096, 8, 4.0, 0.3, 0.5, 3.0, 0.25, 3),      # 1024, 2048, 3072
]


@pytest.fixture(scope="module")
def hr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07651_gb300 as hr
    return hr


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("i", range(len(GEOMETRIES)))
def test_fft_schedules_match_oracle(hr, i):
    Nt, Nx, T, X, qmax, sigma, omega_c, order = GEOMETRIES[i]
    geo = synth.Geometry(Nt, Nx, Nt, Nx, T / (Nt - 1), X / (Nx - 1), 0.2, qmax)
    args = (geo.Nt, geo.Nx, geo.Ntau, geo.Nq, geo.dt, geo.dx, geo.qmin, geo.qmax)
    plan = hr.Plan(*args, sigma=sigma, omega_c=omega_c, tsplit=(0.25, 0.5), spline_order=order,
                   rows_per_band=(2, 4, 6)[i % 3])
    lp = LogPolar(Desc(*args, sigma=sigma, omega_c=omega_c, tsplits=(0.25, 0.5), order=order))
    rng = np.random.default_rng(i)
    f, g = rng.standard_normal((Nx, Nt)), rng.standard_normal((Nx, Nt))
    f, g = f.astype(np.float32), g.astype(np.float32)
    assert_parity(plan.forward(_cuda(f)).cpu().numpy(), lp.forward(f.astype(np.float64)), what=f"{GEOMETRIES[i]} forward")
    assert_parity(plan.adjoint(_cuda(g)).cpu().numpy(), lp.adjoint(g.astype(np.float64)), what=f"{GEOMETRIES[i]} adjoint")
    plan.close()


@pytest.mark.parametrize("size", [(256, 64), (501, 77), (768, 512)])
def test_back_to_back_passes_and_stale_lattices(hr, size):
    """Small transforms start while their predecessor drains and write every
    lattice cell instead of clearing first: passes enqueued without waiting,
    with a NaN gather among them, give the bits of the first pass."""
    Nt, Nx = size
    plan = hr.Plan(Nt, Nx, Nt, Nx, 0.004, 0.0125, 0.2, 0.7, rows_per_band=3)
    gen = torch.Generator(device="cuda").manual_seed(5)
    fs = [torch.randn((Nx, Nt), device="cuda", generator=gen) for _ in range(3)]
    fs[1][Nx // 2] = float("nan")
    fs[2][:, : Nt // 2] = 0.0                       # units and tiles without a non-zero sample
    want = []
    for f in (fs[0], fs[2]):
        g = plan.forward(f)
        torch.cuda.synchronize()
        a = plan.adjoint(g)
        torch.cuda.synchronize()
        want.append((g.clone(), a.clone()))
    got = []
    for _ in range(40):
        for k in (0, 1, 2):
            g = plan.forward(fs[k])
            a = plan.adjoint(g)
            if k != 1:
                got.append((k // 2, g, a))
    torch.cuda.synchronize()
    for k, g, a in got:
        assert torch.equal(g, want[k][0]) and torch.equal(a, want[k][1])
    plan.close()


@pytest.mark.parametrize("ntau", [256, 257, 258, 263])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_buffers_off_16_bytes(hr, ntau, offset):
    """The profiles read eight outputs at a time where they are aligned: odd
    image lengths and buffers that start off a 16-byte boundary give the bits
    of an aligned copy, in both directions."""
    plan = hr.Plan(257, 48, ntau, 33, 0.004, 0.0125, 0.2, 0.7, rows_per_band=3)
    buf = torch.randn(48 * 257 + 4, device="cuda", generator=torch.Generator(device="cuda").manual_seed(6))
    view = lambda b, *shape: b[offset:offset + shape[0] * shape[1]].view(*shape)
    f, g = view(buf, 48, 257), view(buf, 33, ntau)
    assert torch.equal(plan.adjoint(g, out=view(torch.empty_like(buf), 48, 257)), plan.adjoint(g.clone()))
    assert torch.equal(plan.forward(f, out=view(torch.empty_like(buf), 33, ntau)), plan.forward(f.clone()))
    plan.close()


@pytest.mark.parametrize("order", [3, 5])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("gathers", [[(301, 64), (97, 33)], [(1501, 201), (902, 150)]])
def test_batch_gridding_equals_single_plans(hr, gathers, dtype, order):
    """A batch's gridding copies its position entries through shared memory
    and takes chunks of four samples below about 400 000 samples, eight above;
    single plans of these gathers take four and read their own entries. Both
    round every contribution to 2^-29 or less of the cell bound (1e-6, as the
    batches' own tests)."""
    desc = [dict(Nt=nt, Nx=nx, Ntau=nt - 3, Nq=nx, dt=0.004, dx=0.025, qmin=0.2, qmax=0.7, spline_order=order,
                 rows_per_band=4) for nt, nx in gathers]
    gen = torch.Generator(device="cuda").manual_seed(9)
    fs = [torch.randn((nx, nt), device="cuda", generator=gen).to(dtype) for nt, nx in gathers]
    batch = hr.Batch(desc)
    out = batch.unpack_images(batch.forward(batch.pack(fs, dtype=dtype)))
    for d, f, g in zip(desc, fs, out):
        plan = hr.Plan(**d)
        want = plan.forward(f.float())
        assert float((g - want).norm()) <= 1e-6 * float(want.norm())
        plan.close()
