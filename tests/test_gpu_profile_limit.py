"""The longest lattice along rho that the output interpolation's profiles fit
in shared memory: nine time pieces of which one block's profiles and the
kernel's own arrays (448 bytes with four taps, 512 with six) fill the opt-in
limit to within 32 bytes. Such a plan is made and its two transforms are each
other's transpose to the parity bound of one transform."""
import ctypes

import pytest
import torch

from parity import PARITY_TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07651_gb300 as hr
    return hr


def _sigma_filling(room, d, L):
    """Oversampling whose nine profiles take (room - 32, room] bytes (host-only geometry)."""
    from paper_1604_07651_gb300 import _lib
    lo, hi = 6.0, 16.0
    for _ in range(40):
        d.sigma = 0.5 * (lo + hi)
        n = ctypes.c_int(0)
        infos = (_lib.RadonPieceInfo * 16)()
        _lib.check(L.radon_geometry(ctypes.byref(d), ctypes.byref(n), infos, 16))
        need = n.value * max(infos[i].Nrho for i in range(n.value)) * 4
        if room - 32 < need <= room:
            assert n.value == 9
            return d.sigma
        lo, hi = (d.sigma, hi) if need <= room - 32 else (lo, d.sigma)
    raise AssertionError("no geometry in the margin")


@pytest.mark.parametrize("order,arrays", [(3, 448), (5, 512)])
def test_longest_profiles_are_taken(hr, order, arrays):
    from paper_1604_07651_gb300 import _lib
    L = _lib.load()
    Nt, Nx, Nq = 512, 448, 16
    ts = tuple(0.7 / 1.6 ** k for k in range(8))[::-1]
    d = _lib.RadonDesc()
    _lib.check(L.radon_desc_init(ctypes.byref(d), Nt, Nx, Nt, Nq, 2.0 / (Nt - 1), 2.0 / (Nx - 1), 0.0, 3.0))
    d.n_tsplit, d.spline_order = len(ts), order
    for i, v in enumerate(ts):
        d.tsplit[i] = v
    room = torch.cuda.get_device_properties(0).shared_memory_per_block_optin - arrays
    plan = hr.Plan(Nt, Nx, Nt, Nq, 2.0 / (Nt - 1), 2.0 / (Nx - 1), 0.0, 3.0, sigma=_sigma_filling(room, d, L), tsplit=ts,
                   spline_order=order)
    gen = torch.Generator(device="cuda").manual_seed(17)
    f = torch.randn((Nx, Nt), device="cuda", generator=gen)
    g = torch.randn((Nq, Nt), device="cuda", generator=gen)
    Rf, Rtg = plan.forward(f).double(), plan.adjoint(g).double()
    f, g = f.double(), g.double()
    bound = PARITY_TOL * float(Rf.norm() * g.norm() + f.norm() * Rtg.norm())
    assert abs(float((Rf * g).sum() - (f * Rtg).sum())) <= bound
    plan.close()
