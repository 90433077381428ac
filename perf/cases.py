"""What this library is used for, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` makes what a user's program has
in hand (plan or batch, gathers or images on the GPU), ``run`` is one pass
through the public entry points, ``exact`` the same result in 64 bits from
plain torch (the log-polar method of arXiv:1604.07651 step by step, on the
lattices that the descriptor prescribes).

Kinds of pass:
  forward        Plan.forward of one gather
  adjoint        Plan.adjoint of one Radon image
  pair           forward of a gather and adjoint of an image on one plan
  autograd       the differentiable op: forward, then the gradient of <g, w>
  batch_forward  Batch.forward of many gathers of different sizes
  batch_adjoint  Batch.adjoint of their images
  fista          Plan.ista on a gather with missing traces
  demultiple     Plan.demultiple (sparse image, mute, subtraction)
"""
import math

import numpy as np
import torch

import paper_1604_07651_gb300 as hr

QMIN, QMAX = 0.2, 0.7          # s/km, every workload of the repository's tests and benchmark


def _single(name, kind, Nt, Nx, T=2.0, X=2.0, **more):
    """One gather: Nt samples on [0, T] s, Nx offsets on [0, X] km, image of the same size."""
    return {"name": name, "kind": kind, "Nt": Nt, "Nx": Nx, "Ntau": Nt, "Nq": Nx, "T": T, "X": X, "order": 3,
            "rows": 3, "jitter": 0.0, "near": 0.0, **more}


def listed():
    return [
        # a quick look at one small gather (256 samples at 4 ms, 64 offsets): latency and launches count
        _single("forward_256x64", "forward", 256, 64, T=1.02, X=1.6),
        _single("adjoint_256x64", "adjoint", 256, 64, T=1.02, X=1.6),
        # an inversion or training loop in PyTorch on a moderate gather: forward and its gradient
        _single("autograd_512", "autograd", 512, 512),
        # the benchmark gather, each direction by itself (rows per band timed by the plan, as the benchmark asks)
        _single("forward_2048", "forward", 2048, 2048, rows=0),
        _single("adjoint_2048", "adjoint", 2048, 2048, rows=0),
        # the same gather with the quintic B-spline option
        _single("pair_2048_quintic", "pair", 2048, 2048, rows=0, order=5),
        # the largest gather the repository's workloads hold
        _single("pair_4096", "pair", 4096, 4096, rows=0),
        # a field gather: offsets off the grid, a near-offset gap, odd sizes, denser slownesses at qmin
        _single("pair_jittered_1501x233", "pair", 1501, 233, T=3.0, X=2.4, jitter=0.4, near=0.15, Ntau=1407, Nq=301),
        # a survey: many gathers of different sizes, stored in bfloat16 for the forward, float32 images for the adjoint
        {"name": "batch_forward_bf16_128", "kind": "batch_forward", "gathers": 128, "nt_lo": 500, "nt_hi": 3000,
         "nx_lo": 60, "nx_hi": 480, "bf16": True, "order": 3, "rows": 0, "sizes": 4},
        {"name": "batch_adjoint_128", "kind": "batch_adjoint", "gathers": 128, "nt_lo": 500, "nt_hi": 3000,
         "nx_lo": 60, "nx_hi": 480, "bf16": False, "order": 3, "rows": 0, "sizes": 4},
        # trace interpolation: 40 % of the traces missing, 50 FISTA iterations
        _single("fista_1024x256", "fista", 1024, 256, T=2.046, iters=50, missing=0.4),
        # multiple attenuation of a small gather, 30 ISTA iterations
        _single("demultiple_512x128", "demultiple", 512, 128, T=2.044, iters=30),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "adjoint", "adjoint", "pair", "autograd", "batch_forward",
                       "batch_adjoint", "fista", "demultiple"])
    if kind.startswith("batch"):
        nt_lo, nx_lo = _log_int(rng, 200, 800), _log_int(rng, 40, 150)
        return {"kind": kind, "gathers": _log_int(rng, 2, 128), "nt_lo": nt_lo, "nt_hi": nt_lo + rng.randint(100, 2200),
                "nx_lo": nx_lo, "nx_hi": nx_lo + rng.randint(20, 330), "bf16": kind == "batch_forward" and rng.random() < 0.5,
                "order": rng.choice([3, 3, 3, 5]), "rows": rng.choice([0, 3]), "sizes": rng.randint(1, 1 << 20)}
    big = 1100 if kind in ("fista", "demultiple") else 4000
    Nt = _log_int(rng, 200, big)
    Nx = _log_int(rng, 48, min(Nt, 400) if kind in ("fista", "demultiple") else Nt)
    c = _single("", kind, Nt, Nx, T=rng.uniform(1.0, 4.0), X=rng.uniform(1.5, 3.0), rows=rng.choice([0, 3, 3]),
                order=rng.choice([3, 3, 3, 5]))
    del c["name"]
    if rng.random() < 0.4:      # an image on its own grid
        c["Ntau"], c["Nq"] = max(2, int(Nt * rng.uniform(0.6, 1.0))), max(2, int(Nx * rng.uniform(0.6, 1.0)))
    if kind in ("forward", "adjoint", "pair") and rng.random() < 0.3:
        c["jitter"], c["near"] = rng.uniform(0.1, 0.45), rng.choice([0.0, 0.15])
    if kind in ("fista", "demultiple"):
        c["iters"] = rng.randint(5, 50)
    if kind == "fista":
        c["missing"] = rng.uniform(0.1, 0.5)
    return c


# --------------------------------------------------------------------------
# Geometry and inputs
# --------------------------------------------------------------------------

def _grids(case):
    """Given offsets and slownesses of a jittered geometry (None: the regular grids)."""
    if not case["jitter"]:
        return None, None
    rng = np.random.default_rng(case["Nt"] * 8191 + case["Nx"])
    h = (case["X"] - case["near"]) / (case["Nx"] - 1)
    x = case["near"] + np.arange(case["Nx"]) * h
    x[1:-1] += rng.uniform(-case["jitter"], case["jitter"], case["Nx"] - 2) * h
    q = QMIN + (QMAX - QMIN) * np.linspace(0.0, 1.0, case["Nq"]) ** 1.3
    return x, q


def _kwargs(case):
    x, q = _grids(case)
    d = dict(Nt=case["Nt"], Nx=case["Nx"], Ntau=case["Ntau"], Nq=case["Nq"], dt=case["T"] / (case["Nt"] - 1),
             dx=case["X"] / (case["Nx"] - 1), qmin=QMIN, qmax=QMAX, rows_per_band=case["rows"],
             spline_order=case["order"])
    if x is not None:
        d.update(x=x.tolist(), q=q.tolist())
    return d


def _batch_geometries(case):
    """Gathers at 4 ms and 25 m, sizes uniform over the case's ranges; images of the gathers' sizes."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["gathers"]):
        Nt, Nx = int(rng.integers(case["nt_lo"], case["nt_hi"] + 1)), int(rng.integers(case["nx_lo"], case["nx_hi"] + 1))
        out.append({"Nt": Nt, "Nx": Nx, "Ntau": Nt, "Nq": Nx, "T": (Nt - 1) * 0.004, "X": (Nx - 1) * 0.025,
                    "order": case["order"], "rows": case["rows"], "jitter": 0.0, "near": 0.0})
    return out


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gather(geo, seed, kind="events"):
    """A gather [Nx][Nt]: Ricker events on hyperbolas (10-40 Hz within the sampling), 5 % noise."""
    dev = _device()
    rng = np.random.default_rng([seed, geo["Nt"], geo["Nx"]])
    T, Nt, Nx = geo["T"], geo["Nt"], geo["Nx"]
    x, _ = _grids(geo)
    x = np.linspace(0.0, geo["X"], Nx) if x is None else x
    t = torch.linspace(0.0, T, Nt, dtype=torch.float64, device=dev)[None, :]
    xx = torch.as_tensor(x, dtype=torch.float64, device=dev)[:, None]
    n = 16
    tau0 = rng.uniform(0.05 * T, 0.9 * T, n)
    if kind == "multiples":    # primaries, and as many slower multiples
        q0 = np.concatenate([rng.uniform(0.25, 0.40, n // 2), rng.uniform(0.50, 0.65, n - n // 2)])
    else:
        q0 = rng.uniform(0.25, 0.65, n)
    top = min(40.0, 0.16 * (Nt - 1) / T)
    nu, amp = rng.uniform(0.4 * top, top, n), rng.standard_normal(n)
    f = torch.zeros((Nx, Nt), dtype=torch.float64, device=dev)
    for k in range(n):
        a = (math.pi * nu[k] * (t - torch.sqrt(tau0[k] ** 2 + (q0[k] * xx) ** 2))) ** 2
        f += amp[k] * (1.0 - 2.0 * a) * torch.exp(-a)
    gen = torch.Generator(device="cpu").manual_seed(int(rng.integers(1 << 40)))
    noise = torch.randn(f.shape, generator=gen, dtype=torch.float32).to(dev)
    return (f + 0.05 * f.square().mean().sqrt() * noise).to(torch.float32).contiguous()


def _image(geo, seed):
    """A Radon image [Nq][Ntau]: noise smoothed along tau, with focused events, zero (tapered) at the two ends of
    the slowness aperture."""
    dev = _device()
    rng = np.random.default_rng([seed, geo["Nq"], geo["Ntau"], 7])
    gen = torch.Generator(device="cpu").manual_seed(int(rng.integers(1 << 40)))
    g = torch.randn((geo["Nq"], geo["Ntau"]), generator=gen, dtype=torch.float32).to(dev)
    g[:, 1:-1] = 0.25 * g[:, :-2] + 0.5 * g[:, 1:-1] + 0.25 * g[:, 2:]
    l = torch.as_tensor(rng.integers(0, geo["Nq"], 32), device=dev)
    i = torch.as_tensor(rng.integers(0, geo["Ntau"], 32), device=dev)
    g[l, i] += torch.as_tensor(20.0 * rng.standard_normal(32), dtype=torch.float32, device=dev)
    if geo["Nq"] > 2:
        g[[0, -1]] = 0.0
    return g.contiguous()


def _mask(case, seed):
    keep = np.ones(case["Nx"], np.float32)
    rng = np.random.default_rng([seed, 11])
    keep[rng.choice(case["Nx"], int(round(case["missing"] * case["Nx"])), replace=False)] = 0.0
    return torch.as_tensor(keep, device=_device())


def _inputs(case, seed):
    """The arrays of a case: the same for prepare and exact."""
    kind = case["kind"]
    if kind == "batch_forward":
        dtype = torch.bfloat16 if case["bf16"] else torch.float32
        return {"f": [_gather(g, seed + i).to(dtype) for i, g in enumerate(_batch_geometries(case))]}
    if kind == "batch_adjoint":
        return {"g": [_image(g, seed + i) for i, g in enumerate(_batch_geometries(case))]}
    d = {}
    if kind != "adjoint":
        d["f"] = _gather(case, seed, "multiples" if kind == "demultiple" else "events")
    if kind in ("adjoint", "pair", "autograd"):
        d["g"] = _image(case, seed)
    if kind == "fista":
        d["mask"] = _mask(case, seed)
        d["f"] = d["f"] * d["mask"][:, None]
    return d


def _two_digits(v):
    return float("%.1e" % v)


def prepare(case, seed):
    state = {"case": case, **_inputs(case, seed)}
    if case["kind"].startswith("batch"):
        state["batch"] = b = hr.Batch([_kwargs(g) for g in _batch_geometries(case)])
        if "f" in state:
            state["f"] = b.pack(state["f"], dtype=state["f"][0].dtype)
        else:
            state["g"] = torch.cat([g.reshape(-1) for g in state["g"]])
        return state
    state["plan"] = p = hr.Plan(**_kwargs(case))
    if case["kind"] in ("fista", "demultiple"):
        # step and threshold, found once per survey and noted to two digits
        state["step"] = _two_digits(0.9 / p.opnorm(30))
        state["mu"] = _two_digits(2e-3 * float(p.forward(state["f"]).abs().max()))
    return state


def run(state):
    kind, p = state["case"]["kind"], state.get("plan")
    if kind == "forward":
        return p.forward(state["f"])
    if kind == "adjoint":
        return p.adjoint(state["g"])
    if kind == "pair":
        return p.forward(state["f"]), p.adjoint(state["g"])
    if kind == "autograd":
        f = state["f"].detach().requires_grad_(True)
        g = hr.radon(f, p)
        g.backward(state["g"])
        return g.detach(), f.grad
    if kind == "batch_forward":
        return state["batch"].forward(state["f"])
    if kind == "batch_adjoint":
        return state["batch"].adjoint(state["g"])
    if kind == "fista":
        return p.ista(state["f"], state["mu"], state["case"]["iters"], mask=state["mask"], step=state["step"])
    return p.demultiple(state["f"], 0.45, 0.0, state["mu"], state["case"]["iters"], step=state["step"])


def work(case):
    """Bytes: each input read and each output written once. Flops: the taps
    of the samples and outputs and the real 2-D FFT pair of the zero-padded
    lattices, about four points per sample (2048 x 2048: 17 M)."""
    if case["kind"].startswith("batch"):
        w = {"bytes": 0.0, "flops": 0.0}
        for g in _batch_geometries(case):
            one = work({**g, "kind": "forward"})
            w["bytes"] += one["bytes"] - (2.0 * g["Nt"] * g["Nx"] if case["bf16"] else 0.0)
            w["flops"] += one["flops"]
        return w
    n, m, taps = case["Nt"] * case["Nx"], case["Ntau"] * case["Nq"], case["order"] + 1
    flops = 2.0 * taps * taps * 1.3 * n + 2.0 * taps * 1.5 * m + 5.0 * 4.0 * n * math.log2(4.0 * n)
    passes = {"forward": 1, "adjoint": 1, "pair": 2, "autograd": 2, "fista": 2 * case.get("iters", 0),
              "demultiple": 2 * case.get("iters", 0) + 1}[case["kind"]]
    one_way = {"forward": n + m, "adjoint": n + m, "pair": 2 * (n + m), "autograd": 2 * (n + m), "fista": n + m,
               "demultiple": 2 * n + m}[case["kind"]]
    return {"bytes": 4.0 * one_way, "flops": passes * flops}


# --------------------------------------------------------------------------
# The method in 64 bits, plain torch
# --------------------------------------------------------------------------

_SIGMA, _OMEGA_C, _SPLITS, _OVERLAP = 1.1, 0.4, (0.25, 0.5), 1.25


def _fft_size(n):
    sizes = []
    for a in range(1, 15):
        p = 1 << a
        sizes += [p, 3 * p, 5 * p] + ([9 * p] if p <= 256 else [])
    return min(s for s in sizes if s >= n)


def _spline(x, order):
    a = x.abs()
    if order == 3:
        return torch.where(a < 1, 2 / 3 - a * a + 0.5 * a ** 3, (2 - a).clamp(min=0) ** 3 / 6)
    return ((3 - a).clamp(min=0) ** 5 - 6 * (2 - a).clamp(min=0) ** 5 + 15 * (1 - a).clamp(min=0) ** 5) / 120


def _symbol(n, P, order, dev):
    return torch.sinc(torch.arange(n, dtype=torch.float64, device=dev) / P) ** (order + 1)


class _Method:
    """Forward and adjoint of one geometry, every piece's tables in 64 bits."""

    def __init__(self, case):
        self.dev = dev = _device()
        self.Nt, self.Nx, self.Ntau, self.Nq, self.order = (case[k] for k in ("Nt", "Nx", "Ntau", "Nq", "order"))
        x, q = _grids(case)
        n_t, n_x = self.Nt - 1, self.Nx - 1
        dt, dx = case["T"] / n_t, case["X"] / n_x
        T, X = n_t * dt, (n_x * dx if x is None else float(x[-1]))
        xb = np.arange(self.Nx) / n_x if x is None else x / X
        if x is None:
            xs, wk = xb, np.ones(self.Nx)
            wk[[0, -1]] = 0.5
        else:
            xs = (x[0] + np.arange(self.Nx) * ((X - x[0]) / n_x)) / X
            wk = 0.5 * (np.append(xb[1:], xb[-1]) - np.insert(xb[:-1], 0, xb[0])) * n_x
        if q is None:
            q = np.array([QMIN]) if self.Nq == 1 else QMIN + np.arange(self.Nq) * ((QMAX - QMIN) / (self.Nq - 1))
        m = (q * X / T) ** 2
        psi = np.arctan(m)
        lo, hi = psi[0], psi[-1]
        if hi - lo < 1e-3:
            mid = max(0.5 * (lo + hi), 0.5e-3)
            lo, hi = mid - 0.5e-3, mid + 0.5e-3
        al, be = 0.5 * (hi + lo), hi - lo
        s2a, sb, cb, th = math.sin(2 * al), math.sin(be), math.cos(be), math.tan(be / 2)
        a = sb / math.sqrt(s2a * sb + cb * (s2a + sb) + 1.0)
        O1 = a * math.sin(al + math.pi / 4) / (math.sqrt(2.0) * th)
        O2 = a * math.cos(al + math.pi / 4) * th / math.sqrt(2.0)
        ca, sa = math.cos(al), math.sin(al)

        def square(s, y):
            return a * (ca * (s - 0.5) - sa * (y - 0.5)) + O1, a * (sa * (s - 0.5) + ca * (y - 0.5)) + O2

        def t64(v):
            return torch.as_tensor(v, dtype=torch.float64, device=dev)

        splits = []
        for b in _SPLITS:
            if b * _OVERLAP < 1 and (not splits or b / _OVERLAP >= splits[-1] * _OVERLAP):
                splits.append(b)
        self.pieces = []
        for p in range(len(splits) + 1):
            j0 = 0 if p == 0 else math.ceil(splits[p - 1] / _OVERLAP * n_t - 1e-9)
            j1 = n_t if p == len(splits) else math.floor(splits[p] * _OVERLAP * n_t + 1e-9)
            tb = t64(np.arange(j0, j1 + 1) / n_t)     # numpy: a true division, so samples on the mute line fall as in the plan

            def edge(b):
                u = (torch.log(tb.clamp(min=1e-300) / b) / math.log(_OVERLAP)).clamp(-1, 1)
                return 0.5 * (1 + torch.sin(0.5 * math.pi * u))

            window = (1.0 if p == 0 else edge(splits[p - 1])) - (0.0 if p == len(splits) else edge(splits[p]))
            # the data region: the rectangle of the piece, cut by the mute line s = m[0] y
            s0, s1, c = (j0 / n_t) ** 2, (j1 / n_t) ** 2, m[0]
            rect, poly = [(s0, 0.0), (s1, 0.0), (s1, 1.0), (s0, 1.0)], []
            for i in range(4):
                (ps, py), (rs, ry) = rect[i], rect[(i + 1) % 4]
                vp, vr = ps - c * py, rs - c * ry
                if vp >= 0:
                    poly.append((ps, py))
                if (vp >= 0) != (vr >= 0):
                    w = vp / (vp - vr)
                    poly.append((ps + w * (rs - ps), py + w * (ry - py)))
            us = [square(*v) for v in poly]
            a_r = min(u1 * math.cos(g) + u2 * math.sin(g) for g in (-be / 2, be / 2) for u1, u2 in us)
            r_max = max(math.hypot(*u) for u in us)
            # lattice spacing: the largest step between neighbouring samples, over sigma
            u1, u2 = square(tb[None, :] ** 2, t64(xs)[:, None] ** 2)
            ph, et = torch.atan2(u2, u1), 0.5 * torch.log(u1 * u1 + u2 * u2)
            step = [max(float(v.diff(dim=d).abs().max()) for d in (0, 1)) for v in (ph, et)]
            L = math.log(r_max) - math.log(a_r)
            n_th = max(1, math.ceil(_SIGMA * be / step[0] - 1e-9))
            n_rh = max(1, math.ceil(_SIGMA * L / step[1] - 1e-9))
            dth, drh, guard = be / n_th, L / n_rh, (self.order + 1) // 2
            th0, rh0 = -be / 2 - guard * dth, math.log(a_r) - guard * drh
            Nth, Nrh = n_th + 2 * guard + 1, n_rh + 2 * guard + 1
            thm = min((Nth - 1) * dth, math.acos(math.exp(-(Nrh - 1) * drh)))
            Pth = _fft_size(Nth + math.ceil(thm / dth - 1e-9))
            Prh = _fft_size(Nrh + math.ceil(-math.log(math.cos(thm)) / drh - 1e-9))
            k1, k2 = min(math.floor(_OMEGA_C * Pth), Pth // 2 - 1), min(math.floor(_OMEGA_C * Prh), Prh // 2 - 1)
            # samples: positions in cells, weights
            u1, u2 = square(tb[None, :] ** 2, t64(xb)[:, None] ** 2)
            r2 = u1 * u1 + u2 * u2
            pos_t, pos_r = (torch.atan2(u2, u1) - th0) / dth, (0.5 * torch.log(r2) - rh0) / drh
            w = (window * (2 * a * a * tb / (n_t * n_x * dth * drh)))[None, :] * t64(wk)[:, None] / r2.sqrt()
            back = self.order // 2
            m0, n0 = pos_t.floor().long() - back, pos_r.floor().long() - back
            ok = (tb[None, :] ** 2 >= c * (t64(xb)[:, None] ** 2)) & (m0 >= 0) & (m0 + self.order < Nth) & (n0 >= 0) & \
                (n0 + self.order < Nrh)
            at = torch.nonzero(ok.reshape(-1)).reshape(-1)
            j = torch.arange(j0, j1 + 1, device=dev)
            src = (torch.arange(self.Nx, device=dev)[:, None] * self.Nt + j[None, :]).reshape(-1)[at]
            samples = (src, w.reshape(-1)[at], m0.reshape(-1)[at], n0.reshape(-1)[at], pos_t.reshape(-1)[at],
                       pos_r.reshape(-1)[at])
            # outputs: angle of every column, radius of every line
            ps = t64(psi)
            theta = al - ps
            tau = t64(np.arange(self.Ntau) * (T / (self.Ntau - 1)) / T)
            e = a * torch.cos(ps)[:, None] * (tau[None, :] ** 2 - 0.5 + 0.5 * t64(m)[:, None]) + \
                (O1 * torch.cos(theta) + O2 * torch.sin(theta))[:, None]
            out_r = (torch.log(e.clamp(min=1e-300)) - rh0) / drh
            on0 = out_r.floor().long() - back
            valid = (e >= a_r) & (e <= r_max) & (on0 >= 0) & (on0 + self.order < Nrh)
            out_t = (theta - th0) / dth
            om0 = (out_t.floor().long() - back).clamp(0, Nth - self.order - 1)
            outputs = (valid, on0.clamp(0, Nrh - self.order - 1), out_r, om0, out_t, 2 * X * torch.cos(ps) / a)
            # kernel spectrum on the frequency rectangle: composite Gauss-Legendre
            dw1, dw2 = 1.0 / (Pth * dth), 1.0 / (Prh * drh)
            npan = math.ceil(k1 * dw1 * thm + k2 * dw2 * abs(math.log(math.cos(thm)))) + 4
            gx, gw = np.polynomial.legendre.leggauss(20)
            h = thm / npan
            nodes = t64(((np.arange(npan)[:, None] + 0.5) * h + 0.5 * h * gx[None, :]).reshape(-1))
            wq = t64(np.tile(0.5 * h * gw, npan)) / torch.cos(nodes)
            A = torch.cos(2 * math.pi * nodes[None, :] * (torch.arange(k1 + 1, dtype=torch.float64, device=dev) * dw1)[:, None])
            arg = -2 * math.pi * torch.log(torch.cos(nodes))[:, None] * \
                (torch.arange(k2 + 1, dtype=torch.float64, device=dev) * dw2)[None, :]
            zeta = 2 * torch.complex(A @ (wq[:, None] * torch.cos(arg)), A @ (wq[:, None] * torch.sin(arg)))
            del A, arg
            zeta = zeta / (_symbol(k1 + 1, Pth, self.order, dev)[:, None] * _symbol(k2 + 1, Prh, self.order, dev)[None, :]) ** 2
            K = torch.zeros((Pth, Prh // 2 + 1), dtype=torch.complex128, device=dev)
            K[:k1 + 1, :k2 + 1] = zeta
            K[Pth - k1:, :k2 + 1] = zeta[1:].flip(0)
            self.pieces.append((Nth, Nrh, Pth, Prh, K, samples, outputs))

    def _taps(self, pos, first):
        return [_spline(pos - (first + d), self.order) for d in range(self.order + 1)]

    def _convolve(self, lat, P, conj):
        Nth, Nrh, Pth, Prh, K = P[:5]
        F = torch.fft.rfft2(lat, s=(Pth, Prh)) * (K.conj() if conj else K)
        return torch.fft.irfft2(F, s=(Pth, Prh))[:Nth, :Nrh].contiguous()

    def forward(self, f):
        g = torch.zeros((self.Nq, self.Ntau), dtype=torch.float64, device=self.dev)
        f = f.to(torch.float64).reshape(-1)
        for P in self.pieces:
            Nth, Nrh = P[:2]
            src, w, m0, n0, pt, pr = P[5]
            lat = torch.zeros(Nth * Nrh, dtype=torch.float64, device=self.dev)
            v, wr = f[src] * w, self._taps(pr, n0)
            for i, wt in enumerate(self._taps(pt, m0)):
                for k in range(self.order + 1):
                    lat.index_add_(0, (m0 + i) * Nrh + n0 + k, v * wt * wr[k])
            Q = self._convolve(lat.reshape(Nth, Nrh), P, False)
            valid, on0, out_r, om0, out_t, scale = P[6]
            prof = sum(wt[:, None] * Q[om0 + i] for i, wt in enumerate(self._taps(out_t, om0)))
            line = sum(wr * prof.gather(1, on0 + k) for k, wr in enumerate(self._taps(out_r, on0)))
            g += torch.where(valid, scale[:, None] * line, torch.zeros_like(line))
        return g

    def adjoint(self, g):
        out = torch.zeros(self.Nx * self.Nt, dtype=torch.float64, device=self.dev)
        g = g.to(torch.float64)
        for P in self.pieces:
            Nth, Nrh = P[:2]
            valid, on0, out_r, om0, out_t, scale = P[6]
            v = torch.where(valid, scale[:, None] * g, torch.zeros_like(g))
            prof = torch.zeros((self.Nq, Nrh), dtype=torch.float64, device=self.dev)
            for k, wr in enumerate(self._taps(out_r, on0)):
                prof.scatter_add_(1, on0 + k, v * wr)
            lat = torch.zeros((Nth, Nrh), dtype=torch.float64, device=self.dev)
            for i, wt in enumerate(self._taps(out_t, om0)):
                lat.index_add_(0, om0 + i, wt[:, None] * prof)
            Q = self._convolve(lat, P, True).reshape(-1)
            src, w, m0, n0, pt, pr = P[5]
            s, wr = torch.zeros_like(w), self._taps(pr, n0)
            for i, wt in enumerate(self._taps(pt, m0)):
                for k in range(self.order + 1):
                    s += wt * wr[k] * Q[(m0 + i) * Nrh + n0 + k]
            out.index_add_(0, src, w * s)
        return out.reshape(self.Nx, self.Nt)

    def norm2(self, iters):
        gen = torch.Generator(device="cpu").manual_seed(0)
        v = torch.randn((self.Nq, self.Ntau), generator=gen).to(self.dev, torch.float64)
        for _ in range(iters):
            v = self.forward(self.adjoint(v / v.norm()))
        return float(v.norm())

    def thresholded(self, f, mask, mu, c2, iters, accelerate):
        f = f.to(torch.float64)
        g = torch.zeros((self.Nq, self.Ntau), dtype=torch.float64, device=self.dev)
        y, t = g, 1.0
        for _ in range(iters):
            r = self.adjoint(y)
            v = y + c2 * self.forward(f - (r if mask is None else mask.to(torch.float64)[:, None] * r))
            new = torch.sign(v) * (v.abs() - 0.5 * c2 * mu).clamp(min=0)
            tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t)) if accelerate else 1.0
            y, g, t = new + ((t - 1) / tn if accelerate else 0.0) * (new - g), new, tn
        return g


def exact(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    if kind.startswith("batch"):
        out = []
        for i, g in enumerate(_batch_geometries(case)):
            M = _Method(g)
            out.append((M.forward(d["f"][i]) if kind == "batch_forward" else M.adjoint(d["g"][i])).reshape(-1))
        return torch.cat(out)
    M = _Method(case)
    if kind == "forward":
        return M.forward(d["f"])
    if kind == "adjoint":
        return M.adjoint(d["g"])
    if kind in ("pair", "autograd"):
        return M.forward(d["f"]), M.adjoint(d["g"])
    step = _two_digits(0.9 / M.norm2(30))
    mu = _two_digits(2e-3 * float(M.forward(d["f"]).abs().max()))
    if kind == "fista":
        return M.thresholded(d["f"], d["mask"], mu, step, case["iters"], True)
    g = M.thresholded(d["f"], None, mu, step, case["iters"], False)
    q = torch.linspace(QMIN, QMAX, case["Nq"], dtype=torch.float64, device=M.dev)[:, None]
    return d["f"].to(torch.float64) - M.adjoint(torch.where(q > 0.45, g, torch.zeros_like(g))), g
