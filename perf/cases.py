"""Timed cases of the library: what its users run, through the public entry
points, over the ranges of sizes, models and options that they use.

  listed()             the fixed cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the inputs a program holds before the call, on the GPU
  run(state)           one pass through the public entry points
  work(case)           bytes and operations one pass cannot do without
  exact(case, seed)    the outputs of run() in 64-bit arithmetic, plain torch
"""
import math

import numpy as np
import torch

from paper_2407_18015_gb300 import ucp

DEV = "cuda"

# side lengths (smallest, largest) of the drawn grids and the member counts
SIDES = {"models": (48, 1400), "host": (128, 1400), "bound": (64, 2048), "single": (48, 1600),
         "saddle": (64, 1400), "step": (64, 2048), "mvn": (32, 400), "semi": (64, 700),
         "stencil": (64, 1200), "volume": (12, 128), "batch": (128, 1024)}
MEMBERS = (5, 60)
BINS = (2, 3, 4, 5, 6, 8, 8, 10, 12, 16, 16, 20)


def listed():
    return [
        # the paper's validation grid: every closed-form model of one small
        # ensemble, minimum and maximum (launch latency counts)
        dict(name="validation_64x64x20", kind="models", H=64, W=64, N=20, bins=8, boundary=0),
        # a decompressed climate field with an error bound: uniform parameters
        # from the bound, then minimum and maximum from the parameters
        dict(name="climate_240x960", kind="bound", H=240, W=960, bound=0.8),
        # saddles of a 500 x 500 ocean ensemble of 20 members
        dict(name="saddle_500x500x20", kind="saddle", model="epanechnikov", H=500, W=500, N=20,
             bins=8, boundary=0),
        # the three closed-form models of one megapixel ensemble, resident on
        # the GPU: the benchmark's step
        dict(name="models_1024x1024x20", kind="models", H=1024, W=1024, N=20, bins=8, boundary=0),
        # the same step from pinned host arrays and back: end to end
        dict(name="host_1024x1024x20", kind="host", H=1024, W=1024, N=20, bins=8, boundary=0),
        # one model of an ensemble with odd sides, one type: the 50-member,
        # 5-bin comparison with outliers, local maxima
        dict(name="single_hist5_1021x1023x50", kind="single", model="histogram", H=1021, W=1023,
             N=50, bins=5, types=2, boundary=0),
        # sensitivity of minima to the data's uncertainty: fit, probability
        # field and its gradient through autograd, bin masses
        dict(name="step_hist16_2048x2048x50", kind="step", model="histogram", H=2048, W=2048,
             N=50, bins=16, boundary=0),
        # the same for centres and widths
        dict(name="step_epan_2048x2048x50", kind="step", model="epanechnikov", H=2048, W=2048,
             N=50, bins=8, boundary=0),
        # correlated noise: the multivariate Gaussian by Monte Carlo
        dict(name="mvn_512x512x40", kind="mvn", H=512, W=512, N=40, samples=10000),
        # a time series or parameter study: many fields of uneven sizes and
        # mixed models in one batched call
        dict(name="batch_64_fields", kind="batch", fields=64, lo=128, hi=2048, pick=5, bins=16),
        # the paper's semianalytical histogram estimator
        dict(name="semi_hist8_1024x1024x20", kind="semi", H=1024, W=1024, N=20, bins=8,
             samples=1000),
        # eight neighbours of a pixel grid
        dict(name="stencil8_hist8_1024x1024x20", kind="stencil", stencil=2, model="histogram",
             H=1024, W=1024, N=20, bins=8, types=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, kind):
    """Two side lengths: mostly any integer, sometimes multiples of 4 or 32."""
    lo, hi = SIDES[kind]
    mult = rng.choice((1, 1, 1, 4, 32))
    return tuple(max(mult, _log_int(rng, lo, hi) // mult * mult) for _ in range(2))


def draw(rng):
    kind = rng.choice(("models", "host", "bound", "single", "single", "saddle", "step", "step",
                       "mvn", "batch", "semi", "stencil", "volume"))
    if kind == "batch":
        return dict(kind=kind, fields=rng.randint(4, 32), lo=SIDES[kind][0], hi=SIDES[kind][1],
                    pick=rng.randrange(1 << 20), bins=rng.choice((4, 8, 16, 16)))
    if kind == "volume":
        D, H = _sides(rng, kind)
        return dict(kind="stencil", stencil=3, model=rng.choice(("uniform", "epanechnikov",
                                                                 "histogram")),
                    D=D, H=H, W=_log_int(rng, *SIDES[kind]), N=rng.randint(*MEMBERS),
                    bins=rng.choice((4, 5, 8)), types=3)
    H, W = _sides(rng, kind)
    if kind == "bound":
        return dict(kind=kind, H=H, W=W, bound=round(rng.uniform(0.2, 2.0), 3))
    N = rng.randint(*MEMBERS)
    if kind == "mvn":
        return dict(kind=kind, H=H, W=W, N=max(N, 8), samples=_log_int(rng, 1000, 10000))
    if kind == "semi":
        return dict(kind=kind, H=H, W=W, N=N, bins=rng.choice((4, 5, 8, 16)),
                    samples=_log_int(rng, 100, 1000))
    boundary = rng.choice((0, 0, 1))
    if kind in ("models", "host"):
        return dict(kind=kind, H=H, W=W, N=N, bins=rng.choice((3, 4, 5, 8, 8, 16)),
                    boundary=boundary)
    model = rng.choice(("uniform", "epanechnikov", "histogram", "histogram"))
    bins = rng.choice(BINS)
    if kind == "single":
        if rng.random() < 0.15:
            model, H, W = "gaussian", min(H, 256), min(W, 256)
        return dict(kind=kind, model=model, H=H, W=W, N=N, bins=bins,
                    types=rng.choice((1, 2, 3, 3)), boundary=boundary)
    if kind == "stencil":
        return dict(kind=kind, stencil=rng.choice((1, 2)), model=model, H=H, W=W, N=N,
                    bins=rng.choice((4, 5, 8)), types=rng.choice((1, 2, 3)))
    return dict(kind=kind, model=model, H=H, W=W, N=N, bins=bins, boundary=boundary)


# ---------------------------------------------------------------------------
# inputs


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1000003 + 17)


def _u(g, n, lo, hi):
    return torch.rand(n, generator=g, device=DEV) * (hi - lo) + lo


def _base(g, H, W, scale):
    """Sum of six plane waves, amplitudes 0.5..2, wavelengths 8..32 cells
    times `scale`."""
    amp, lam = _u(g, 6, 0.5, 2.0), _u(g, 6, 8.0, 32.0) * scale
    th, ph = _u(g, 6, 0.0, 2 * math.pi), _u(g, 6, 0.0, 2 * math.pi)
    y = torch.arange(H, device=DEV, dtype=torch.float32)[:, None]
    x = torch.arange(W, device=DEV, dtype=torch.float32)[None, :]
    f = torch.zeros((H, W), device=DEV)
    for j in range(6):
        f += amp[j] * torch.sin(2 * math.pi * (x * torch.cos(th[j]) + y * torch.sin(th[j]))
                                / lam[j] + ph[j])
    return f


def _bimodal(g, N, H, W):
    """Members around a smooth field: two modes whose gap grows from 0 to 1.5
    along x, noise of 0.1 to 0.4 along y."""
    gap = torch.linspace(0.0, 1.5, W, device=DEV)[None, :]
    sd = torch.linspace(0.1, 0.4, H, device=DEV)[:, None]
    ens = torch.randn((N, H, W), generator=g, device=DEV).mul_(sd)
    base = _base(g, H, W, 4.0)
    for k in range(N):
        sign = (torch.rand((H, W), generator=g, device=DEV) < 0.5).float() * 2 - 1
        ens[k] += base + 0.5 * gap * sign
    return ens


def _correlated(g, N, H, W):
    """Members around a smooth field: white noise smoothed by a Gaussian of 3
    cells, standard deviation 0.2."""
    t = torch.arange(-12, 13, device=DEV, dtype=torch.float32)
    k = torch.exp(-0.5 * (t / 3.0) ** 2)
    k = k / k.sum()
    z = torch.randn((N, H + 24, W + 24), generator=g, device=DEV)
    z = sum(k[i] * z[:, i:i + H, :] for i in range(25))
    z = sum(k[i] * z[:, :, i:i + W] for i in range(25))
    return (z * (0.2 / float((k * k).sum())) + _base(g, H, W, 1.0)).contiguous()


def _slabs(case):
    return int(case.get("D", 1))


def _batch_specs(case):
    rng = np.random.default_rng(case["pick"])
    specs = []
    for _ in range(case["fields"]):
        H, W = (int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
                for _ in range(2))
        specs.append((H, W, int(rng.choice([10, 20, 50, 100])),
                      ("uniform", "epanechnikov", "histogram")[int(rng.integers(0, 3))],
                      int(rng.integers(1, 3))))
    return specs


def _inputs(case, seed):
    """The case's input tensors, from the seed alone."""
    g = _generator(seed)
    kind, H, W = case["kind"], case.get("H"), case.get("W")
    if kind == "bound":
        # a smooth field and the compressor's error, inside the bound
        f = 8.0 * _base(g, H, W, 4.0)
        return (f + (torch.rand((H, W), generator=g, device=DEV) - 0.5) * case["bound"],)
    if kind == "mvn":
        return (_correlated(g, case["N"], H, W),)
    if kind == "batch":
        return tuple(_bimodal(g, N, h, w) for h, w, N, _, _ in _batch_specs(case))
    D = _slabs(case)
    ens = _bimodal(g, case["N"], D * H, W)
    if kind == "step":
        return ens, torch.rand((H, W), generator=g, device=DEV)
    return (ens.view(case["N"], D, H, W) if D > 1 else ens,)


MODELS3 = ("uniform", "epanechnikov", "histogram")


def _desc(case, model=None):
    kind = case["kind"]
    model = model or {"mvn": "mvn", "semi": "histogram_semi"}.get(kind) or case["model"]
    return ucp.make_desc(model, bins=case.get("bins", 8), mc_samples=case.get("samples", 1),
                         seed=0x5EED, boundary=case.get("boundary", 0),
                         stencil=case.get("stencil", 0), depth=case.get("D", 0))


def prepare(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    st = {"case": case, "kind": kind, "x": x[0], "ctx": ucp.default_context()}
    if kind in ("models", "host"):
        st["descs"] = [_desc(case, m) for m in MODELS3]
        shape = x[0].shape[1:]
        outs = [[torch.empty(shape, device=DEV) for _ in MODELS3] for _ in range(2)]
        if kind == "host":
            st["x"] = x[0].cpu().pin_memory()
            outs = [[torch.empty(shape).pin_memory() for _ in MODELS3] for _ in range(2)]
        st["outs"] = outs
    elif kind == "bound":
        st["desc"] = ucp.make_desc("uniform")
        st["params"] = torch.empty((2,) + tuple(x[0].shape), device=DEV)
    elif kind == "batch":
        b = ucp.Batch(st["ctx"])
        outs = []
        for ens, (H, W, N, model, types) in zip(x, _batch_specs(case)):
            o = torch.empty((H, W), device=DEV)
            b.add(ens, _desc(case, model), types, o if types == 1 else None,
                  o if types == 2 else None)
            outs.append(o)
        st["batch"], st["outs"] = b, outs
    else:
        st["desc"] = _desc(case)
        if kind == "step":
            st["weight"] = x[1]
    return st


def run(st):
    kind, case, ctx, x = st["kind"], st["case"], st["ctx"], st["x"]
    if kind == "models":
        ucp.ucp_probability_models(ctx.handle, x, st["descs"], 3, st["outs"][0], st["outs"][1])
        return st["outs"]
    if kind == "host":
        ucp.ucp_probability_host_models(ctx.handle, x, st["descs"], 3, st["outs"][0],
                                        st["outs"][1])
        return st["outs"]
    if kind == "bound":
        ucp.ucp_params_from_error_bound(ctx.handle, x, case["bound"], st["params"])
        pmin, pmax, status = ctx.probability_from_params(st["params"], st["desc"])
        return [st["params"], pmin, pmax, status]
    if kind == "saddle":
        return list(ctx.saddle(x, st["desc"]))
    if kind == "batch":
        st["batch"].run()
        return st["outs"]
    if kind == "step":
        params = ctx.fit(x, st["desc"]).requires_grad_()
        P = ucp.UcpProbability.apply(params, case["model"], case["bins"], ucp.UCP_MIN,
                                     case["boundary"])
        P.backward(st["weight"])
        return [params.detach(), P.detach(), params.grad]
    return list(ctx.probability(x, st["desc"], case.get("types", 3)))


# ---------------------------------------------------------------------------
# work


def _vertex_flops(model, bins, K=4):
    """Operations of one vertex and type: K + 1 pieces (uniform: a product of
    K linear factors each; Epanechnikov: eight nodes of K cubic factors),
    (K + 1)(bins + 1) pieces at most for histograms, of which about six in
    ten lie inside the centre's support."""
    if model == "uniform":
        return (K + 1) * 8 * K
    if model == "epanechnikov":
        return (K + 1) * 8 * (8 * K + 3)
    if model == "gaussian":
        return 16 * 16 * 20 * K
    return 0.6 * (K + 1) * (bins + 1) * (18 * K + 3)


def _fit_flops(model, N):
    return (2 if model in ("uniform", "gaussian") else 6) * N


def work(case):
    kind, bins = case["kind"], case.get("bins", 8)
    if kind == "batch":
        b = f = 0.0
        for H, W, N, model, _ in _batch_specs(case):
            b += H * W * 4.0 * (N + 1)
            f += H * W * (_fit_flops(model, N) + _vertex_flops(model, bins))
        return {"bytes": b, "flops": f}
    V = float(_slabs(case) * case["H"] * case["W"])
    if kind == "bound":
        return {"bytes": V * (4 + 8 + 8 + 1), "flops": V * (2 + 2 * _vertex_flops("uniform", 0))}
    N = case["N"]
    if kind in ("models", "host"):
        return {"bytes": V * (4 * N + 24),
                "flops": V * sum(_fit_flops(m, N) + 2 * _vertex_flops(m, bins) for m in MODELS3)}
    if kind == "mvn":
        return {"bytes": V * (4 * N + 9), "flops": V * (55 * N + 250.0 * case["samples"])}
    if kind == "semi":
        return {"bytes": V * (4 * N + 9), "flops": V * (6 * N + 70.0 * case["samples"])}
    model = case["model"]
    if kind == "saddle":
        return {"bytes": V * (4 * N + 5),
                "flops": V * (_fit_flops(model, N) + 2 * _vertex_flops(model, bins))}
    if kind == "step":
        P = 2 + bins if model == "histogram" else 2
        return {"bytes": V * (4 * N + 4 + 4 * (2 * P + 1)),
                "flops": V * (_fit_flops(model, N) + 3 * _vertex_flops(model, bins))}
    K = {0: 4, 1: 6, 2: 8, 3: 6}[case.get("stencil", 0)]
    types = bin(case["types"]).count("1")
    return {"bytes": V * (4 * N + 4 * types + 1),
            "flops": V * (_fit_flops(model, N) + types * _vertex_flops(model, bins, K))}


# ---------------------------------------------------------------------------
# the same values in 64 bits: plain torch, every integrand cut at all the
# breakpoints of its factors and integrated by a Gauss-Legendre rule that is
# exact for the polynomial degree of the pieces

OFFSETS = {0: [(0, 0, 1), (0, -1, 0), (0, 0, -1), (0, 1, 0)]}
OFFSETS[1] = OFFSETS[0] + [(0, -1, 1), (0, 1, -1)]
OFFSETS[2] = OFFSETS[0] + [(0, -1, 1), (0, -1, -1), (0, 1, -1), (0, 1, 1)]
OFFSETS[3] = OFFSETS[0] + [(-1, 0, 0), (1, 0, 0)]
GAUSS_RANGE = 8.0


def _fit64(ens, model, bins):
    """Parameters [P][D][H][W] in 64 bits; the histogram's bin of a member is
    a binary32 decision by definition."""
    if ens.dim() == 3:
        ens = ens[:, None]
    N = ens.shape[0]
    if model in ("epanechnikov", "gaussian"):
        x = ens.double()
        sd = x.std(dim=0, unbiased=True)
        return torch.stack([x.mean(dim=0), sd * (math.sqrt(5.0) if model == "epanechnikov"
                                                 else 1.0)])
    lo, hi = ens.amin(dim=0), ens.amax(dim=0)
    if model == "uniform":
        return torch.stack([lo, hi]).double()
    scale = torch.full_like(lo, float(bins)) / (hi - lo)
    counts = torch.zeros((bins,) + tuple(lo.shape), device=ens.device)
    for k in range(N):
        j = torch.floor((ens[k] - lo) * scale).clamp_(0, bins - 1).long()
        counts.scatter_add_(0, j[None], torch.ones_like(lo)[None])
    return torch.cat([lo[None].double(), hi[None].double(), counts.double() / N])


class _Var:
    """One variable of each of a set of vertices: parameters p [P][V]."""

    def __init__(self, model, p):
        self.model, self.p, self.bins = model, p, p.shape[0] - 2
        if model in ("uniform", "histogram"):
            self.lo, self.hi = p[0], p[1]
        else:
            r = p[1] * (GAUSS_RANGE if model == "gaussian" else 1.0)
            self.lo, self.hi = p[0] - r, p[0] + r
        if model == "histogram":
            self.m = p[2:].t().contiguous()
            z = torch.zeros_like(self.m[:, :1])
            self.c = torch.cat([z, self.m.cumsum(1)], 1)
            self.total = self.c[:, -1]

    def edges(self):
        if self.model == "histogram":
            t = torch.arange(self.bins + 1, device=self.p.device, dtype=torch.float64) / self.bins
            return self.lo[:, None] + (self.hi - self.lo)[:, None] * t
        if self.model == "gaussian":
            return torch.stack([self.lo, self.p[0] - 3 * self.p[1], self.p[0],
                                self.p[0] + 3 * self.p[1], self.hi], 1)
        return torch.stack([self.lo, self.hi], 1)

    def _bin(self, x):
        v = (x - self.lo[:, None]) * (self.bins / (self.hi - self.lo))[:, None]
        j = v.detach().floor().clamp_(0, self.bins - 1)
        return v, j, j.long()

    def pdf(self, x):
        if self.model == "uniform":
            return (1.0 / (self.hi - self.lo))[:, None].expand_as(x)
        if self.model == "histogram":
            _, _, j = self._bin(x)
            return self.m.gather(1, j) * (self.bins / (self.hi - self.lo))[:, None]
        u = (x - self.p[0][:, None]) / self.p[1][:, None]
        if self.model == "gaussian":
            return torch.exp(-0.5 * u * u) / (math.sqrt(2 * math.pi) * self.p[1][:, None])
        return 0.75 / self.p[1][:, None] * (1 - u * u)

    def tails(self, x):
        """(survival, CDF) at x."""
        if self.model == "histogram":
            v, k, j = self._bin(x)
            F = self.c.gather(1, j) + self.m.gather(1, j) * (v - k).clamp(0, 1)
            F = torch.where(v <= 0, torch.zeros_like(F), F)
            F = torch.where(v >= self.bins, self.total[:, None].expand_as(F), F)
            return self.total[:, None] - F, F
        if self.model == "uniform":
            F = ((x - self.lo[:, None]) / (self.hi - self.lo)[:, None]).clamp(0, 1)
            return 1 - F, F
        u = (x - self.p[0][:, None]) / self.p[1][:, None]
        if self.model == "gaussian":
            z = u / math.sqrt(2.0)
            return 0.5 * torch.erfc(z), 0.5 * torch.erfc(-z)
        u = u.clamp(-1, 1)
        G = 0.25 * (1 - u) * (1 - u) * (2 + u)
        return G, 1 - G


def _integrals(model, centre, nbrs, present, saddle):
    """(P_min, P_max) or, with saddle, the saddle probability of the vertices
    whose variables are centre [P][V] and nbrs (K of [P][V]); present: K of
    [V]."""
    c, ns = _Var(model, centre), [_Var(model, p) for p in nbrs]
    e = torch.cat([c.edges()] + [n.edges() for n in ns], 1)
    e = torch.maximum(torch.minimum(e, c.hi[:, None]), c.lo[:, None]).sort(1).values
    K = len(ns)
    degree = {"uniform": K, "histogram": K, "epanechnikov": 2 + 3 * K, "gaussian": 31}[model]
    xs, ws = (torch.from_numpy(v).to(e) for v in np.polynomial.legendre.leggauss(degree // 2 + 1))
    half, mid = 0.5 * (e[:, 1:] - e[:, :-1]), 0.5 * (e[:, 1:] + e[:, :-1])
    x = (mid[:, :, None] + half[:, :, None] * xs).flatten(1)
    w = (half[:, :, None] * ws).flatten(1) * c.pdf(x)
    a = b = w
    for i, n in enumerate(ns):
        G, F = n.tails(x)
        if saddle and i % 2:
            G, F = F, G
        on = present[i][:, None]
        a = a * torch.where(on, G, torch.ones_like(G))
        b = b * torch.where(on, F, torch.ones_like(F))
    a, b = a.sum(1), b.sum(1)
    return a + b if saddle else (a, b)


def _field64(params, model, stencil=0, boundary=0, saddle=False, weight=None, nodes=1 << 24):
    """Probability fields of parameters [P][D][H][W]; with a weight also the
    gradient of sum(weight * P_min) by the parameters (a histogram's support
    held fixed).  Works through the vertices in blocks of rows."""
    P, D, H, W = params.shape
    offs = OFFSETS[stencil]
    K, B = len(offs), (P - 2 if model == "histogram" else 1)
    per = (K + 1) * (B + 1) * max(2, K // 2 + 1) * (4 if model in ("epanechnikov", "gaussian")
                                                      else 1)
    rows = max(1, nodes // (per * W))
    if weight is not None:
        rows = max(1, rows // 3)
    flat = params.reshape(P, D * H, W)
    out = [torch.empty((D * H, W), dtype=torch.float64, device=params.device) for _ in range(2)]
    grad = torch.zeros_like(flat) if weight is not None else None
    for r0 in range(0, D * H, rows):
        r1 = min(D * H, r0 + rows)
        pad = H if D > 1 else 1
        s0, s1 = max(0, r0 - pad), min(D * H, r1 + pad)
        slab = flat[:, s0:s1].contiguous()
        if weight is not None:
            slab.requires_grad_()
        q = slab.reshape(P, -1)
        r = torch.arange(r0, r1, device=params.device)[:, None].expand(r1 - r0, W).reshape(-1)
        xx = torch.arange(W, device=params.device)[None, :].expand(r1 - r0, W).reshape(-1)
        z, y = r // H, r % H
        nbrs, present = [], []
        for dz, dy, dx in offs:
            on = ((z + dz >= 0) & (z + dz < D) & (y + dy >= 0) & (y + dy < H) & (xx + dx >= 0)
                  & (xx + dx < W))
            at = (r + torch.where(on, dz * H + dy, 0) - s0) * W + xx + torch.where(on, dx, 0)
            nbrs.append(q[:, at])
            present.append(on)
        res = _integrals(model, q[:, (r - s0) * W + xx], nbrs, present, saddle)
        full = torch.stack(present).all(0)
        keep = full if (boundary == 1 or saddle) else torch.ones_like(full)
        res = [torch.where(keep, v, torch.zeros_like(v)) for v in (res, res)[:1]] if saddle else \
            [torch.where(keep, v, torch.zeros_like(v)) for v in res]
        if weight is not None:
            g, = torch.autograd.grad((res[0] * weight[r0:r1].reshape(-1).double()).sum(), slab)
            if model == "histogram":
                g[:2] = 0
            grad[:, s0:s1] += g
        for o, v in zip(out, res):
            o[r0:r1] = v.detach().reshape(r1 - r0, W)
    shape = (D, H, W) if D > 1 else (H, W)
    out = [o.reshape(shape) for o in out]
    return out if weight is None else (out, grad.reshape((P,) + shape))


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al., SC'11) on 32-bit words held in int64."""
    M = 0xFFFFFFFF
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((b >> 32) & M) ^ c1 ^ k0, b & M, ((a >> 32) & M) ^ c3 ^ k1, a & M)
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _grid_neighbours(H, W, device):
    """Vertex indices [V], and for e, n, w, s the index and presence."""
    v = torch.arange(H * W, device=device)
    y, x = v // W, v % W
    nb = []
    for _, dy, dx in OFFSETS[0]:
        on = (y + dy >= 0) & (y + dy < H) & (x + dx >= 0) & (x + dx < W)
        nb.append((torch.where(on, v + dy * W + dx, v), on))
    return v, nb


def _mvn64(ens, samples, seed, chunk=1 << 24):
    """Monte Carlo hits of the multivariate Gaussian on the documented random
    stream.  Absent neighbours at the border would change the order of the
    variables: those vertices take theirs in the order of the present ones."""
    N, H, W = ens.shape
    e = ens.reshape(N, -1).double()
    v, nb = _grid_neighbours(H, W, ens.device)
    pmin = torch.zeros(H * W, dtype=torch.float64, device=ens.device)
    pmax = torch.zeros_like(pmin)
    code = sum(on.long() << i for i, (_, on) in enumerate(nb))
    for c in code.unique().tolist():
        sel = v[code == c]
        cols = [sel] + [at[sel] for i, (at, _) in enumerate(nb) if c >> i & 1]
        n = len(cols)
        mu = torch.stack([e[:, q].mean(0) for q in cols])
        X = torch.stack([e[:, q] - m for q, m in zip(cols, mu)])
        L = torch.linalg.cholesky(torch.einsum("akv,bkv->vab", X, X) / (N - 1))
        per = max(1, chunk // sel.numel())
        for s0 in range(0, samples, per):
            s = torch.arange(s0, min(samples, s0 + per), device=ens.device)[:, None]
            u = []
            for j in range(2):
                words = _philox(*torch.broadcast_tensors(
                    s, sel[None, :], torch.zeros_like(s), torch.full_like(s, j)),
                    seed & 0xFFFFFFFF, seed >> 32)
                u += [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in words]
            z = []
            for a, b in zip(u[0:6:2], u[1:6:2]):
                rad = torch.sqrt(-2 * torch.log(a))
                z += [rad * torch.cos(2 * math.pi * b), rad * torch.sin(2 * math.pi * b)]
            xv = mu[0] + L[:, 0, 0] * z[0]
            lt = torch.ones_like(xv, dtype=torch.bool)
            gt = lt.clone()
            for i in range(1, n):
                xn = mu[i] + sum(L[:, i, b] * z[b] for b in range(i + 1))
                lt &= xv < xn
                gt &= xv > xn
            pmin[sel] += lt.sum(0)
            pmax[sel] += gt.sum(0)
    return [(p / samples).reshape(H, W) for p in (pmin, pmax)]


def _semi64(ens, bins, samples, seed, chunk=1 << 24):
    """The semianalytical estimator on the documented random stream; the bin
    of a sample is a binary32 decision by definition."""
    N, H, W = ens.shape
    p = _fit64(ens, "histogram", bins).reshape(2 + bins, -1)
    m32 = p[2:].float()
    C = torch.zeros_like(m32)
    run_sum = torch.zeros_like(m32[0])
    for q in range(bins):
        run_sum = run_sum + m32[q]
        C[q] = run_sum
    v, nb = _grid_neighbours(H, W, ens.device)
    pmin = torch.zeros(H * W, dtype=torch.float64, device=ens.device)
    pmax = torch.zeros_like(pmin)
    per = max(1, chunk // samples)
    s = torch.arange(0, samples, 2, device=ens.device)[:, None] >> 1
    for v0 in range(0, H * W, per):
        sel = v[v0:v0 + per]
        words = _philox(*torch.broadcast_tensors(s, sel[None, :], torch.zeros_like(s),
                                                 torch.full_like(s, 2)),
                        seed & 0xFFFFFFFF, seed >> 32)
        u = [(((w >> 8).double() + 0.5) * 2.0 ** -24).float() for w in words]
        # (the last block's second half is not drawn for an odd count)
        ua, ub = torch.cat([u[0], u[2]])[:samples], torch.cat([u[1], u[3]])[:samples]
        T = C[-1, sel]
        t = ua * T
        j = sum((C[q, sel] <= t).long() for q in range(bins)).clamp_(max=bins - 1)
        h = (p[1] - p[0])[sel] / bins
        x = (p[0][sel] + (j.double() + ub.double()) * h).t().contiguous()
        a = torch.ones_like(x)
        b = torch.ones_like(x)
        for at, on in nb:
            G, F = _Var("histogram", p[:, at[sel]]).tails(x)
            one = torch.ones_like(G)
            a = a * torch.where(on[sel][:, None], G, one)
            b = b * torch.where(on[sel][:, None], F, one)
        total = p[2:, sel].sum(0)
        pmin[sel], pmax[sel] = a.mean(1) * total, b.mean(1) * total
    return [q.reshape(H, W) for q in (pmin, pmax)]


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    bins, boundary = case.get("bins", 8), case.get("boundary", 0)
    if kind in ("models", "host"):
        res = [_field64(_fit64(x[0], m, bins), m, boundary=boundary) for m in MODELS3]
        return [[r[0] for r in res], [r[1] for r in res]]
    if kind == "bound":
        # the parameters are binary32 by definition
        p = torch.stack([x[0] - 0.5 * case["bound"], x[0] + 0.5 * case["bound"]])
        return [p.double()] + _field64(p.double()[:, None], "uniform") + [None]
    if kind == "saddle":
        m = case["model"]
        return [_field64(_fit64(x[0], m, bins), m, saddle=True)[0], None]
    if kind == "batch":
        return [_field64(_fit64(e, m, bins), m)[t - 1]
                for e, (_, _, _, m, t) in zip(x, _batch_specs(case))]
    if kind == "step":
        m = case["model"]
        p = _fit64(x[0], m, bins)
        (pmin, _), grad = _field64(p, m, boundary=boundary, weight=x[1])
        return [p[:, 0], pmin, grad]
    if kind == "mvn":
        return _mvn64(x[0], case["samples"], 0x5EED) + [None]
    if kind == "semi":
        return _semi64(x[0], bins, case["samples"], 0x5EED) + [None]
    m = case["model"]
    res = _field64(_fit64(x[0], m, bins), m, stencil=case.get("stencil", 0), boundary=boundary)
    return [res[0] if case["types"] & 1 else None, res[1] if case["types"] & 2 else None, None]
