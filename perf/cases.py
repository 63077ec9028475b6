"""Performance cases of the gap-filling library: the work its users have it do,
through its public entry points, on synthetic fields of the kinds the tests and
the benchmark use (Gaussian random fields with exponential covariance, gaps at
random or as a union of discs).

A case is a dict of plain values; ``kind`` selects the work:

  fill       one field from host arrays to predictions (create, calibrate,
             simulate, predict): GapFiller
  fill3      the same for a D x H x W cube: GapFiller3
  calibrate  temperatures of one field, or of a batch of uneven fields
  simulate   realizations and predictions at given temperatures, of one field
             or of a batch; FP32 / BF16 / FP16 state, both stop rules, block or
             smoothed site temperatures
  chains     the conditional mean from sampled chains
  gradient   block energies and their gradient (autograd)
  create     a context and its block statistics (transform, Eq. 2, gap lists)
  stats      block statistics without allocation
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2212_01317_gb300 import mpr
from paper_2212_01317_gb300.autograd import BlockEnergy

DEV = "cuda"
# The calibration the benchmark runs: trisection from the unconditional e(T)
# curve, 14 iterations.
WARM = {"points": 2, "warm": 1.5, "iters": 14}
# The library's defaults: 24 bisections over the whole bracket.
COLD = {"points": 1, "warm": 0.0, "iters": 24}


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # the smallest field of the benchmark's workloads, whole call, default options:
        # launches and latency
        {"name": "fill_128", "kind": "fill", "h": 128, "w": 128, "block": 8, "gap": 0.33,
         "discs": False, "xi_lo": 8.0, "xi_hi": 8.0, "reals": 10, "storage": 0, **COLD},
        # a 3-D field (space-time cube), whole call
        {"name": "fill_cube_128", "kind": "fill3", "d": 128, "h": 128, "w": 128, "block": 16,
         "gap": 0.5, "xi_lo": 8.0, "reals": 20, **COLD},
        # the benchmark's single field: temperatures of a field that a GPU holds in one wave
        {"name": "calibrate_1024", "kind": "calibrate", "h": 1024, "w": 1024, "block": 16,
         "gap": 0.5, "discs": False, "xi_lo": 4.0, "xi_hi": 32.0, "fields": 1, **WARM},
        # a batch of uneven time slices: calibration of many waves
        {"name": "calibrate_slices", "kind": "calibrate", "h": 256, "w": 2048, "block": 32,
         "gap": 0.5, "discs": False, "xi_lo": 4.0, "xi_hi": 32.0, "fields": 32, **WARM},
        # the benchmark's single field: many realizations of an FP32 state
        {"name": "simulate_1024", "kind": "simulate", "h": 1024, "w": 1024, "block": 16,
         "gap": 0.5, "discs": False, "xi_lo": 4.0, "xi_hi": 32.0, "fields": 1, "reals": 100,
         "storage": 0, "window": False, "smooth": 0},
        # a large field with cloud gaps, few realizations, BF16 state
        {"name": "simulate_4096_bf16", "kind": "simulate", "h": 4096, "w": 4096, "block": 32,
         "gap": 0.6, "discs": True, "xi_lo": 4.0, "xi_hi": 64.0, "fields": 1, "reals": 10,
         "storage": 1, "window": False, "smooth": 0},
        # the benchmark's headline form: uneven slices in one context, BF16 state
        {"name": "simulate_slices_bf16", "kind": "simulate", "h": 256, "w": 2048, "block": 32,
         "gap": 0.5, "discs": False, "xi_lo": 4.0, "xi_hi": 32.0, "fields": 32, "reals": 50,
         "storage": 1, "window": False, "smooth": 0},
        # site-specific temperatures on an odd-sized field with partial blocks
        {"name": "simulate_sst_odd", "kind": "simulate", "h": 1021, "w": 1531, "block": 16,
         "gap": 0.3, "discs": False, "xi_lo": 6.0, "xi_hi": 6.0, "fields": 1, "reals": 20,
         "storage": 0, "window": False, "smooth": 16},
        # the sampling variant: eight chains, FP16 state, odd sides
        {"name": "chains_2011_f16", "kind": "chains", "h": 2011, "w": 2011, "block": 32,
         "gap": 0.6, "discs": True, "xi_lo": 4.0, "xi_hi": 32.0, "chains": 8, "equil": 25,
         "samples": 50, "storage": 2},
        # differentiable energy matching: forward and backward
        {"name": "gradient_1024", "kind": "gradient", "h": 1024, "w": 1024, "block": 32,
         "gap": 0.5, "discs": True, "xi_lo": 8.0, "xi_hi": 32.0, "chains": 4, "equil": 25,
         "meas": 20},
        # setting a large field up: transform, block statistics, gap lists
        {"name": "create_4096", "kind": "create", "h": 4096, "w": 4096, "block": 32, "gap": 0.6,
         "discs": True, "xi_lo": 16.0, "xi_hi": 16.0},
        # the allocation-free statistics of a small tile: the shortest call
        {"name": "stats_256", "kind": "stats", "h": 256, "w": 256, "block": 16, "gap": 0.4,
         "discs": False, "xi_lo": 8.0, "xi_hi": 8.0},
    ]


def _log(rng, lo, hi):
    """A whole number spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fill", "fill3", "calibrate", "calibrate", "simulate", "simulate", "simulate",
                       "batch", "chains", "gradient", "create", "stats"])
    gap = round(rng.uniform(0.1, 0.85), 3)
    discs = rng.random() < 0.5
    xi = round(rng.uniform(4.0, 32.0), 2)
    field = {"gap": gap, "discs": discs, "xi_lo": xi, "xi_hi": xi}
    cal = rng.choice([COLD, WARM, WARM, {"points": 4, "warm": 1.5, "iters": 8}])
    if kind == "fill":
        return {"kind": kind, "h": _log(rng, 48, 512), "w": _log(rng, 48, 512),
                "block": rng.choice([8, 16, 32]), **field, "reals": _log(rng, 4, 24),
                "storage": rng.choice([0, 0, 1]), **cal}
    if kind == "fill3":
        return {"kind": kind, "d": _log(rng, 12, 128), "h": _log(rng, 24, 128),
                "w": _log(rng, 24, 128), "block": rng.choice([8, 16]), "gap": gap, "xi_lo": 8.0,
                "reals": _log(rng, 4, 20), **COLD}
    if kind == "calibrate":
        return {"kind": kind, "h": _log(rng, 200, 2048), "w": _log(rng, 200, 2048),
                "block": rng.choice([8, 16, 32]), **field, "fields": 1, **cal}
    if kind == "simulate":
        h, w = _log(rng, 200, 4096), _log(rng, 200, 4096)
        most = max(2, min(100, 160_000_000 // (h * w)))
        return {"kind": kind, "h": h, "w": w, "block": rng.choice([16, 32] if h * w < 1 << 22 else [32, 64]),
                **field, "fields": 1, "reals": _log(rng, 2, most),
                "storage": rng.choice([0, 0, 1, 2]), "window": rng.random() < 0.25,
                "smooth": rng.choice([0, 0, 0, 16]) if h * w < 1 << 22 else 0}
    if kind == "batch":
        lo = _log(rng, 200, 400)
        return {"kind": "simulate", "h": lo, "w": _log(rng, lo + 100, 1500), "block": 32, "gap": gap,
                "discs": False, "xi_lo": 4.0, "xi_hi": 32.0, "fields": _log(rng, 2, 20),
                "reals": _log(rng, 8, 40), "storage": rng.choice([0, 1]), "window": False,
                "smooth": 0}
    if kind == "chains":
        return {"kind": kind, "h": _log(rng, 256, 3000), "w": _log(rng, 256, 3000), "block": 32,
                **field, "chains": _log(rng, 2, 16), "equil": 25, "samples": _log(rng, 20, 60),
                "storage": rng.choice([0, 1, 2])}
    if kind == "gradient":
        return {"kind": kind, "h": _log(rng, 128, 2048), "w": _log(rng, 128, 2048),
                "block": rng.choice([16, 32, 64]), **field, "chains": _log(rng, 1, 8), "equil": 25,
                "meas": 20}
    if kind == "create":
        return {"kind": kind, "h": _log(rng, 256, 4096), "w": _log(rng, 256, 4096),
                "block": rng.choice([16, 32, 64]), **field}
    return {"kind": "stats", "h": _log(rng, 48, 4000), "w": _log(rng, 48, 4000),
            "block": rng.choice([16, 32]), **field}


# ----------------------------------------------------------------- inputs --
def _spectrum(n, xi, dims):
    d = torch.arange(n, device=DEV, dtype=torch.float32)
    d = torch.minimum(d, n - d)
    r2 = 0.0
    for k in range(dims):
        r2 = r2 + (d * d).reshape([-1 if j == k else 1 for j in range(dims)])
    return torch.fft.rfftn(torch.exp(-torch.sqrt(r2) / xi)).real.clamp_min(0.0).sqrt()


def _grf(shape, xi_lo, xi_hi, gen):
    """Gaussian random field of exponential covariance by spectral synthesis on
    a torus (zero mean, unit variance); the correlation length runs from xi_lo
    at the left to xi_hi at the right (blended from four filtered fields)."""
    n = 1 << max(4, (max(shape) - 1).bit_length())
    noise = torch.fft.rfftn(torch.randn([n] * len(shape), generator=gen, device=DEV))
    cut = tuple(slice(0, s) for s in shape)

    def filtered(xi):
        f = torch.fft.irfftn(_spectrum(n, xi, len(shape)) * noise, s=[n] * len(shape))[cut]
        return (f - f.mean()) / f.std()

    if xi_lo == xi_hi:
        return filtered(xi_lo).contiguous()
    xs = [xi_lo * (xi_hi / xi_lo) ** (k / 3.0) for k in range(4)]
    at = torch.linspace(xi_lo, xi_hi, shape[-1], device=DEV).log()
    out = torch.zeros(shape, device=DEV)
    for k, x in enumerate(xs):
        step = math.log(xs[1] / xs[0])
        out += filtered(x) * (1.0 - (at - math.log(x)).abs() / step).clamp_min(0.0)
    return ((out - out.mean()) / out.std()).contiguous()


def _discs(h, w, gap, gen):
    """Union of discs of radius 5-60 (at most an eighth of the field's shorter
    side) covering about the fraction `gap`."""
    r_hi = max(3, min(60, min(h, w) // 8))
    r_lo = min(5, r_hi)
    mean_area = math.pi * sum(r * r for r in range(r_lo, r_hi + 1)) / (r_hi - r_lo + 1)
    n = max(1, int(round(-math.log(1.0 - gap) * (h + r_hi) * (w + r_hi) / mean_area)))
    draws = torch.rand(n, 3, generator=gen, device=DEV).cpu().numpy()
    table = {}
    m = torch.zeros(h + 2 * r_hi, w + 2 * r_hi, dtype=torch.uint8, device=DEV)
    for u, v, s in draws:
        r = r_lo + int(s * (r_hi - r_lo + 1) * 0.999999)
        if r not in table:
            d = torch.arange(-r, r + 1, device=DEV)
            table[r] = ((d[:, None] ** 2 + d[None, :] ** 2) <= r * r).to(torch.uint8)
        y, x = int(u * (h + r_hi)) + r_hi // 2, int(v * (w + r_hi)) + r_hi // 2
        y0, x0 = max(0, y - r), max(0, x - r)
        part = m[y0:y + r + 1, x0:x + r + 1]
        part |= table[r][y0 - (y - r):, x0 - (x - r):][:part.shape[0], :part.shape[1]]
    return m[r_hi:r_hi + h, r_hi:r_hi + w].contiguous()


def _field(h, w, gap, discs, xi_lo, xi_hi, gen):
    """(values float32 with the gap sites' truth left out, mask uint8) on the GPU."""
    z = _grf((h, w), xi_lo, xi_hi, gen)
    if discs:
        m = _discs(h, w, gap, gen)
    else:
        m = (torch.rand(h, w, generator=gen, device=DEV) < gap).to(torch.uint8)
    m[0, :2] = 0   # one sample pair at least
    return torch.where(m != 0, torch.full_like(z, float("nan")), z), m


def _fields(case, gen):
    if case["fields"] == 1:
        return [_field(case["h"], case["w"], case["gap"], case["discs"], case["xi_lo"],
                       case["xi_hi"], gen)]
    # a batch: square fields, sides log-uniform over [h, w], each its own gap
    # fraction, correlation length and kind of mask
    out = []
    u = torch.rand(case["fields"], 3, generator=gen, device=DEV).cpu().numpy()
    # (the sides are the case's, the same for every seed, so that the work is)
    sides = np.random.default_rng(case["fields"]).uniform(math.log(case["h"]), math.log(case["w"]),
                                                          case["fields"])
    for k, (a, b, c) in enumerate(u):
        side = int(round(math.exp(sides[k])))
        xi = case["xi_lo"] + (case["xi_hi"] - case["xi_lo"]) * float(b)
        spread = min(case["gap"] - 0.05, 0.9 - case["gap"], 0.4)
        out.append(_field(side, side, case["gap"] + spread * (2.0 * float(a) - 1.0), bool(c < 0.5),
                          xi, xi, gen))
    return out


class _Context:
    """An mpr context that is destroyed with its owner."""

    def __init__(self, fields, block, options):
        if len(fields) == 1:
            v, m = fields[0]
            self.ctx = mpr.mpr_create(m.shape[0], m.shape[1], block, m, v, options)
        else:
            self.ctx = mpr.mpr_create_batch([(m.shape[0], m.shape[1], block) for _, m in fields],
                                            [m for _, m in fields], [v for v, _ in fields], options)

    def close(self):
        if self.ctx:
            mpr.mpr_destroy(self.ctx)
            self.ctx = None

    __del__ = close


def _cal_options(case):
    return {"cal_points": case["points"], "cal_warm": case["warm"], "n_bisect": case["iters"]}


def prepare(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)
    s = {"case": case, "seed": int(seed)}
    if kind == "fill3":
        z = _grf((case["d"], case["h"], case["w"]), case["xi_lo"], case["xi_lo"], gen)
        m = (torch.rand(z.shape, generator=gen, device=DEV) < case["gap"]).to(torch.uint8)
        m[0, 0, :2] = 0
        s["values"] = torch.where(m != 0, torch.full_like(z, float("nan")), z).cpu().numpy()
        s["mask"] = m.cpu().numpy()
        return s
    fields = _fields({"fields": 1, **case}, gen)
    if kind == "fill":
        s["values"], s["mask"] = (x.cpu().numpy() for x in fields[0])
        return s
    if kind == "create":
        s["fields"] = fields
        return s
    if kind == "stats":
        n = -(-case["h"] // case["block"]) * -(-case["w"] // case["block"])
        s["fields"] = fields
        s["out"] = {"Es": torch.zeros(n, dtype=torch.float64, device=DEV),
                    "Nsp": torch.zeros(n, dtype=torch.int32, device=DEV),
                    "Nb": torch.zeros(n, dtype=torch.int32, device=DEV),
                    "mean_angle": torch.zeros(n, device=DEV),
                    "n_gap": torch.zeros(n, dtype=torch.int32, device=DEV),
                    "zrange": torch.zeros(2, dtype=torch.float64, device=DEV)}
        return s
    opts = {"seed": s["seed"]}
    if kind == "calibrate":
        opts.update(_cal_options(case))
    else:
        opts.update(_cal_options(WARM))   # the realizations follow a calibration
    if kind in ("simulate", "chains"):
        opts.update(storage=case["storage"])
    if kind == "simulate" and case["window"]:
        opts.update(stop_rule=mpr.MPR_STOP_WINDOW)
    if kind == "gradient":
        opts.update(cal_chains=case["chains"])
    s["context"] = c = _Context(fields, case["block"], mpr.mpr_default_options(**opts))
    info = mpr.mpr_get_info(c.ctx)
    s["T"] = torch.zeros(info.nblk, device=DEV)
    if kind == "calibrate":
        return s
    mpr.mpr_calibrate(c.ctx, s["T"])
    if kind == "gradient":
        s["beta"] = (1.0 / s["T"]).requires_grad_(True)
        s["grad_y"] = torch.randn(info.nblk, generator=gen, device=DEV, dtype=torch.float64)
        return s
    s["out"] = [torch.zeros_like(v) for v, _ in fields]
    if case.get("smooth"):
        s["T_site"] = torch.zeros_like(fields[0][0])
    return s


# -------------------------------------------------------------------- run --
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fill":
        f = mpr.GapFiller(s["values"], s["mask"], case["block"], seed=s["seed"],
                          storage=case["storage"], **_cal_options(case))
        T = f.calibrate()
        f.simulate(case["reals"])
        pred, _ = f.predict()
        f.close()
        return {"T": T, "pred": pred}
    if kind == "fill3":
        f = mpr.GapFiller3(s["values"], s["mask"], case["block"], seed=s["seed"],
                           n_bisect=case["iters"])
        T = f.calibrate()
        f.simulate(case["reals"])
        pred, _ = f.predict()
        f.close()
        return {"T": T, "pred": pred}
    if kind == "stats":
        (v, m), o = s["fields"][0], s["out"]
        mpr.mpr_block_stats_noalloc(case["h"], case["w"], case["block"], m, v, o["Es"], o["Nsp"],
                                    o["Nb"], o["mean_angle"], o["n_gap"], o["zrange"])
        return o
    if kind == "create":
        c = _Context(s["fields"], case["block"], None)
        n = mpr.mpr_get_info(c.ctx).nblk
        o = {"Es": torch.empty(n, dtype=torch.float64, device=DEV),
             "Nsp": torch.empty(n, dtype=torch.int32, device=DEV),
             "Nb": torch.empty(n, dtype=torch.int32, device=DEV),
             "mean_angle": torch.empty(n, device=DEV),
             "n_gap": torch.empty(n, dtype=torch.int32, device=DEV)}
        mpr.mpr_get_block_stats(c.ctx, o["Es"], o["Nsp"], o["Nb"], o["mean_angle"], o["n_gap"])
        c.close()
        return o
    ctx = s["context"].ctx
    if kind == "calibrate":
        mpr.mpr_calibrate(ctx, s["T"])
        return {"T": s["T"]}
    if kind == "gradient":
        y = BlockEnergy.apply(s["beta"], ctx, case["equil"], case["meas"], 1, True)
        g, = torch.autograd.grad(y, s["beta"], s["grad_y"])
        return {"y": y, "grad_beta": g}
    # realizations (or samples) join the context's running mean
    if kind == "chains":
        mpr.mpr_sample_chains(ctx, case["chains"], case["equil"], case["samples"])
    else:
        if case["smooth"]:
            mpr.mpr_smooth_temperatures(ctx, case["smooth"], 5, s["T_site"])
        mpr.mpr_simulate(ctx, case["reals"])
    if len(s["out"]) == 1:
        mpr.mpr_predict(ctx, s["out"][0])
    else:
        mpr.mpr_predict_batch(ctx, s["out"])
    return {"pred": s["out"], "T_site": s["T_site"]} if case.get("smooth") else {"pred": s["out"]}


# ------------------------------------------------------------------- work --
# Arithmetic of one site update that the method cannot do without: the local
# field (a cos / sin pair and an add each per neighbour), two cos / sin pairs,
# two energies, one exp, one atan2 and the reflection, two uniforms.
FLOPS_2D, FLOPS_3D = 60.0, 68.0
# Sweeps of a realization: the median block stops after 20 to 30.
SWEEPS = 25


def _sites(case):
    if case.get("fields", 1) == 1:
        return case.get("d", 1) * case["h"] * case["w"]
    sides = np.random.default_rng(case["fields"]).uniform(math.log(case["h"]), math.log(case["w"]),
                                                          case["fields"])
    return sum(int(round(math.exp(x))) ** 2 for x in sides)


def work(case):
    kind, n = case["kind"], _sites(case)
    gaps = case["gap"] * n
    blocks = n / case["block"] ** (3 if kind == "fill3" else 2)
    if kind in ("create", "stats"):
        # values and mask read; a cosine, a difference and an add per sample bond
        return {"bytes": 5.0 * n + 24.0 * blocks, "flops": 2 * (1 - case["gap"]) ** 2 * n * 8.0}
    state = {0: 4.0, 1: 2.0, 2: 2.0}[case.get("storage", 0)]
    sweeps = 0.0   # site updates per gap site
    if kind in ("fill", "fill3", "calibrate"):
        sweeps += case["iters"] * 45.0 * case["points"]
    if kind in ("fill", "fill3", "simulate"):
        sweeps += SWEEPS * case["reals"]
    if kind == "chains":
        sweeps += case["chains"] * (case["equil"] + case["samples"])
    if kind == "gradient":
        sweeps += case["chains"] * (case["equil"] + case["meas"])
    flops = (FLOPS_3D if kind == "fill3" else FLOPS_2D) * gaps * sweeps
    lanes = case.get("reals", case.get("chains", 1))
    # inputs and outputs once, and the realizations' states once
    return {"bytes": 9.0 * n + state * gaps * lanes + 12.0 * blocks, "flops": flops}


# ------------------------------------------------------------------ exact --
def exact(case, seed):
    """Block statistics in 64 bits; None for the Monte Carlo results, which
    depend on every rounding of their chains."""
    kind = case["kind"]
    if kind not in ("create", "stats"):
        return None
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 13)
    v, m = _fields({"fields": 1, **case}, gen)[0]
    h, w, lb = case["h"], case["w"], case["block"]
    nby, nbx = -(-h // lb), -(-w // lb)
    ok = m == 0
    lo, hi = v[ok].min().double(), v[ok].max().double()
    phi = torch.where(ok, v.double() - lo, torch.zeros((), dtype=torch.float64, device=DEV))
    phi *= 2.0 * math.pi / (hi - lo)
    block = ((torch.arange(h, device=DEV) // lb)[:, None] * nbx
             + (torch.arange(w, device=DEV) // lb)[None, :])

    def per_block(x, b):
        return torch.zeros(nby * nbx, dtype=torch.float64, device=DEV).index_add_(
            0, b.reshape(-1), x.double().reshape(-1))

    Es = Nsp = Nb = 0.0
    for a, b in ((slice(None), slice(None, -1)), (slice(None, -1), slice(None))):
        c, d = (a, slice(1, None)) if a == slice(None) else (slice(1, None), b)
        both = ok[a, b] & ok[c, d]
        Es = Es - per_block(torch.cos(0.5 * (phi[a, b] - phi[c, d])) * both, block[a, b])
        Nsp = Nsp + per_block(both, block[a, b])
        Nb = Nb + per_block(torch.ones_like(both), block[a, b])
    ns = per_block(ok, block)
    mean = torch.where(ns > 0, per_block(phi, block) / ns.clamp_min(1), phi.sum() / ok.sum())
    whole = {k: x.to(torch.int32) for k, x in
             {"Nsp": Nsp, "Nb": Nb, "n_gap": per_block(~ok, block)}.items()}
    out = {"Es": Es, "mean_angle": mean, **whole}
    if kind == "stats":
        out["zrange"] = torch.stack([lo, hi])
    return out
