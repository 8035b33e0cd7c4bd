"""The workloads that this library's speed is judged by.

A case is one call, or one short sequence of calls, that a user of the scatter
simulator makes again and again: transport of a slice of histories, a whole
iteration of the joint activity / scatter estimation, the finalize of an
accumulated sinogram, and the exact post-processing of accumulators.  Sizes
are those of the repository's configurations: a test-sized scanner (64
crystals x 8 rings), the small one (288 x 16, 13 TOF bins, 425-650 keV) and
the paper-scale one (448 x 45, up to 27 TOF bins with a 400 ps blur, 300-650
keV), with phantoms from 64 x 64 x 32 to 192 x 192 x 120 voxels, history
budgets from 1e4 to 1e9 and smoothing widths from none to the paper's upper
bound.  Where three copies of a paper-scale sinogram and its working memory
would not fit on the card, the TOF axis is mashed to 9 bins or fewer.

Accumulators are the caller's device tensors (psc_acc_wrap).  A simulation
case adds the next slice of histories to its accumulator on every pass, as a
program that extends a simulation does, so no pass repeats another.
"""
from __future__ import annotations

import functools
import math
import weakref
from types import SimpleNamespace

import numpy as np
import torch

import paper_2509_05047_gb300 as psc

MM_PER_PS = 0.299792458
FWHM = 2.0 * math.sqrt(2.0 * math.log(2.0))
# the widths of the paper's Sec. 2.3.2 (FWHM 9 / 6 / 10.5 bins: the chosen ones) and its upper bound
PAPER_SIGMA = (9.0 / FWHM, 6.0 / FWHM, 10.5 / FWHM)
UPPER_SIGMA = (4.25, 2.12, 7.64)
LUT_DTYPES = {"f32": psc.PSC_LUT_F32, "f16": psc.PSC_LUT_F16, "bf16": psc.PSC_LUT_BF16}


def listed():
    return [
        # the smallest whole estimate: a test-sized scanner and 20,000 histories (latency and launches)
        _step("step_test_scanner", "test", (40, 40, 16), 20_000, sigma=(1.0, 1.0, 1.0)),
        # one iteration of the joint estimation on the small scanner: new activity, 1e6 histories, smoothed estimate
        _step("iteration_small_1e6", "small", (64, 64, 32), 1_000_000, sigma=(2.0, 2.0, 2.0), update=True),
        # the plain method's small configuration: 1e6 histories through the f32 LUT
        _simulate("simulate_small_1e6", "small", (64, 64, 32), 1_000_000, "f32"),
        # low-count estimate at paper scale with the half-precision LUT
        _simulate("simulate_paper_f16_1e7", "paper", (128, 128, 89), 10_000_000, "f16"),
        # the headline workload: 1e9 histories of the torso through the paper-scale scanner
        _simulate("simulate_paper_1e9", "paper", (128, 128, 89), 1_000_000_000, "f32"),
        # gaps between modules and blocks, with the crystals' energy resolution
        _simulate("simulate_gaps_eres_1e8", "gaps", (128, 128, 89), 100_000_000, "f32", tof=9, e_res=0.112),
        # uneven requests (phantom sizes, budgets over three decades) in one launch
        {"name": "batch_uneven_6", "kind": "batch", "requests": 6, "lo": 96, "hi": 192, "budget_lo": 200_000,
         "budget_hi": 100_000_000},
        # the finalize of the headline workload, TOF bins mashed 3 to 1: sigma 2, per-LOR sensitivity
        _finalize("finalize_paper_tof9", 448, 45, 9, (2.0, 2.0, 2.0)),
        # a scanner without TOF at the paper's chosen widths, with the smoothing normalisation
        _finalize("finalize_nontof_norm", 448, 45, 1, PAPER_SIGMA, norm=True),
        # no smoothing: the sensitivity product alone
        _finalize("finalize_plain_small", 288, 16, 13, None),
        # the sensitivity sinogram's average over the scanner's 28 module rotations
        {"name": "rotate_paper_tof5", "kind": "rotate", "crystals": 448, "rings": 45, "n_rad": 447, "tof": 5, "step": 16},
        # mashing a sinogram to fewer counts per estimate: two views to one, then ring differences in threes
        {"name": "mash_span_paper_tof5", "kind": "mash", "crystals": 448, "rings": 45, "n_rad": 447, "tof": 5,
         "view_factor": 2, "tof_factor": 1, "span": 3},
    ]


def draw(rng):
    kind = rng.choice(["simulate", "simulate", "simulate", "step", "batch", "finalize", "finalize", "finalize",
                       "rotate", "mash"])
    side, nz = rng.randint(40, 160), rng.randint(16, 96)
    if kind == "simulate":
        scanner = rng.choice(["test", "small", "paper", "paper", "gaps"])
        tof = {"test": 7, "small": 13, "paper": rng.choice([1, 5, 9, 13, 27]), "gaps": rng.choice([1, 5, 9])}[scanner]
        return _simulate(None, scanner, (side, side, nz), _log_int(rng, 1e4, 3e8), rng.choice(["f32", "f32", "f16", "bf16", "none"]),
                         tof=tof, e_res=rng.choice([0.0, 0.0, 0.112]))
    if kind == "step":
        return _step(None, rng.choice(["test", "small"]), (min(side, 96), min(side, 96), min(nz, 64)), _log_int(rng, 1e4, 3e7),
                     sigma=rng.choice([(1.0, 1.0, 1.0), (2.0, 2.0, 2.0), PAPER_SIGMA]), update=rng.random() < 0.5)
    if kind == "batch":
        lo = rng.randint(64, 120)
        return {"kind": "batch", "requests": rng.randint(2, 6), "lo": lo, "hi": rng.randint(lo, 192),
                "budget_lo": _log_int(rng, 1e5, 1e6), "budget_hi": _log_int(rng, 2e6, 1e8)}
    # sinogram shapes: even crystal counts whose views need not be even, whole or clipped radial axes,
    # at most the bins of the largest listed finalize
    crystals = 2 * rng.randint(19, 224)
    n_rad = crystals - 1 - 2 * rng.choice([0, 0, rng.randint(1, crystals // 5)])
    rings, tof = rng.randint(4, 45), rng.choice([1, 1, 3, 5, 9, 13, 27])
    if kind == "rotate":
        divisors = [d for d in range(2, crystals // 2 + 1) if crystals % d == 0]
        small = [d for d in divisors if d >= crystals // 40] or divisors
        return {"kind": "rotate", "crystals": crystals, "rings": rings, "n_rad": n_rad,
                "tof": _fit(crystals, n_rad, rings, tof, 1.0e9), "step": rng.choice(small)}
    if kind == "mash":
        V = crystals // 2
        tof = _fit(crystals, n_rad, rings, tof, 1.0e9)
        return {"kind": "mash", "crystals": crystals, "rings": rings, "n_rad": n_rad, "tof": tof,
                "view_factor": rng.choice([f for f in (1, 2, 3, 4, 5, 7, 8) if V % f == 0]),
                "tof_factor": rng.choice([f for f in (1, 3, 9) if tof % f == 0]), "span": rng.choice([3, 5, 7])}
    return _finalize(None, crystals, rings, _fit(crystals, n_rad, rings, tof, 1.8e9),
                     rng.choice([None, (2.0, 2.0, 2.0), (2.0, 2.0, 2.0), (0.7, 1.3, 0.0), (4.0, 4.0, 4.0), PAPER_SIGMA, UPPER_SIGMA]),
                     norm=rng.random() < 0.3, sens_first=rng.random() < 0.2, n_rad=n_rad)


def prepare(case, seed):
    return {"simulate": _prepare_simulate, "step": _prepare_step, "batch": _prepare_batch, "finalize": _prepare_finalize,
            "rotate": _prepare_post, "mash": _prepare_post}[case["kind"]](case, seed)


def run(state):
    return state.run(state)


def work(case):
    """Bytes: inputs and outputs once.  Operations of a simulation: the modelled
    lane operations per history (Philox blocks, steps, rejection tries,
    interactions, detections) at the counts of the torso workload."""
    if case["kind"] in ("simulate", "step"):
        n = case["histories"]
        b = {"bytes": 16.0 * 0.04 * n + 16.0 * case["nx"] * case["ny"] * case["nz"], "flops": 850.0 * n}
        if case["kind"] == "step":  # zeroing, then the finalize
            bins = _bins(_scanner(case))
            b["bytes"] += 8.0 * bins + 16.0 * bins + 8.0 * bins / _scanner(case).n_tof
            b["flops"] += bins * _taps(case)
        return b
    if case["kind"] == "batch":
        n = sum(_budgets(case))
        return {"bytes": 16.0 * 0.04 * n, "flops": 850.0 * n}
    sc = _sinogram_scanner(case)
    bins = _bins(sc)
    if case["kind"] == "finalize":
        factors = 8.0 * bins / sc.n_tof * (2 if case["norm"] else 1)
        return {"bytes": 16.0 * bins + factors, "flops": bins * (2.0 + _taps(case))}
    if case["kind"] == "rotate":
        return {"bytes": 16.0 * bins, "flops": bins}
    planes = bins / sc.n_rings ** 2
    spanned = planes * _span_planes(sc.n_rings, case["span"])
    mashed = bins / case["view_factor"] / case["tof_factor"]
    return {"bytes": 8.0 * (2.0 * bins + mashed + spanned), "flops": 2.0 * bins}


def exact(case, seed):
    """The finalize in 64 bits (torch).  Simulations and post-processing give whole numbers."""
    if case["kind"] != "finalize":
        return None
    sc = _sinogram_scanner(case)
    shape = (sc.n_rings ** 2, sc.n_crystals // 2, sc.n_rad, sc.n_tof)
    x = _accumulator(sc, seed, case["density"]).view(shape).double().mul_(math.ldexp(_scale(case), -32))
    sens = torch.from_numpy(_sensitivity(sc)).cuda()[..., None]
    norm = torch.from_numpy(_normalisation(sc)).cuda()[..., None] if case["norm"] else None
    if case["sens_first"]:
        x *= sens
    if case["smooth"]:
        if norm is not None:
            x *= norm
        x = _smooth64(_smooth64(x, 2, case["sigma_r"]), 1, case["sigma_v"])
        n = sc.n_rings
        for d in range(1 - n, n):  # the planes of one ring difference
            planes = [ra * n + ra + d for ra in range(max(0, -d), min(n, n - d))]
            x[planes] = _smooth64(x[planes], 0, case["sigma_a"])
        if norm is not None:
            x /= norm
    if not case["sens_first"]:
        x *= sens
    return x


# ---------------------------------------------------------------------------
# case dicts
# ---------------------------------------------------------------------------
def _named(name, d):
    return {"name": name, **d} if name else d


def _simulate(name, scanner, dims, histories, lut, tof=0, e_res=0.0):
    return _named(name, {"kind": "simulate", "scanner": scanner, "nx": dims[0], "ny": dims[1], "nz": dims[2],
                         "histories": histories, "lut": lut, "tof": tof, "e_res": e_res})


def _widths(sigma):
    s = sigma or (0.0, 0.0, 0.0)
    return {"smooth": sigma is not None, "sigma_r": s[0], "sigma_v": s[1], "sigma_a": s[2]}


def _step(name, scanner, dims, histories, sigma, update=False):
    return _named(name, {"kind": "step", "scanner": scanner, "nx": dims[0], "ny": dims[1], "nz": dims[2],
                         "histories": histories, "lut": "f32", "tof": 0, "e_res": 0.0, "update": update, **_widths(sigma)})


def _finalize(name, crystals, rings, tof, sigma, norm=False, sens_first=False, n_rad=0):
    return _named(name, {"kind": "finalize", "crystals": crystals, "rings": rings, "tof": tof, "n_rad": n_rad or crystals - 1,
                         "norm": bool(norm and sigma), "sens_first": bool(sens_first), "density": 0.02, **_widths(sigma)})


def _log_int(rng, lo, hi):
    return int(round(10 ** rng.uniform(math.log10(lo), math.log10(hi))))


def _fit(crystals, n_rad, rings, tof, most):
    """The largest of the usual TOF bin counts, at most `tof`, that keeps the sinogram within `most` bins."""
    per = rings * rings * (crystals // 2) * n_rad
    return max(t for t in (1, 3, 5, 9, 13, 27) if t <= tof and (t == 1 or per * t <= most))


def _taps(case):
    if not case["smooth"]:
        return 0.0
    return sum(2.0 * (2 * math.ceil(4.0 * case[k]) + 1) for k in ("sigma_r", "sigma_v", "sigma_a"))


def _scale(case):
    return 1e-9


def _span_planes(n, span):
    h, total = (span - 1) // 2, 0
    for k in range(-((n - 1 + h) // span), (n - 1 + h) // span + 1):
        lo, hi = max(k * span - h, 1 - n), min(k * span + h, n - 1)
        m = 0 if lo <= 0 <= hi else min(abs(lo), abs(hi))
        total += (2 * n - 2 - 2 * m) // (1 if hi > lo else 2) + 1
    return total


# ---------------------------------------------------------------------------
# scanners, materials, phantoms, LUTs, sinograms
# ---------------------------------------------------------------------------
def _scanner(case):
    blur = MM_PER_PS * 400.0 / 2.0 / FWHM
    base = dict(n_rad=0, e_res=case["e_res"], gap_mode=0, gap_t=2.0, gap_a=2.0, crystal_depth=25.0, doi=7.0, mu_block=0.0869)
    if case["scanner"] == "test":
        base.update(radius=200.0, ring_pitch=6.0, n_crystals=64, n_rings=8, module_t=4, module_a=2, e_lo=350.0, e_hi=650.0,
                    n_tof=7, tof_bin_mm=30.0, tof_sigma_mm=20.0)
    elif case["scanner"] == "small":
        base.update(radius=310.0, ring_pitch=4.0, n_crystals=288, n_rings=16, module_t=4, module_a=4, e_lo=425.0, e_hi=650.0,
                    n_tof=13, tof_bin_mm=50.0, tof_sigma_mm=0.0)
    else:
        tof = case["tof"] or 27
        base.update(radius=311.8, ring_pitch=250.4 / 45, n_crystals=448, n_rings=45, module_t=16, module_a=9, e_lo=300.0,
                    e_hi=650.0, n_tof=tof, tof_bin_mm=27 * 24.0 / tof, tof_sigma_mm=blur)
        if case["scanner"] == "gaps":
            base["gap_mode"] = 2
    if case["e_res"] > 0.0:
        base["e_lo"] = 425.0
    sc = SimpleNamespace(**base)
    sc.n_rad = sc.n_crystals - 1
    return sc


def _sinogram_scanner(case):
    return SimpleNamespace(radius=311.8, ring_pitch=250.4 / 45, n_crystals=case["crystals"], n_rings=case["rings"], module_t=1,
                           module_a=1, e_lo=300.0, e_hi=650.0, n_tof=case["tof"], n_rad=case["n_rad"], tof_bin_mm=24.0,
                           tof_sigma_mm=0.0)


def _bins(sc):
    return sc.n_rings ** 2 * (sc.n_crystals // 2) * sc.n_rad * sc.n_tof


@functools.lru_cache(maxsize=None)
def _materials():
    """Vacuum, water, lung and bone on the 1 keV grid: Klein-Nishina totals, E^-3 photoelectric and E^-2 Rayleigh parts."""
    e = np.maximum(np.arange(513, dtype=np.float64), 1.0)
    a = e / 511.0
    log = np.log1p(2.0 * a)
    kn = 2.0 * math.pi * 2.8179403262e-13 ** 2 * ((1.0 + a) / a ** 2 * (2.0 * (1.0 + a) / (1.0 + 2.0 * a) - log / a)
                                                   + log / (2.0 * a) - (1.0 + 3.0 * a) / (1.0 + 2.0 * a) ** 2)
    made = [SimpleNamespace(compton=0.0 * e, rayleigh=0.0 * e, photo=0.0 * e, kappa=0.0)]
    for z_over_a, photo, rayleigh, kappa in ((10.0 / 18.01528, 2.76e-3, 2.76e-3, 500.0), (10.0 / 18.01528, 2.76e-3, 2.76e-3, 500.0),
                                             (0.5148, 1.9e-2, 5.0e-3, 800.0)):
        made.append(SimpleNamespace(compton=z_over_a * 6.02214076e23 * kn, rayleigh=rayleigh * (e / 100.0) ** -2,
                                    photo=photo * (e / 100.0) ** -3, kappa=kappa))
    return made


def _torso(dims, fov, seed):
    """A water ellipse of the whole axial length with lungs, a spine and six seeded hot spheres: (phantom, activity)."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = dims
    voxel = (fov / nx, fov / ny, 2.78)
    ax = [(torch.arange(n, device="cuda", dtype=torch.float32) + 0.5 - n / 2.0) * d for n, d in zip(dims, voxel)]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    a, b = 0.47 * fov, 0.33 * fov
    body = ((x / a) ** 2 + (y / b) ** 2 <= 1.0).expand(nz, ny, nx)
    material = body.to(torch.uint8)
    density = body.float()
    activity = body.float()
    for side in (-1.0, 1.0):
        lung = body & (((x - side * 0.41 * a) / (0.28 * a)) ** 2 + ((y - 0.1 * b) / (0.5 * b)) ** 2 + (z / (1.07 * nz)) ** 2 <= 1.0)
        material = material.masked_fill(lung, 2)
        density = density.masked_fill(lung, 0.3)
        activity = activity.masked_fill(lung, 0.3)
    spine = body & (x ** 2 + (y + 0.66 * b) ** 2 <= (0.11 * a) ** 2)
    material = material.masked_fill(spine, 3)
    density = density.masked_fill(spine, 1.9)
    activity = activity.masked_fill(spine, 0.5)
    for d in np.linspace(10.0, 37.0, 6):
        cx, cy, cz = rng.uniform(-0.4, 0.4) * a, rng.uniform(-0.3, 0.4) * b, rng.uniform(-0.3, 0.3) * nz * 2.78
        hot = body & ~spine & ((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2 <= (0.5 * d) ** 2)
        material = material.masked_fill(hot, 1)
        density = density.masked_fill(hot, 1.0)
        activity = activity.masked_fill(hot, 4.0 * rng.uniform(0.7, 1.3))
    return SimpleNamespace(dims=dims, voxel=voxel, origin=tuple(-0.5 * n * d for n, d in zip(dims, voxel)),
                           material=material.cpu().numpy(), density=density.cpu().numpy(), activity=activity.cpu().numpy())


@functools.lru_cache(maxsize=4)
def _lut(n_e, n_a, n_b, n_tpos, n_apos, e_min):
    """Smooth detection probabilities in [0.2, 1], one table per scanner."""
    def axis(n, lo, hi):
        return lo + (torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) * ((hi - lo) / n)
    t = torch.arange(n_tpos, device="cuda").float()[None, :, None, None, None] / n_tpos
    z = torch.arange(n_apos, device="cuda").float()[:, None, None, None, None] / n_apos
    e, a, b = axis(n_e, 0.0, 1.0)[:, None, None], axis(n_a, -1.0, 1.0)[:, None], axis(n_b, -1.0, 1.0)
    h = torch.sin(5.7 * e + 0.4) * torch.cos(3.3 * a + 1.1) * torch.cos(2.6 * b + 0.2) * (
        0.6 + 0.4 * torch.cos(6.28 * t + 0.9) * torch.cos(6.28 * z + 2.1))
    data = (0.6 + 0.4 * h).clamp(0.2, 1.0).contiguous().cpu().numpy()
    return SimpleNamespace(n_e=n_e, n_a=n_a, n_b=n_b, n_tpos=n_tpos, n_apos=n_apos, e_min=e_min, e_max=511.0, a_min=-90.0,
                           a_max=90.0, b_min=-90.0, b_max=90.0, data=data)


def _lut_for(case, sc):
    bins = (64, 32, 32) if case["scanner"] == "paper" else (16, 8, 8)
    if sc.gap_mode:
        positions = (sc.module_t + 2, sc.n_rings // sc.module_a * (sc.module_a + 2))
    else:
        positions = (sc.module_t, sc.module_a)
    return _lut(*bins, *positions, sc.e_lo)


@functools.lru_cache(maxsize=2)
def _lor_values(n_rings, views, n_rad, lo, hi, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.rand(n_rings * n_rings, views, n_rad, device="cuda", dtype=torch.float64, generator=g)
    return v.mul_(hi - lo).add_(lo).cpu().numpy()


def _sensitivity(sc):
    """Per-LOR scatter sensitivities of a scanner, uniform in [0.5, 1.5)."""
    return _lor_values(sc.n_rings, sc.n_crystals // 2, sc.n_rad, 0.5, 1.5, 1)


def _normalisation(sc):
    """Per-LOR smoothing normalisation of a scanner, uniform in [0.2, 2)."""
    return _lor_values(sc.n_rings, sc.n_crystals // 2, sc.n_rad, 0.2, 2.0, 2)


def _accumulator(sc, seed, density):
    """What a simulation leaves: int64 sums of weights in [0.04, 1] 2^32, `density` events per bin."""
    n = _bins(sc)
    g = torch.Generator(device="cuda").manual_seed(seed)
    acc = torch.zeros(n, dtype=torch.int64, device="cuda")
    left = int(n * density) + 1
    while left > 0:
        k = min(left, 1 << 24)
        at = torch.randint(0, n, (k,), device="cuda", generator=g)
        w = torch.rand(k, device="cuda", generator=g).mul_(0.96).add_(0.04).mul_(4294967296.0).to(torch.int64)
        acc.scatter_add_(0, at, w)
        left -= k
    return acc


# ---------------------------------------------------------------------------
# states and passes
# ---------------------------------------------------------------------------
class _State:
    """What a user's program keeps: a context with its loaded objects, released with the state."""

    def __init__(self):
        self.ctx = psc.psc_create(0)
        weakref.finalize(self, psc.psc_destroy, self.ctx)

    def stream(self):
        return torch.cuda.current_stream().cuda_stream


def _prepare_simulate(case, seed):
    s = _State()
    sc = _scanner(case)
    s.scanner = psc.psc_load_scanner(s.ctx, psc.scanner_desc(sc))
    materials = psc.psc_load_materials(s.ctx, psc.materials_desc(_materials()).desc)
    s.image = _torso((case["nx"], case["ny"], case["nz"]), 240.0 if case["scanner"] == "test" else 300.0, seed)
    s.phantom = psc.psc_load_phantom(s.ctx, psc.phantom_desc(s.image).desc, materials)
    s.lut = 0 if case["lut"] == "none" else psc.psc_load_lut(s.ctx, psc.lut_desc(_lut_for(case, sc), LUT_DTYPES[case["lut"]]).desc)
    s.sums = torch.zeros(_bins(sc), dtype=torch.int64, device="cuda")
    s.acc = psc.psc_acc_wrap(s.ctx, s.scanner, s.sums)
    s.seed, s.first, s.histories = 1000 + seed, 0, case["histories"]
    s.run = _run_simulate
    return s


def _run_simulate(s):
    args = psc.sim_args(s.seed, s.first, s.histories, s.scanner, s.phantom, s.acc, lut=s.lut)
    s.first += s.histories
    psc.psc_simulate(s.ctx, args, stream=s.stream())
    return s.sums


def _prepare_step(case, seed):
    s = _prepare_simulate(case, seed)
    sc = _scanner(case)
    s.sens = psc.psc_load_sinogram(s.ctx, s.scanner, _sensitivity(sc), True)
    s.estimate = torch.empty((sc.n_rings ** 2, sc.n_crystals // 2, sc.n_rad, sc.n_tof), dtype=torch.float64, device="cuda")
    s.sigma = (case["sigma_r"], case["sigma_v"], case["sigma_a"]) if case["smooth"] else None
    s.update = case["update"]
    s.run = _run_step
    return s


def _run_step(s):
    stream = s.stream()
    if s.update:
        psc.psc_update_activity(s.ctx, s.phantom, s.image.activity)
    psc.psc_acc_zero(s.ctx, s.acc, stream)
    psc.psc_simulate(s.ctx, psc.sim_args(s.seed, s.first, s.histories, s.scanner, s.phantom, s.acc, lut=s.lut), stream=stream)
    s.first += s.histories
    psc.psc_finalize(s.ctx, psc.finalize_args(s.acc, sens=s.sens, sigma=s.sigma, scale=1.0 / s.histories), s.estimate, stream)
    return {"estimate": s.estimate, "sums": s.sums}


def _budgets(case):
    """History budgets spread over the logarithm of their range, largest first."""
    n, lo, hi = case["requests"], case["budget_lo"], case["budget_hi"]
    return [int(round(hi * (lo / hi) ** (i / max(1, n - 1)))) for i in range(n)]


def _prepare_batch(case, seed):
    s = _State()
    rng = np.random.default_rng(seed)
    where = {"scanner": "small", "tof": 0, "e_res": 0.0}
    sc = _scanner(where)
    scanner = psc.psc_load_scanner(s.ctx, psc.scanner_desc(sc))
    materials = psc.psc_load_materials(s.ctx, psc.materials_desc(_materials()).desc)
    lut = psc.psc_load_lut(s.ctx, psc.lut_desc(_lut_for(where, sc)).desc)
    s.sums, s.args, s.budgets = [], [], _budgets(case)
    for i, n in enumerate(s.budgets):
        side, nz = int(rng.integers(case["lo"], case["hi"] + 1)), int(rng.integers(64, 121))
        image = _torso((side, side, nz), min(3.0, 400.0 / side) * side, seed + i)
        phantom = psc.psc_load_phantom(s.ctx, psc.phantom_desc(image).desc, materials)
        s.sums.append(torch.zeros(_bins(sc), dtype=torch.int64, device="cuda"))
        acc = psc.psc_acc_wrap(s.ctx, scanner, s.sums[-1])
        s.args.append((2000 + seed + i, scanner, phantom, acc, lut))
    s.passes = 0
    s.run = _run_batch
    return s


def _run_batch(s):
    args = [psc.sim_args(seed, s.passes * n, n, scanner, phantom, acc, lut=lut)
            for n, (seed, scanner, phantom, acc, lut) in zip(s.budgets, s.args)]
    s.passes += 1
    psc.psc_simulate_batch(s.ctx, args, stream=s.stream())
    return s.sums


def _prepare_finalize(case, seed):
    s = _State()
    sc = _sinogram_scanner(case)
    s.scanner = psc.psc_load_scanner(s.ctx, psc.scanner_desc(sc))
    s.sums = _accumulator(sc, seed, case["density"])
    s.acc = psc.psc_acc_wrap(s.ctx, s.scanner, s.sums)
    s.sens = psc.psc_load_sinogram(s.ctx, s.scanner, _sensitivity(sc), True)
    s.norm = psc.psc_load_sinogram(s.ctx, s.scanner, _normalisation(sc), True) if case["norm"] else 0
    s.sigma = (case["sigma_r"], case["sigma_v"], case["sigma_a"]) if case["smooth"] else None
    s.sens_first, s.scale = case["sens_first"], _scale(case)
    s.estimate = torch.empty((sc.n_rings ** 2, sc.n_crystals // 2, sc.n_rad, sc.n_tof), dtype=torch.float64, device="cuda")
    s.run = _run_finalize
    return s


def _run_finalize(s):
    psc.psc_finalize(s.ctx, psc.finalize_args(s.acc, sens=s.sens, norm=s.norm, sigma=s.sigma, scale=s.scale, sens_first=s.sens_first),
                     s.estimate, s.stream())
    return s.estimate


def _prepare_post(case, seed):
    s = _State()
    sc = _sinogram_scanner(case)
    s.scanner = psc.psc_load_scanner(s.ctx, psc.scanner_desc(sc))
    s.sums = _accumulator(sc, seed, 0.5)
    s.acc = psc.psc_acc_wrap(s.ctx, s.scanner, s.sums)
    V = sc.n_crystals // 2
    if case["kind"] == "rotate":
        s.step = case["step"]
        s.out = torch.zeros(_bins(sc), dtype=torch.int64, device="cuda")
        s.out_acc = psc.psc_acc_wrap(s.ctx, s.scanner, s.out)
        s.run = _run_rotate
        return s
    s.factors, s.span = (case["view_factor"], case["tof_factor"]), case["span"]
    planes = psc.psc_acc_span(s.ctx, s.acc, s.span)
    s.mashed = torch.empty((sc.n_rings ** 2, V // s.factors[0], sc.n_rad, sc.n_tof // s.factors[1]), dtype=torch.int64, device="cuda")
    s.spanned = torch.empty((planes, V, sc.n_rad, sc.n_tof), dtype=torch.int64, device="cuda")
    s.run = _run_mash
    return s


def _run_rotate(s):
    psc.psc_acc_rotate_sum(s.ctx, s.acc, s.step, s.out_acc, s.stream())
    return s.out


def _run_mash(s):
    psc.psc_acc_mash(s.ctx, s.acc, s.factors[0], s.factors[1], s.mashed, s.stream())
    psc.psc_acc_span(s.ctx, s.acc, s.span, s.spanned, s.stream())
    return {"mashed": s.mashed, "spanned": s.spanned}


def _smooth64(x, axis, sigma):
    """Gaussian of ceil(4 sigma) taps a side, normalised, edges reflected half-sample symmetrically."""
    if sigma <= 0.0:
        return x
    K, n = int(math.ceil(4.0 * sigma)), x.shape[axis]
    w = np.exp(-0.5 * (np.arange(-K, K + 1) / sigma) ** 2)
    w /= w.sum()
    out = torch.zeros_like(x)
    at = torch.arange(n, device=x.device)
    for k, g in zip(range(-K, K + 1), w):
        m = torch.remainder(at + k, 2 * n)
        out.add_(x.index_select(axis, torch.where(m >= n, 2 * n - 1 - m, m)), alpha=float(g))
    return out
