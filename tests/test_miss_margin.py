"""The axial margin beyond which a straight line counts as missing the detector
(make_job), against the FP32 arithmetic it has to cover: up to 64 rounded steps
along the line, then the hit on the cylinder.  Also for scanners far longer
than wide, where a small transverse error moves the hit's z the most; there a
production launch, which ends such histories at once, has to bin what a listmode
launch does, which follows them."""
import numpy as np
import pytest

import workloads as W

F = np.float32
STEPS = 64


def _hit_z(x, y, z, dx, dy, dz, r2):
    a = dx * dx + dy * dy
    b = x * dx + y * dy
    c = x * x + y * y - r2
    sq = np.sqrt(np.maximum(b * b - a * c, F(0)))
    t = np.where(b >= 0, -c / np.where(b >= 0, b + sq, F(1)), (sq - b) / a)
    return z + t * dz


@pytest.mark.parametrize("half_over_radius", [0.02, 0.4, 4.0, 40.0, 1000.0])
@pytest.mark.parametrize("zmax_over_half", [0.3, 1.0, 3.0])
def test_rounded_lines_stay_within_the_margin(half_over_radius, zmax_over_half):
    rng = np.random.default_rng(int(half_over_radius * 100))
    n, R = 200_000, 311.8
    half = half_over_radius * R
    zmax = zmax_over_half * half
    margin = (R + half + zmax) / 512.0
    # emission points out to 0.95 R, lines that meet the cylinder around the scanner's end
    rho, th = 0.95 * R * np.sqrt(rng.uniform(0.5, 1.0, n)), rng.uniform(0, 2 * np.pi, n)
    x, y, z = rho * np.cos(th), rho * np.sin(th), rng.uniform(-zmax, zmax, n)
    phi = rng.uniform(0, 2 * np.pi, n)
    b = x * np.cos(phi) + y * np.sin(phi)
    chord = -b + np.sqrt(b * b - (x * x + y * y - R * R))
    target = np.where(rng.random(n) < 0.5, -1.0, 1.0) * (half + rng.uniform(0.0, 3.0, n) * margin)
    cot = (target - z) / chord
    st = 1.0 / np.sqrt(1.0 + cot * cot)
    dx, dy, dz = F(st * np.cos(phi)), F(st * np.sin(phi)), F(st * cot)
    px, py, pz = F(x), F(y), F(z)
    r2 = F(R * R)
    # the test at emission: za + (sq - b) dz against lim a
    a = dx * dx + dy * dy
    bb = px * dx + py * dy
    c = px * px + py * py - r2
    sq = np.sqrt(np.maximum(bb * bb - a * c, F(0)))
    misses = np.abs(pz * a + (sq - bb) * dz) > F(half + margin) * a
    # steps to the grid's edge at 0.95 R (and zmax), each rounded once (a fused multiply-add)
    inside = np.minimum(-b + np.sqrt(np.maximum(b * b - (x * x + y * y - (0.95 * R) ** 2), 0.0)),
                        st * np.abs((np.sign(dz) * zmax - z) / np.where(dz == 0, 1, dz))) / st
    for _ in range(STEPS):
        d = F(np.abs(inside) / STEPS * rng.uniform(0.0, 1.0, n))
        px, py, pz = (F(p.astype(np.float64) + d.astype(np.float64) * v.astype(np.float64)) for p, v in ((px, dx), (py, dy), (pz, dz)))
    hit = _hit_z(px, py, pz, dx, dy, dz, r2)
    assert misses.any() and not misses.all()
    assert np.all(np.abs(hit[misses]) > half)
    # and by far: no hit lies further from the exact line than a quarter of the margin
    ddx, ddy, ddz = (v.astype(np.float64) for v in (dx, dy, dz))
    exact = _hit_z(F(x).astype(np.float64), F(y).astype(np.float64), F(z).astype(np.float64), ddx, ddy, ddz, np.float64(R * R))
    assert np.max(np.abs(hit - exact)[misses]) < margin / 4.0


@pytest.mark.gpu
@pytest.mark.parametrize("ring_pitch", [100.0, 1500.0])     # half lengths of 40 and 600 radii
@pytest.mark.parametrize("bin_mask", [1, 2, 3])
def test_long_scanner_bins_what_listmode_does(ring_pitch, bin_mask):
    from gpu_helpers import Session, sinogram_from
    sc = W.scanner_small(n_crystals=48, n_rings=24, n_tof=5, radius=30.0, ring_pitch=ring_pitch, e_lo=200.0)
    # the grid's corners at 0.94 of the radius, its ends beyond the scanner's
    ph = W.phantom_water_cylinder(dims=(16, 16, 26), voxel=(2.5, 2.5, ring_pitch), radius=28.0, half_length=13.0 * ring_pitch)
    s = Session(sc, W.standard_materials(), ph, W.lut_smooth(8, 6, 6, sc.n_tpos, sc.n_apos, sc.e_lo))
    try:
        n = 400_001
        lm = s.run(23, 1, n, bin_mask=bin_mask)
        exp = sinogram_from(lm["key"], lm["q"], lm["cls"], sc.n_bins, [c for c, b in ((7, 1), (6, 2)) if bin_mask & b])
        assert np.count_nonzero(exp) > 0
        s.zero()
        s.run(23, 1, n, listmode=False, stats=False, bin_mask=bin_mask)
        np.testing.assert_array_equal(s.acc().cpu().numpy(), exp)
    finally:
        s.close()
