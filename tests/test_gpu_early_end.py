"""Production launches end a history as soon as it is certain to add nothing
and follow its less likely photon first; listmode launches follow photon A,
then B, to the end.  Both must put the same weights into the same bins,
whatever is binned, near and far from the grid's and the scanner's edges."""
import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W

from gpu_helpers import Session, sinogram_from

pytestmark = pytest.mark.gpu


def _scanner(kind):
    if kind == "blur":
        return W.scanner_small(n_crystals=64, n_rings=8, n_tof=7, radius=200.0, ring_pitch=6.0, tof_bin_mm=30.0,
                               tof_sigma_mm=20.0, e_lo=350.0)
    if kind == "long":    # hardly any straight line misses
        return W.scanner_small(n_crystals=48, n_rings=24, n_tof=5, radius=150.0, ring_pitch=40.0, e_lo=300.0)
    if kind == "one_ring":  # nearly every straight line misses
        return W.scanner_small(n_crystals=64, n_rings=1, n_tof=3, radius=200.0, ring_pitch=4.0, tof_bin_mm=80.0, module_a=1)
    sc = W.scanner_small(n_crystals=64, n_rings=8, n_tof=5, radius=200.0, ring_pitch=8.0, module_t=8, module_a=4)
    sc.e_res, sc.gap_mode = 0.112, 2 if kind == "gaps" else 1
    sc.gap_t, sc.gap_a = 3.0, 2.0
    return sc


@pytest.mark.parametrize("kind,voxel", [("blur", 5.0), ("long", 5.0), ("one_ring", 5.0), ("gaps", 5.0), ("gaps_lost", 5.0),
                                        ("blur", 7.05)])   # 7.05 mm: the grid's corners lie beyond 0.95 of the radius
@pytest.mark.parametrize("bin_mask", [1, 2, 3])
def test_production_accumulator_equals_listmode(kind, voxel, bin_mask):
    sc = _scanner(kind)
    # the phantom reaches past the scanner's axial ends on the one-ring and the 48 mm scanners
    ph = W.phantom_water_cylinder(dims=(40, 40, 24), voxel=(voxel, voxel, 5.0), radius=75.0, half_length=60.0)
    lut = W.lut_smooth(8, 6, 6, sc.n_tpos, sc.n_apos, sc.e_lo)
    s = Session(sc, W.standard_materials(), ph, lut)
    try:
        n = 120_001
        lm = s.run(41, 3, n, bin_mask=bin_mask)
        exp = sinogram_from(lm["key"], lm["q"], lm["cls"], sc.n_bins, [c for c, b in ((7, 1), (6, 2)) if bin_mask & b])
        assert np.count_nonzero(exp) > 0
        np.testing.assert_array_equal(s.acc().cpu().numpy(), exp)
        for block in (0, 256):
            s.zero()
            s.run(41, 3, n, listmode=False, stats=False, bin_mask=bin_mask, block=block)
            np.testing.assert_array_equal(s.acc().cpu().numpy(), exp)
    finally:
        s.close()
