"""The slot's word window (one Philox block) at the counts where it can lose a
word: every number of words left, sections that read four, and photons that
leave the grid without reading any (no attenuation at their energy)."""
import numpy as np
import pytest

import oracle
import workloads as W

from gpu_helpers import Session, compare_histories

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e_res,gap_mode", [(0.0, 0), (0.112, 0), (0.112, 1), (0.0, 2), (0.112, 2)])
@pytest.mark.parametrize("clear_below", [0.0, 470.0])
def test_words_match_the_oracle(e_res, gap_mode, clear_below):
    sc = W.scanner_small(n_crystals=64, n_rings=8, n_tof=5, radius=200.0, ring_pitch=12.0, module_t=8, module_a=4, e_lo=300.0)
    sc.e_res, sc.gap_mode, sc.gap_t, sc.gap_a = e_res, gap_mode, 4.0, 3.0
    mats = W.standard_materials()
    for m in mats:  # below clear_below nothing attenuates: photons fly on without a step's words
        for t in (m.compton, m.rayleigh, m.photo):
            t[: int(clear_below)] = 0.0
        m.rayleigh *= 40.0  # as many Rayleigh as Compton events: three- and four-word sections mixed
    ph = W.phantom_water_cylinder(dims=(24, 24, 16), voxel=(8.0, 8.0, 6.0), radius=90.0, half_length=48.0)
    lut = W.lut_smooth(8, 6, 6, sc.n_tpos, sc.n_apos, 200.0)
    s = Session(sc, mats, ph, lut)
    try:
        n = 150_000
        gpu = s.run(17, 5, n, bin_mask=3)
        ref = oracle.simulate(sc, mats, ph, lut, 17, 5, n, bin_mask=3, threads=4)
        assert np.count_nonzero(ref["key"] >= 0) > 100
        compare_histories(gpu, ref)
    finally:
        s.close()
