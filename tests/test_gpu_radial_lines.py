"""The radial pass of short TOF axes works on whole lines staged in shared
memory, two lines a thread: against the FP64 oracle, and the same bits for a
range of segments as for all planes."""
import numpy as np
import pytest

import oracle
import workloads as W

from test_gpu_finalize import Fin, SMOOTH_RTOL

pytestmark = pytest.mark.gpu


# crystals, radial bins, TOF bins: odd and even view counts (a pair without its second line), lines of one partial
# block of 8 rows, several CTAs a plane, longer TOF axes of small sinograms, and one of 224,000 columns, which the
# column kernel takes as a whole and this one for the segment range
@pytest.mark.parametrize("n_crystals,n_rad,n_tof", [(8, 7, 1), (10, 9, 3), (46, 33, 1), (46, 45, 4), (200, 199, 1), (44, 41, 5),
                                                     (22, 21, 27), (200, 9, 140)])
@pytest.mark.parametrize("radius", [0, 1, 5, 7])     # at most the shortest line
@pytest.mark.parametrize("factors", [None, "sens_first", "norm"])
def test_lines_match_oracle(n_crystals, n_rad, n_tof, radius, factors):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=n_crystals, n_rings=4, n_tof=n_tof, n_rad=n_rad)
    f = Fin(sc)
    try:
        rng = np.random.default_rng(radius)
        acc = rng.integers(0, 1 << 62, size=sc.shape) >> rng.integers(0, 62, size=sc.shape)
        acc[rng.uniform(size=sc.shape) < 0.3] = 0
        f.write_acc(acc)
        sens, norm = rng.uniform(0.5, 1.5, size=sc.lor_shape), rng.uniform(0.2, 2.0, size=sc.shape)
        sigma = (radius / 4.0, 0.0, 0.0)
        kw, host = dict(sigma=sigma, scale=0.37), {}
        if factors:
            kw["sens"], host["sens"] = f.sino(sens, True), sens
        if factors == "sens_first":
            kw["sens_first"], host["smooth_before_sensitivity"] = True, False
        if factors == "norm":
            kw["norm"], host["norm"] = f.sino(norm, False), norm
        got = f.run(**kw).cpu().numpy()
        np.testing.assert_allclose(got, oracle.finalize(acc, sc.n_rings, sigma=sigma, scale=0.37, **host), rtol=SMOOTH_RTOL,
                                   atol=1e-300)
        # a segment range starts its planes elsewhere: the same bits
        part = f.run(segments=(2, 4), **kw).cpu().numpy()
        for d in (-1, 0):
            for ra in range(max(0, -d), 4):
                np.testing.assert_array_equal(part[ra * 4 + ra + d], got[ra * 4 + ra + d])
    finally:
        f.close()
