"""The unsmoothed estimate's two FP64 products are computed from integer
significands: every bit must be IEEE's, over counts beyond 53 bits, products
that round up into a new exponent, ties, and factors outside the normal range."""
import math

import numpy as np
import pytest

import workloads as W

from test_gpu_finalize import Fin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tof,per_lor", [(1, True), (5, True), (5, False)])
@pytest.mark.parametrize("scale", [1.0, -0.37, 1e-9, 2.0**32 * (1 - 2.0**-53), 2.0**-990, 5e-310, 0.0, 1e300])
def test_products_are_ieee(n_tof, per_lor, scale):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=38, n_rings=3, n_tof=n_tof, n_rad=33)   # 627 n_tof bins a plane: odd, ragged
    f = Fin(sc)
    try:
        rng = np.random.default_rng(3)
        n = sc.n_bins
        acc = rng.integers(0, 1 << 62, size=n) >> rng.integers(0, 62, size=n)
        acc[rng.uniform(size=n) < 0.3] = 0
        acc[:70] = [(1 << k) - 1 for k in range(1, 64)] + [(1 << 53) + 1, (1 << 53) + 3, (1 << 54) + 2, 0, 0, 1, 3]
        shape = sc.lor_shape if per_lor else sc.shape
        sens = rng.uniform(0.5, 1.5, size=shape)
        flat = sens.ravel()
        k = rng.integers(0, flat.size, size=flat.size // 4)
        flat[k] = rng.choice([0.0, -0.0, -1.25, 5e-324, 1e-310, 1e308, np.inf, -np.inf, np.nan, 2.0**-1022,
                              1 - 2.0**-53, 1 + 2.0**-52], size=k.size)
        f.write_acc(acc.reshape(sc.shape))
        with np.errstate(all="ignore"):
            plain = acc.astype(np.float64).reshape(sc.shape) * math.ldexp(scale, -32)
            exp = plain * (sens[..., None] if per_lor else sens)
        np.testing.assert_array_equal(f.run(scale=scale).cpu().numpy().view(np.int64), plain.view(np.int64))
        got = f.run(sens=f.sino(sens, per_lor), scale=scale).cpu().numpy()
        nan = np.isnan(exp)
        np.testing.assert_array_equal(np.isnan(got), nan)
        np.testing.assert_array_equal(got.view(np.int64)[~nan], exp.view(np.int64)[~nan])
    finally:
        f.close()


@pytest.mark.parametrize("density", [1.0, 0.6, 0.05, 0.0])   # all of a lane's bins filled, about half, few, none
@pytest.mark.parametrize("n_tof", [1, 5])                    # 627 and 3135 bins a plane: less and more than a CTA's 2048
def test_filled_bins_in_any_number(density, n_tof):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = W.scanner_small(n_crystals=38, n_rings=3, n_tof=n_tof, n_rad=33)
    f = Fin(sc)
    try:
        rng = np.random.default_rng(8)
        acc = rng.integers(1, 1 << 40, size=sc.shape)
        acc[rng.uniform(size=sc.shape) >= density] = 0
        sens = rng.uniform(0.5, 1.5, size=sc.lor_shape)
        sens.ravel()[::97] = np.inf
        f.write_acc(acc)
        with np.errstate(all="ignore"):
            exp = (acc.astype(np.float64) * math.ldexp(0.37, -32)) * sens[..., None]
        got = f.run(sens=f.sino(sens, True), scale=0.37).cpu().numpy()
        np.testing.assert_array_equal(got, exp)
    finally:
        f.close()
