"""The plain finalize's two kernels, one bin a thread for few bins and eight for
more, on both sides of the line between them: IEEE products of every kind of
operand, all filled, half filled and sparse."""
import math

import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W

from gpu_kernels import kernels_of
from test_gpu_finalize import Fin

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [-1, 0])          # one plane fewer than a CTA of eight bins a thread for each SM, and as many
@pytest.mark.parametrize("per_lor", [True, False])
@pytest.mark.parametrize("scale", [1.0, -0.37, 1e-9, 2.0**32 * (1 - 2.0**-53), 2.0**-990, 5e-310, 0.0, 1e300])
@pytest.mark.parametrize("density", [1.0, 0.55, 0.02])
def test_products_are_ieee_on_both_sides(side, per_lor, scale, density):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rings = math.isqrt(sms + side)
    while rings * rings < sms + side + 1 and side == 0:
        rings += 1
    sc = W.scanner_small(n_crystals=38, n_rings=rings, n_tof=3, n_rad=33)   # 1881 bins a plane: one CTA's, ragged
    many = rings * rings >= sms
    f = Fin(sc)
    try:
        rng = np.random.default_rng(3)
        n = sc.n_bins
        acc = rng.integers(1, 1 << 62, size=n) >> rng.integers(0, 62, size=n)
        acc[rng.uniform(size=n) >= density] = 0
        acc[:70] = [(1 << k) - 1 for k in range(1, 64)] + [(1 << 53) + 1, (1 << 53) + 3, (1 << 54) + 2, 0, 0, 1, 3]
        sens = rng.uniform(0.5, 1.5, size=sc.lor_shape if per_lor else sc.shape)
        flat = sens.ravel()
        k = rng.integers(0, flat.size, size=flat.size // 4)
        flat[k] = rng.choice([0.0, -0.0, -1.25, 5e-324, 1e-310, 1e308, np.inf, -np.inf, np.nan, 2.0**-1022,
                              1 - 2.0**-53, 1 + 2.0**-52], size=k.size)
        f.write_acc(acc.reshape(sc.shape))
        with np.errstate(all="ignore"):
            plain = acc.astype(np.float64).reshape(sc.shape) * math.ldexp(scale, -32)
            exp = plain * (sens[..., None] if per_lor else sens)
        np.testing.assert_array_equal(f.run(scale=scale).cpu().numpy().view(np.int64), plain.view(np.int64))
        out = torch.full(sc.shape, -7.0, dtype=torch.float64, device="cuda")
        args = psc.finalize_args(f.a_id, sens=f.sino(sens, per_lor), scale=scale)
        names = kernels_of(lambda stream: psc.psc_finalize(f.ctx, args, out, stream))
        assert ("finalize_plain_kernel" in names) == many and ("finalize_plain_few_kernel" in names) != many
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        nan = np.isnan(exp)
        np.testing.assert_array_equal(np.isnan(got), nan)
        np.testing.assert_array_equal(got.view(np.int64)[~nan], exp.view(np.int64)[~nan])
    finally:
        f.close()
