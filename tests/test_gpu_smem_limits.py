"""Two host threads with a context each run the same kernels with different
amounts of shared memory.  The limit on dynamic shared memory belongs to a
kernel on its device, so neither thread's launch may lower it under the
other's: every call is accepted, and gives the bits it gives alone."""
import threading

import numpy as np
import pytest

import paper_2509_05047_gb300 as psc
import workloads as W

pytestmark = pytest.mark.gpu


def _finalize(n_crystals, n_rad, n_rings, n_tof, sigma):
    import torch
    sc = W.scanner_small(n_crystals=n_crystals, n_rings=n_rings, n_tof=n_tof, n_rad=n_rad)
    ctx = psc.psc_create(0)
    scanner = psc.psc_load_scanner(ctx, psc.scanner_desc(sc))
    sums = torch.from_numpy(np.random.default_rng(n_tof).integers(0, 1 << 40, size=sc.n_bins)).cuda()
    acc = psc.psc_acc_wrap(ctx, scanner, sums)
    out = torch.empty(sc.shape, dtype=torch.float64, device="cuda")
    return ctx, out, lambda stream: psc.psc_finalize(ctx, psc.finalize_args(acc, sigma=sigma, scale=1e-6), out, stream), sums


def _simulate(materials):
    import torch
    sc = W.scanner_tiny()
    ctx = psc.psc_create(0)
    scanner = psc.psc_load_scanner(ctx, psc.scanner_desc(sc))
    mats = psc.psc_load_materials(ctx, psc.materials_desc(W.standard_materials()[:materials]).desc)
    ph = W.phantom_water_cylinder(dims=(8, 8, 8), voxel=(20.0, 20.0, 10.0), radius=60.0)
    phantom = psc.psc_load_phantom(ctx, psc.phantom_desc(ph).desc, mats)
    out = torch.zeros(sc.n_bins, dtype=torch.int64, device="cuda")
    acc = psc.psc_acc_wrap(ctx, scanner, out)

    def call(stream):
        psc.psc_acc_zero(ctx, acc, stream)
        psc.psc_simulate(ctx, psc.sim_args(3, 0, 500, scanner, phantom, acc, bin_mask=3), stream=stream)
    return ctx, out, call, ph


@pytest.mark.parametrize("small,large,calls", [
    (lambda: _finalize(40, 25, 2, 1, (6.0, 0.5, 0.5)), lambda: _finalize(40, 25, 2, 120, (6.0, 0.5, 0.5)), 4000),   # radial lines: 2 and 77 KB
    (lambda: _finalize(8, 7, 2, 5, (9.0, 0.5, 2.0)), lambda: _finalize(8, 7, 34, 5, (9.0, 0.5, 2.0)), 4000),        # axial tiles: 2 and 34 KB
    (lambda: _finalize(8, 7, 40, 5, (9.0, 0.5, 2.0)), lambda: _finalize(8, 7, 90, 5, (9.0, 0.5, 2.0)), 2000),       # half-width tiles: 20 and 45 KB
    (lambda: _simulate(2), lambda: _simulate(4), 3000),                                                             # two and four materials' tables
], ids=["lines", "tiles", "narrow_tiles", "transport"])
def test_calls_of_two_threads_are_accepted(small, large, calls):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    work, errors = [small(), large()], []
    try:
        alone = []
        for _, out, call, _ in work:
            call(torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            alone.append(out.clone())
            out.zero_()
        torch.cuda.synchronize()

        def run(w, stream):
            try:
                for i in range(calls):
                    w[2](stream.cuda_stream)
                    if i % 50 == 49:
                        stream.synchronize()
            except psc.PscError as e:
                errors.append(str(e))
        threads = [threading.Thread(target=run, args=(w, torch.cuda.Stream())) for w in work]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert errors == []
        for w, a in zip(work, alone):
            assert torch.equal(w[1], a)
    finally:
        for w in work:
            psc.psc_destroy(w[0])
