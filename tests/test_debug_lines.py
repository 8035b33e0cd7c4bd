"""The debug build checks every index that the staged radial lines read a count
or a factor by: each read's index comes from a check, and a run with both factors
fires none and gives the release library's bits."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_read_of_the_lines_kernel_is_checked():
    text = open(os.path.join(ROOT, "paper_2509_05047_gb300", "csrc", "finalize.cu")).read()
    text = re.sub(r"//[^\n]*", "", text)
    body = text[text.index("smooth_radial_lines_kernel("):text.index("smooth_view_kernel(")]
    checked = set()
    for name, value in re.findall(r"const long long (\w+) = ([^;]*);", body):
        branches = value.split("?")[1].split(" : ") if "?" in value else [value]
        if all(b.strip().startswith("dbg_idx(") for b in branches):
            checked.add(name)
    reads = [a.split(",")[2].strip(" )") for a in re.findall(r"\bfactor\(([^;]*)\);", body)]
    assert len(reads) == 4 and all(r in checked for r in reads), (reads, checked)
    counts = re.findall(r"__ldg\(P\.acc \+ (\w+)", body)
    assert len(counts) == 2 and set(counts) == {"dbg_idx"}


_RUN = r'''
import sys
sys.path.insert(0, ".")
import numpy as np, torch
import paper_2509_05047_gb300 as psc
import workloads as W
stream = torch.cuda.current_stream().cuda_stream
ctx, got = psc.psc_create(0), {}
for i, (crystals, rad, tof, per_lor) in enumerate([(22, 21, 5, True), (22, 21, 5, False), (46, 45, 1, False), (46, 45, 1, True)]):
    sc = W.scanner_small(n_crystals=crystals, n_rings=3, n_tof=tof, n_rad=rad)
    rng = np.random.default_rng(i)
    s = psc.psc_load_scanner(ctx, psc.scanner_desc(sc))
    sums = torch.from_numpy(rng.integers(0, 1 << 40, size=sc.n_bins)).cuda()
    acc = psc.psc_acc_wrap(ctx, s, sums)
    shape = sc.lor_shape if per_lor else sc.shape
    f = [psc.psc_load_sinogram(ctx, s, rng.uniform(0.5, 2.0, shape), per_lor) for _ in range(2)]
    for first in (False, True):
        out = torch.empty(sc.shape, dtype=torch.float64, device="cuda")
        psc.psc_finalize(ctx, psc.finalize_args(acc, sens=f[0], norm=f[1], sigma=(1.5, 0.5, 0.5), scale=1e-6, sens_first=first), out, stream)
        torch.cuda.synchronize()
        got[f"{i}{first}"] = out.cpu().numpy()
psc.psc_destroy(ctx)
np.savez(sys.argv[1], **got)
'''


@pytest.mark.gpu
def test_lines_with_both_factors_in_the_debug_build(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_05047_gb300 import build
    build.build()
    got = []
    for extra in ({"PSC_LIBRARY": "debug"}, {}):
        env = {k: v for k, v in os.environ.items() if k != "PSC_LIBRARY"}
        path = str(tmp_path / f"{len(got)}.npz")
        r = subprocess.run([sys.executable, "-c", _RUN, path], cwd=ROOT, env={**env, **extra}, text=True, capture_output=True, timeout=600)
        assert r.returncode == 0, r.stderr[-2000:]
        got.append(np.load(path))
    for k in got[0].files:
        np.testing.assert_array_equal(got[0][k], got[1][k])
