"""The routes between kernels with the same results (csrc/finalize_routes.h,
compiled here for the host) at sizes where both sides were measured."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_05047_gb300", "csrc")


def _evaluate(tmp_path, expressions):
    lines = "\n".join(f'  std::printf("%d\\n", (int)({e}));' for e in expressions)
    (tmp_path / "main.cpp").write_text(
        f'#include "finalize_routes.h"\n#include <cstdio>\nusing namespace psc;\nint main() {{\n{lines}\n}}\n')
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-o", str(tmp_path / "routes"), str(tmp_path / "main.cpp")])
    return [int(x) for x in subprocess.check_output([str(tmp_path / "routes")], text=True).split()]


# crystals, radial bins, TOF bins, rings, radius, form: tiles slower than the direct pass by 1.2 to 2.4, and faster by 1.15 to 6
@pytest.mark.parametrize("V,R,T,rings,radius,form,tiles", [
    (19, 37, 1, 37, 2, "Plain", 0), (19, 37, 5, 45, 8, "Plain", 0), (51, 101, 1, 37, 8, "Norm", 0), (27, 25, 5, 64, 8, "Norm", 0),
    (51, 101, 5, 90, 8, "Norm", 0), (11, 21, 1, 45, 12, "Norm", 0), (5, 9, 27, 45, 16, "Plain", 0), (11, 21, 5, 37, 16, "Norm", 0),
    (51, 101, 27, 8, 8, "Divide", 0), (51, 101, 5, 64, 2, "Plain", 0),
    (51, 101, 27, 45, 8, "Plain", 1), (51, 101, 13, 37, 8, "Norm", 1), (105, 99, 13, 36, 12, "Norm", 1), (51, 101, 13, 45, 16, "Plain", 1),
    (51, 101, 5, 90, 16, "Plain", 1), (5, 9, 1, 8, 25, "Plain", 1), (5, 9, 5, 45, 32, "Divide", 1), (105, 99, 13, 16, 12, "Divide", 1)])
def test_padded_axial_tiles(tmp_path, V, R, T, rings, radius, form, tiles):
    columns = (2 * rings - 1) * V * R * T
    assert _evaluate(tmp_path, [f"padded_tiles_pay({radius}, kAxial{form}, {rings}, {columns}LL)"]) == [tiles]


# TOF bins, columns, radius, a factor in the pass: lines slower than columns by 1.04 to 1.2, and faster by 1.1 to 2
@pytest.mark.parametrize("T,columns,radius,factors,lines", [
    (27, 135_000, 0, 0, 0), (27, 135_000, 4, 0, 0), (27, 86_400, 2, 0, 0), (27, 135_000, 8, 1, 0), (9, 135_000, 8, 0, 0), (5, 144_000, 4, 0, 0),
    (13, 93_600, 0, 0, 0), (13, 124_800, 8, 0, 0), (9, 135_000, 12, 0, 0), (9, 230_000, 8, 0, 0), (5, 250_000, 16, 1, 0),
    (1, 10_000_000, 8, 0, 1), (4, 2_000_000, 24, 1, 1), (7, 14_336, 4, 0, 1), (13, 46_000, 8, 0, 1), (5, 189_280, 8, 1, 1), (9, 163_296, 24, 0, 1),
    (20, 162_000, 16, 0, 1), (13, 91_000, 12, 0, 1)])
def test_radial_lines(tmp_path, T, columns, radius, factors, lines):
    assert _evaluate(tmp_path, [f"radial_lines_pay({T}, {columns}LL, {radius}, {factors})"]) == [lines]
