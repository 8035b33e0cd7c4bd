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
    (51, 101, 5, 16, 8, "Divide", 0), (51, 101, 5, 64, 2, "Plain", 0),
    (51, 101, 27, 45, 8, "Plain", 1), (51, 101, 13, 37, 8, "Norm", 1), (105, 99, 13, 36, 12, "Norm", 1), (51, 101, 13, 45, 16, "Plain", 1),
    (51, 101, 5, 90, 16, "Plain", 1), (5, 9, 1, 8, 25, "Plain", 1), (5, 9, 5, 45, 32, "Divide", 1), (105, 99, 13, 16, 12, "Divide", 1)])
def test_padded_axial_tiles(tmp_path, V, R, T, rings, radius, form, tiles):
    columns = (2 * rings - 1) * V * R * T
    assert _evaluate(tmp_path, [f"padded_tiles_pay({radius}, kAxial{form}, {rings}, {columns}LL)"]) == [tiles]


# crystals, rings, TOF bins, radius, a factor in the pass: lines slower than columns by 1.04 to 1.2, and faster by 1.05 to 2
@pytest.mark.parametrize("crystals,rings,T,radius,factors,lines", [
    (100, 10, 27, 4, 0, 0), (100, 10, 27, 8, 0, 0), (300, 10, 9, 8, 0, 0), (100, 24, 5, 4, 0, 0), (100, 15, 13, 0, 0, 0), (200, 10, 13, 8, 0, 0),
    (200, 16, 9, 8, 0, 0), (448, 20, 5, 16, 1, 0),                                                   # above 200,000 columns
    (448, 45, 1, 8, 0, 1), (448, 45, 4, 24, 1, 1), (64, 8, 7, 4, 0, 1), (448, 13, 5, 8, 0, 1),      # short TOF axes; few columns; a second wave
    (40, 16, 27, 8, 0, 1), (40, 44, 5, 8, 0, 1),                                                    # CTAs that are half empty
    (300, 10, 9, 8, 1, 1), (100, 24, 5, 12, 0, 1), (448, 9, 9, 24, 0, 1), (200, 9, 20, 16, 0, 1)])  # factors, wide windows
def test_radial_lines(tmp_path, crystals, rings, T, radius, factors, lines):
    assert _evaluate(tmp_path, [f"radial_lines_pay({T}, {rings * rings}, {crystals // 2}, {radius}, {factors})"]) == [lines]
