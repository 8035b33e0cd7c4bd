"""How a batch is cut into work items (csrc/work_items.h, compiled here for the
host): every history once, at most 65536 to an item, whole rounds of the grid,
and no more items to a CTA than its share of the histories pays for, since a CTA
drains its slots after each."""
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_05047_gb300", "csrc")
MAIN = r'''
#include "work_items.h"
#include <cstdio>
int main() {
  unsigned long long grid, per, most, n[64], c[64];
  int jobs;
  while (std::scanf("%llu %llu %llu %d", &grid, &per, &most, &jobs) == 4) {
    for (int j = 0; j < jobs; ++j) if (std::scanf("%llu", n + j) != 1) return 1;
    psc::work_items(n, jobs, grid, per, most, c);
    for (int j = 0; j < jobs; ++j) std::printf("%llu ", c[j]);
    std::printf("\n");
  }
}
'''


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(d / "items"), str(d / "main.cpp")])

    def run(requests):
        text = "\n".join(f"{g} {per} {most} {len(n)} " + " ".join(map(str, n)) for g, per, most, n in requests)
        out = subprocess.run([str(d / "items")], input=text, text=True, capture_output=True, check=True).stdout
        return [[int(x) for x in line.split()] for line in out.splitlines()]
    return run


@pytest.mark.parametrize("requests,each", [(2, 100_000), (8, 50_000), (16, 20_000), (32, 5_000), (32, 20_000), (32, 60_000),
                                           (32, 200_000), (48, 1_000)])
def test_equal_requests_share_the_rounds(cut, requests, each):
    grid = 304
    (chunk,) = cut([(grid, 1, 65536, [each] * requests)])
    items = sum(-(-each // c) for c in chunk)
    share = -(-requests * each // grid)
    rounds = max(1, share // 1024)
    assert items <= rounds * grid + requests   # at most one left over per request


def test_every_request_is_covered(cut):
    rng = random.Random(5)
    cases = []
    for _ in range(400):
        jobs = rng.choice([1, 1, 2, 5, 48])
        cases.append((rng.choice([1, 3, 64, 304, 1216]), rng.choice([1, 4, 16]), rng.choice([1, 8192, 65536]),
                      [int(10 ** rng.uniform(0, rng.choice([3, 6, 12, 19]))) for _ in range(jobs)]))
    cases.append((304, 1, 65536, [2 ** 64 - 1]))
    for (grid, per, most, n), chunk in zip(cases, cut(cases)):
        for h, c in zip(n, chunk):
            assert 1 <= c <= min(65536, max(1024, most)) and c <= h
            items = -(-h // c)
            if len(n) == 1:  # whole rounds, or one item of at least 128 histories each
                cta = -(-h // grid)
                rounds = max(per, -(-cta // min(65536, max(1024, most))))
                assert items <= rounds * grid
                assert c >= min(h, 128) // 2 + 1 or items <= grid
