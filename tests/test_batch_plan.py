"""The number of chains in flight that a batch chooses: the library's own rule, compiled with the host
compiler (the header needs no CUDA)."""

import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include <cstdio>
#include "batch_plan.cuh"
int main() {  // per problem: free bytes, chains, then n nnz r m caliber fp64 learned of each; prints threads, bytes...
    double free;
    int count;
    while (std::scanf("%lf %d", &free, &count) == 2) {
        std::vector<bamg::BatchChain> v;
        for (int k = 0; k < count; ++k) {
            long long n, nnz;
            int r, m, c, fp64, learned;
            if (std::scanf("%lld %lld %d %d %d %d %d", &n, &nnz, &r, &m, &c, &fp64, &learned) != 7) return 1;
            v.push_back({n, nnz, r, m, c, fp64 != 0, learned != 0});
        }
        std::printf("%d", bamg::batch_workers(v, free));
        for (const auto& k : v) std::printf(" %.1f", bamg::batch_chain_bytes(k));
        std::printf("\n");
    }
}
"""
GIB = 2.0 ** 30


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_1004_1451_gb300", "csrc"),
                    "-o", str(d / "plan"), str(d / "main.cpp")], check=True)

    def run(free, chains):
        text = "%.1f %d\n" % (free, len(chains)) + "\n".join(" ".join(str(int(x)) for x in c) for c in chains)
        out = subprocess.run([str(d / "plan")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return int(out[0]), [float(x) for x in out[1:]]

    return run


def test_chains_that_do_not_fit_side_by_side_are_not_started_side_by_side(plan):
    big = [(724 * 724, 4 * 724 * 724, 8, 50, 2, 1, 0)] * 12  # about 1 GiB each
    assert plan(200 * GIB, big)[0] == 12
    assert plan(6 * GIB, big)[0] == 3  # as many as one thread per four chains, which fits
    assert plan(0, big)[0] == 3
    small = [(2500, 10000, 8, 50, 2, 1, 0)] * 32
    assert plan(200 * GIB, small)[0] == 16 and plan(1.25 * GIB, small)[0] == 16 and plan(0, small)[0] == 8


def test_bounds_hold_for_any_batch(plan):
    rng = random.Random(3)
    for _ in range(60):
        n = sorted((int(100 * 10 ** (5 * rng.random())) for _ in range(rng.randint(1, 70))), reverse=True)
        chains = [(k, k * rng.randint(2, 8), rng.randint(4, 16), rng.choice([20, 50, 256]), rng.randint(1, 4),
                   rng.randint(0, 1), rng.randint(0, 1)) for k in n]
        free = GIB * 250 ** rng.random()
        threads, size = plan(free, chains)
        least = min(16, (len(chains) + 3) // 4)
        assert least <= threads <= min(16, len(chains))
        if threads > least:
            assert sum(size[:threads]) <= min(free / 2, 16 * GIB)


@pytest.mark.parametrize("n,per_row,r,m,c,fp64,peak", [
    (512, 4, 8, 50, 2, 0, 480), (512, 4, 8, 50, 4, 1, 800), (1024, 3, 10, 50, 4, 0, 2336), (1024, 3, 10, 50, 2, 1, 2144),
    (1024, 3, 10, 50, 4, 1, 3264), (512, 6, 16, 50, 4, 1, 960), (1024, 6, 16, 64, 2, 0, 1568)])
def test_estimates_cover_measured_peaks(plan, n, per_row, r, m, c, fp64, peak):
    """Peaks of a setup and solve in MiB (grid walks, tandem queues and triangulations): the budget is half of
    the free memory, so an estimate may be a tenth short but not more."""
    _, (size,) = plan(0, [(n * n, per_row * n * n, r, m, c, fp64, 0)])
    assert size >= 0.9 * peak * 2 ** 20
