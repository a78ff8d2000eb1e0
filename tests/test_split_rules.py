"""The launchers' splits (csrc/sp_split.h, host code): the run lengths are those of a search over
every length, and a launch does not pay for such a search."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <random>
#include "sp_split.h"
using namespace sp;

template <typename Cost> long long every(long long total, int occ, int n_sm, long long limit, const Cost &cost) {
    const long long wave = (long long)n_sm * std::max(occ, 1), p0 = (total + wave - 1) / wave;
    long long best = p0;
    double best_cost = 0;
    for (long long p = p0; p <= limit; ++p) {
        const long long ctas = (total + p - 1) / p, q = (ctas + n_sm - 1) / n_sm;
        const double c = cost(q, p);
        if (p == p0 || c < best_cost * 0.999) best = p, best_cost = c;
        if (q == 1) break;
    }
    return best;
}

int main() {
    std::mt19937_64 rng(7);
    auto pick = [&](double lo, double hi) {
        return (long long)std::exp(std::uniform_real_distribution<>(std::log(lo), std::log(hi))(rng));
    };
    const int sms[] = {1, 7, 132, 152, 160};
    for (int i = 0; i < 3000; ++i) {
        const int n_sm = sms[rng() % 5], occ = 1 + rng() % 32, halo = rng() % 17;
        const long long total = pick(1, 3e6), wave = (long long)n_sm * occ, p0 = (total + wave - 1) / wave;
        const double load = (1 + rng() % 8) / 8.0, latency = rng() % 2 ? 1.0 : 4.0;
        const int wpc = 1 + rng() % 2;
        if (rows_per_cta(total, halo, load, latency, occ, n_sm) !=
            every(total, occ, n_sm, std::min(total, 8 * p0 + 32), [=](long long q, long long p) { return (q * load + latency) * (p + halo); }))
            return std::printf("rows_per_cta %lld\n", total), 1;
        if (warptb_rows(total, halo, wpc, occ, n_sm) !=
            every(total, occ, n_sm, std::min(total, 8 * p0 + 32), [=](long long q, long long p) { return std::max(5.0, q * wpc / 4.0) * (p + halo); }))
            return std::printf("warptb_rows %lld\n", total), 1;
        const long long nz = pick(1, 3000), tiles = pick(1, 2000), t = tiles * nz, b0 = (t + wave - 1) / wave;
        const double h = 0.7 * (1 + rng() % 4);
        if (planes_per_cta(tiles, (int)nz, h, occ, n_sm) !=
            every(t, occ, n_sm, std::min(t, 4 * b0 + 8), [=](long long q, long long p) { return (q + 1.0) * (p + (nz % p ? 2 : 1) * h); }))
            return std::printf("planes_per_cta %lld %lld\n", tiles, nz), 1;
    }
    // 32768^2 in strips of 120 columns, 1024^3 in 32 x 16 tiles, and a grid of one column of tiles
    const auto t0 = std::chrono::steady_clock::now();
    long long sum = 0;
    for (int i = 0; i < 1000; ++i) {
        sum += warptb_rows(137LL * (32768 + i), 8, 2, 12, 152) + rows_per_cta(35LL * (32768 + i), 4, 1.0, 1.0, 4, 152);
        sum += planes_per_cta(2048, 1024 + i, 1.0, 4, 152) + planes_per_cta(1, (1 << 30) + i, 1.0, 4, 152);
    }
    const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - t0).count() / 4000;
    std::printf("%.3f us per call (%lld)\n", us, sum);
    return us < 20 ? 0 : 2;
}
"""


def test_run_lengths(tmp_path):
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text("#include <cmath>\n" + PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I" + os.path.join(ROOT, "paper_2511_10508_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
