"""The normal speeds of a drifting inflow: the bracketed inversion against the 64 bisections that
define it, bit for bit, on the CPU with the source's own functions."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_1311_2286_gb300", "csrc", "inject.cu")

MAIN = """
static float bisected(double q, double u, double vth) {
    const DriftCdf F(u, vth);
    double lo = 0.0, hi = (u > 0.0 ? u : 0.0) + 12.0 * vth;
    for (int it = 0; it < 64; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (F(mid) < q) lo = mid;
        else hi = mid;
    }
    return (float)(0.5 * (lo + hi));
}

int main(int argc, char** argv) {
    const double from = std::atof(argv[1]), to = std::atof(argv[2]);
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> U(from, to), V(-8.0, 8.0);
    long differ = 0;
    for (long k = 0; k < 200000; ++k) {
        const double vth = std::exp(V(g)), u = U(g) * vth;
        unsigned r = (unsigned)g();
        if (k % 50 == 0) r = k % 100 ? (unsigned)(k / 50) : 0xffffffffu - (unsigned)(k / 50);  // the tails
        const double q = 1.0 - ((double)r + 0.5) * 2.3283064365386962890625e-10;
        const float a = bisected(q, u, vth), b = drift_normal_speed(q, u, vth);
        if (std::memcmp(&a, &b, sizeof(a)) != 0) {
            if (differ++ < 5) std::printf("u/vth %.4f q %.10g: %.9g, bisected %.9g\\n", u / vth, q, b, a);
        }
    }
    return differ ? 1 : 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    text = open(SOURCE).read()
    part = text[text.index("struct DriftCdf {") : text.index("struct InjectParams {")].replace("__device__ ", "")
    where = tmp_path_factory.mktemp("drift")
    (where / "drift.cpp").write_text(
        "#include <cmath>\n#include <cstdio>\n#include <cstdlib>\n#include <cstring>\n#include <random>\n" + part + MAIN)
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", where / "drift", where / "drift.cpp"], check=True)
    return where / "drift"


# drifts in thermal speeds: into the domain, across, out of it, and so far out that the flux is rounding
@pytest.mark.parametrize("span", [(2.0, 14.0), (-1.0, 2.0), (-7.0, -1.0), (-8.4, -7.0), (-12.0, -8.4)])
def test_bracketed_inversion_is_the_bisections_bit_for_bit(program, span):
    got = subprocess.run([program, *map(str, span)], capture_output=True, text=True)
    assert got.returncode == 0, got.stdout
