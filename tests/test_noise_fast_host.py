"""The FP32 sensor-noise draw (osog_noise_fast.h), compiled for the host and
checked against the double-precision draw: whatever it reports as decided --
a Poisson count, a rejection, a rounded output -- must be the
double-precision result, and few draws may be left open."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), os.pardir, "paper_2606_21381_gb300", "csrc")

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "osog_noise_fast.h"
using namespace osog;
using namespace osog::noise;
static double unit(uint32_t x) { return ((double)x + 0.5) * (1.0 / 4294967296.0); }
// argv: what, low, high (range of the rate or of the gain, log-uniform);
// prints: draws, undecided, wrong
int main(int, char **argv) {
    const int what = std::atoi(argv[1]);
    const double lo = std::log(std::atof(argv[2])), hi = std::log(std::atof(argv[3]));
    std::mt19937_64 rng(1);
    std::uniform_real_distribution<> range(lo, hi);
    long n = 0, open = 0, wrong = 0;
    for (int i = 0; i < 1000000; ++i) {
        uint32_t a = (uint32_t)rng(), b = (uint32_t)(rng() >> 9);
        if (i % 8 == 7) a >>= rng() % 20;   // the ends of the unit interval
        if (i % 8 == 3) b >>= rng() % 20;
        const double p = std::exp(range(rng));
        ++n;
        if (what == 0) {  // inversion
            float k = 0.f;
            const int r = poisson_small((float)p, a, &k);
            double q = std::exp(-p), F = q;
            int want = 0;
            while (unit(a) > F && want < 1000) F += q *= p / ++want;
            if (r != kYes) ++open;
            else if ((double)k != want) ++wrong;
        } else if (what == 1) {  // one attempt of the rejection
            const float v = 1.37f;
            const double g = p / v, lam = g * (double)v;
            if (lam < 10.0) continue;
            const ff gf = split(g);
            ff lf = two_prod(gf.h, v);
            lf = fast_two_sum(lf.h, fmaf(gf.l, v, lf.l));
            float k = 0.f;
            const int r = ptrs_attempt(ptrs_of(lf), a, b, &k);
            const double U = unit(a) - 0.5, V = unit(b), us = 0.5 - std::fabs(U);
            const double bb = 0.931 + 2.53 * std::sqrt(lam), aa = -0.059 + 0.02483 * bb;
            const double ia = 1.1239 + 1.1328 / (bb - 3.4), vr = 0.9277 - 3.6224 / (bb - 2.0);
            const double kk = std::floor((2.0 * aa / us + bb) * U + lam + 0.43);
            int want;
            if (us >= 0.07 && V <= vr) want = kYes;
            else if (kk < 0.0 || (us < 0.013 && V > us)) want = kNo;
            else want = std::log(V * ia / (aa / (us * us) + bb)) <=
                        -lam + kk * std::log(lam) - std::lgamma(kk + 1.0) ? kYes : kNo;
            if (r == kUndecided) ++open;
            else if (r != want || (r == kYes && (double)k != kk)) ++wrong;
            // the test with the rate's constants in float
            float kc = 0.f;
            uint32_t m = 0;
            if (ptrs_candidate(ptrs_of(lf), a, b, &kc, &m) == kYes && !(us >= 0.07 && V <= vr)) {
                const int s = ptrs_accept_float(lf, kc, m, b);
                if (s != kUndecided && s != want) ++wrong;
            }
        } else {  // the rounded output for counts up to 2^22
            if (a == 0u) continue;
            const float k = i % 7 ? (float)(rng() % (1u << (1 + rng() % 22))) : 0.f;
            const double sigma = i % 3 ? std::exp((double)(rng() % 7) - 3.0) : 0.0;
            const double z = std::sqrt(-2.0 * std::log(unit(a))) *
                             std::cos(6.283185307179586476925286766559 * unit(b));
            float got;
            const ff sz = sigma > 0 ? mul_lazy(split(sigma), normal_ff(a, b)) : ff{0.f, 0.f};
            const bool ok = noisy_value(k, sz, split(1.0 / p), &got);
            if (!ok) ++open;
            else if (got != (float)(((double)k + sigma * z) / p)) ++wrong;
        }
    }
    std::printf("%ld %ld %ld\n", n, open, wrong);
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("noise")
    (d / "n.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(d / "n.cpp"),
                    "-o", str(d / "n")], check=True)
    return d / "n"


# the share that may stay open: a few times the widths of the bounds (6e-6 per
# cumulative sum, some 1e-4 of an acceptance test's unit scale, 2^-37 of the
# normal against half a float ulp), and 2^-39 of the rate near an integer for
# the largest rates; an eighth of the draws is pushed to the interval's ends
@pytest.mark.parametrize("what,low,high,most", [
    (0, 1e-6, 10.0, 5e-4), (1, 10.0, 30.0, 5e-4), (1, 10.0, 3e4, 5e-4), (1, 3e4, 8e6, 2e-3),
    (2, 1e-6, 1e-2, 5e-4), (2, 1.0, 1e5, 5e-4), (2, 1e5, 1e12, 5e-4)])
def test_decided_draws_are_those_of_double_precision(harness, what, low, high, most):
    out = subprocess.run([str(harness), str(what), repr(low), repr(high)], check=True,
                         capture_output=True, text=True).stdout
    n, undecided, wrong = (int(v) for v in out.split())
    assert wrong == 0
    # rates past 2^22 are left to double precision by design
    assert undecided <= most * n or high > 4e6


# the shares above, of all rates below 2^22 and of all counts (none is left to double
# precision by design there)
@pytest.mark.parametrize("what,low,high,most", [(1, 3e4, 4e6, 2e-3), (2, 1e5, 1e12, 5e-4)])
def test_few_draws_of_large_rates_and_gains_stay_open(harness, what, low, high, most):
    out = subprocess.run([str(harness), str(what), repr(low), repr(high)], check=True,
                         capture_output=True, text=True).stdout
    n, undecided, wrong = (int(v) for v in out.split())
    assert wrong == 0
    assert undecided <= most * n
