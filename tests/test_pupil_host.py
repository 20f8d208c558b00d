"""The float-float pupil chord (osog_pupil.h), compiled for the host: every
interval it decides must be that of the double-precision formula, for every
column of shifted and centred circles on canvases of 32 to 2048 rows, and
nearly every column must be decided."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), os.pardir, "paper_2606_21381_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "osog_pupil.h"
using namespace osog;
static ff split(double v) { const float h = (float)v; return {h, (float)(v - (double)h)}; }
// argv: width, height; prints columns, undecided, wrong
int main(int, char **argv) {
    const int W = std::atoi(argv[1]), H = std::atoi(argv[2]);
    std::mt19937_64 rng(W * 4099 + H);
    std::uniform_real_distribution<> u(0.0, 1.0);
    long n = 0, open = 0, wrong = 0;
    for (int k = 0; k < 2000; ++k) {
        const double dx = k % 4 ? 0.05 + 2.0 * u(rng) : 0.5, lambda = k % 3 ? 0.3 + u(rng) : 0.5;
        const double NA = k % 2 ? 0.05 + 1.4 * u(rng) : 0.4;
        const double r = NA / lambda, frac = k % 5 ? u(rng) : 0.0, angle = k % 7 ? 6.3 * u(rng) : 0.0;
        const double ox = frac * r * std::cos(angle), oy = frac * r * std::sin(angle);
        const double fxs = 1.0 / (W * dx), span = H * dx;
        const PupilFF p = {split(fxs), split(ox), split(oy), split(r * r), split(span)};
        for (int fx = -W / 2; fx < W / 2; ++fx) {
            RowRange got;
            ++n;
            if (!pupil_chord_ff(p, fx, &got)) {
                ++open;
                continue;
            }
            const RowRange want = pupil_chord_exact(r * r, ox, oy, fxs, span, fx);
            wrong += got.lo != want.lo || got.hi != want.hi;
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
    d = tmp_path_factory.mktemp("pupil")
    (d / "p.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(d / "p.cpp"),
                    "-o", str(d / "p")], check=True)
    return d / "p"


# a twentieth of the circles lies on the lattice's axes (centred, rational NA /
# lambda), where ends on whole rows are not rare; the rest is decided except in
# intervals of 4e-6 rows
@pytest.mark.parametrize("W,H", [(32, 32), (256, 256), (2048, 32), (32, 2048), (2048, 2048)])
def test_decided_chords_are_those_of_double_precision(harness, W, H):
    out = subprocess.run([str(harness), str(W), str(H)], check=True, capture_output=True,
                         text=True).stdout
    n, undecided, wrong = (int(v) for v in out.split())
    assert wrong == 0
    assert undecided <= 0.01 * n
