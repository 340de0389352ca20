"""Stopping rules of the mixed path (csrc/refine_rules.h), compiled for the host: a mode at
the documented floor of 1e-14 is not reported as unconverged after the last GMRES cycle,
keeps its iterate when GMRES has no memory, and is not restarted from zero."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_11162_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdio>
#include "refine_rules.h"
using namespace pmlbie;
static int bad = 0;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); ++bad; } } while (0)

int main() {
    // refinement: tolerances met; contracting; stalled at the floor, above it, divergent
    CHECK(refine_rule(1, true, 1e-3, 0.0) == RefineStep::kDone);
    CHECK(refine_rule(1, false, 1e-3, 0.0) == RefineStep::kContinue);
    CHECK(refine_rule(2, false, 0.49e-10, 1e-10) == RefineStep::kContinue);
    CHECK(refine_rule(2, false, 4e-16, 5e-16) == RefineStep::kDone);
    CHECK(refine_rule(2, false, 5e-16, 6e-16) == RefineStep::kSlow);
    CHECK(refine_rule(2, false, 1e-2, 1e-3) == RefineStep::kSlow);
    CHECK(refine_rule(2, false, NAN, 1e-3) == RefineStep::kSlow);
    // GMRES: a mode that gains 30 % in each of ten cycles below 1e-14 is done after the last
    double b = 1e-14;
    bool done = gmres_rule(false, 0, 10, b, 1.0);
    CHECK(!done);
    for (int c = 1; c <= 10; ++c) {
        done = gmres_rule(false, c, 10, 0.7 * b, b);
        b *= 0.7;
        CHECK(done == (c == 10));
    }
    CHECK(gmres_rule(false, 3, 10, 9.5e-15, 1e-14) && !gmres_rule(false, 3, 10, 1.1e-14, 1.1e-14));
    CHECK(!gmres_rule(false, 10, 10, 1.1e-14, 1.1e-14) && !gmres_rule(false, 10, 10, NAN, 1e-14));
    CHECK(gmres_rule(true, 0, 10, 1.0, 1.0));
    // start: from zero only above the floor and without progress
    CHECK(!restart_from_zero(5e-15, 4e-15) && !restart_from_zero(1e-8, 1e-7));
    CHECK(restart_from_zero(1e-3, 1e-4) && restart_from_zero(NAN, 1e-4));
    // no memory: modes at the floor keep their iterate, the others are left
    std::vector<int> slow = {0, 1, 1, 1, 1};
    CHECK(accept_refined(slow, {1.0, 1e-14, 2e-14, 5e-16, NAN}) == 2);
    CHECK(slow == (std::vector<int>{0, 0, 1, 0, 1}));
    return bad;
}
"""


def test_refine_rules(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    (tmp_path / "rules.cpp").write_text(SRC)
    exe = str(tmp_path / "rules")
    r = subprocess.run(["g++", "-std=c++17", "-Wall", "-I", CSRC, str(tmp_path / "rules.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
