"""CPU test of the taps of the anisotropic lookup: the header that the kernel
includes, compiled with the host compiler."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_05618_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <limits>
#include "aniso_taps.h"
using namespace htex;

static long bad = 0, inside = 0, outside = 0;

template <int TB>
static void check(int n, float x, float y, float wl, float scale) {
    const uint64_t base = 1u << 20;
    const int64_t N = int64_t(1) << n;
    LevelTaps<TB> L;
    const float W = L.plan(base, n, x, y, wl);
    const TapsG tx = taps_g(x, int(N)), ty = taps_g(y, int(N));
    float sum = 0.0f;
    for (int k = 0; k < 4; ++k) {
        const int64_t i = tx.i + (k & 1), j = ty.i + (k >> 1);
        const bool in = i >= 0 && i < N && j >= 0 && j < N;
        (in ? inside : outside) += 1;
        const float w = wl * (k & 2 ? ty.w1 : ty.w0) * (k & 1 ? tx.w1 : tx.w0);
        if (L.read(k) && (!in || L.at(k) != base + uint64_t(j * N + i) * TB)) ++bad;   // out of the texture
        if (in && w > 1e-30f && !L.read(k)) ++bad;                                     // left out
        const float s = L.w[k] * scale_of(L.w[k], scale), want = L.w[k] * scale;
        if (L.read(k) ? !(s == want || (std::isnan(s) && std::isnan(want))) : s != 0.0f) ++bad;
        if (L.read(k) && w > 1e-30f && !(W > 0.0f)) ++bad;   // the sums' scale is on
        sum += L.w[k];
    }
    if (!(std::fabs(sum - W) <= 1e-5f)) ++bad;
}

int main() {
    const float inf = std::numeric_limits<float>::infinity();
    const float scales[] = {1.0f, 0.0f, -2.5f, 3e38f, 1e-42f, inf, -inf, std::nanf("")};
    const float at[] = {-40.0f, -1.5f, -1.0f, -0.5f, -0.03f, -1e-7f, 0.0f, 1e-7f, 0.03f, 0.25f, 0.5f, 0.7f,
                        0.97f, 0.9999999f, 1.0f, 1.0000001f, 1.03f, 1.5f, 2.0f, 40.0f};
    const float levels[] = {0.0f, 0.3f, 1.0f};
    for (int n = 0; n <= 13; ++n)
        for (float scale : scales)
            for (float wl : levels)
                for (float x : at)
                    for (float y : at) {
                        check<1>(n, x, y, wl, scale);
                        check<3>(n, x, y, wl, scale);
                        check<16>(n, x, y, wl, scale);
                    }
    std::printf("%ld bad, %ld inside, %ld outside\n", bad, inside, outside);
    return bad || !inside || !outside;
}
"""


def test_no_tap_outside_its_texture_is_read(tmp_path):
    """Every size 1..8192, coordinates on, inside, beside and far off the
    quad, level weights down to zero (a lane without work) and every kind of
    code scale (finite, zero, infinite, NaN): a tap that is read lies in the
    texture at its own place, one of positive weight is read, and one that
    is not read weighs exactly zero under any scale.  The level's share of the
    normalisation weight is positive where a tap counts (it switches the
    scale of the sums)."""
    src, exe = tmp_path / "taps.cpp", tmp_path / "taps"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
