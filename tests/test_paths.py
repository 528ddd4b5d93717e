"""The host's choice of clusters and pause counts (csrc/gx_paths.h) on CPU: equal to a plain
restatement that tries every count, and not growing with the square of the scenario count."""
import os
import shutil
import subprocess

import pytest

from paper_2410_13055_gb300 import build as b

PROGRAM = r"""
#include "gx_paths.h"
#include <chrono>
#include <cstdio>
#include <random>
using namespace gx;
struct Choice { double us, room; };
typedef std::vector<Choice> List;
typedef std::vector<const List*> Lists;

// every step by a full pass over the scenarios
static double assign(const Lists& ch, size_t n, std::vector<size_t>& at, bool* fits) {
    at.assign(n, 0);
    double room = 0;
    bool one = true;
    for (size_t i = 0; i < n; ++i) { room += (*ch[i])[0].room; one = one && ch[i] == ch[0]; }
    const double limit = one ? 1.0 + 1e-9 : 0.9;
    *fits = room <= limit;
    if (one) {
        for (size_t k = 1; k < ch[0]->size(); ++k)
            if ((double)n * (*ch[0])[k].room <= limit) std::fill(at.begin(), at.end(), k);
    } else if (*fits) {
        for (;;) {
            size_t w = 0;
            for (size_t i = 1; i < n; ++i)
                if ((*ch[i])[at[i]].us > (*ch[w])[at[w]].us) w = i;
            if (at[w] + 1 >= ch[w]->size()) break;
            const double more = (*ch[w])[at[w] + 1].room - (*ch[w])[at[w]].room;
            if (room + more > limit) break;
            room += more;
            ++at[w];
        }
    }
    double us = 0;
    for (size_t i = 0; i < n; ++i) us = std::max(us, (*ch[i])[at[i]].us);
    return us;
}

int main() {
    std::mt19937 rng(7);
    auto uni = [&](double lo, double hi) { return std::uniform_real_distribution<double>(lo, hi)(rng); };
    auto lists = [&](int keys, double room0, double us0) {
        std::vector<List> v(keys);
        for (auto& l : v) {
            const int n = 1 + (int)uni(0, 6);
            double us = us0 * uni(0.3, 3.0), room = room0 * uni(0.3, 3.0);
            for (int k = 0; k < n; ++k) { l.push_back({us, room}); us *= uni(0.5, 0.95); room *= uni(1.1, 2.0); }
        }
        return v;
    };
    int bad = 0;
    for (int trial = 0; trial < 3000; ++trial) {
        const int keys = 1 + (int)uni(0, trial % 3 ? 8 : 1), n = 1 + (int)uni(0, 64);
        const std::vector<List> v = lists(keys, 1.0 / uni(2, 80), uni(1, 30));
        Lists ch;
        for (int i = 0; i < n; ++i) ch.push_back(&v[(size_t)uni(0, keys)]);
        std::vector<size_t> a, c;
        bool fa, fc;
        const double ua = assign(ch, n, a, &fa), uc = crs_assign(ch, n, c, &fc);
        if (ua != uc || a != c || fa != fc) ++bad;
        std::stable_sort(ch.begin(), ch.end(), [](const List* x, const List* y) { return (*x)[0].room > (*y)[0].room; });
        std::vector<double> dh(n);
        for (auto& x : dh) x = uni(0, 3e5);
        size_t want = 0;  // the pause count up to 64 is the exact one
        const size_t most = trial % 2 ? n : n - 1;
        for (size_t k = most; k >= 1 && !want; --k) {
            double d = 0;
            for (size_t i = 0; i < k; ++i) d += dh[i];
            if (assign(ch, k, a, &fa) < 0.95 * stream_us(d) && fa) want = k;
        }
        if (crs_pause_at(ch, dh, most) != want) ++bad;
        std::stable_sort(ch.begin(), ch.end(), [](const List* x, const List* y) { return (*x)[0].us > (*y)[0].us; });
        const size_t k = crs_regroup_at(ch, uc);
        if (k >= ch.size() && k) ++bad;
        if (k && !(assign(ch, k, a, &fa) < 0.9 * uc && fa)) ++bad;
    }
    // pauses lie on residual checks, after at least the given time, and at the cap at the latest
    for (int trial = 0; trial < 1000; ++trial) {
        const int every = 1 + (int)uni(0, 40), it = every * (int)uni(0, 50), max_it = it + 1 + (int)uni(0, 5000);
        const double us = uni(0.5, 20), part = uni(1, 3000);
        const int e = crs_pause_end(it, us, part, every, max_it);
        if (e <= it || e > max_it || (e < max_it && ((e - it) % every || (e - it) * us < part * (1 - 1e-9)))) ++bad;
    }
    double worst = 0;  // milliseconds of the searches before one loop over 8,192 scenarios
    for (double us0 : {2.0, 60.0}) for (int keys : {1, 20, 8192}) for (double room0 : {1.0 / 700, 1.0 / 20}) {
        const std::vector<List> v = lists(keys, room0, us0);
        Lists ch;
        for (int i = 0; i < 8192; ++i) ch.push_back(&v[i % keys]);
        std::stable_sort(ch.begin(), ch.end(), [](const List* x, const List* y) { return (*x)[0].room > (*y)[0].room; });
        std::vector<double> dh(8192, 500.0);
        const auto t0 = std::chrono::steady_clock::now();
        volatile size_t k = crs_pause_at(ch, dh, 8191) + crs_regroup_at(ch, us0);
        (void)k;
        worst = std::max(worst, std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count());
    }
    std::printf("%d differ, %.2f ms\n", bad, worst);
    return bad || worst > 25.0;
}
"""


def test_choices_equal_the_plain_search_and_stay_cheap(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "paths.cpp", tmp_path / "paths"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", b.CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    print(r.stdout)
