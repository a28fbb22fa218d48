"""CPU check of the label table that every target load builds: the function is compiled here from
the library's own source text and compared with sorting all labels -- the same distinct labels and
places, for few and for many labels, of any values -- and it must not cost what that sorting costs."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST_SRC = os.path.join(ROOT, "paper_1705_09358_gb300", "csrc", "sge_host.cpp")

_HEAD = """#include <algorithm>
#include <chrono>
#include <climits>
#include <cstdint>
#include <cstdio>
#include <mutex>
#include <random>
#include <thread>
#include <vector>
"""

_MAIN = r"""
static void by_sorting(const std::vector<int32_t> &lab, std::vector<int32_t> &labs, std::vector<int32_t> &idx) {
    labs = lab;
    std::sort(labs.begin(), labs.end());
    labs.erase(std::unique(labs.begin(), labs.end()), labs.end());
    idx.resize(lab.size());
    for (size_t v = 0; v < lab.size(); ++v)
        idx[v] = (int32_t)(std::lower_bound(labs.begin(), labs.end(), lab[v]) - labs.begin());
}

static void whole(int n, auto body) { body(0, n); }
static void threads(int n, auto body) {   // seven uneven parts at once
    std::vector<std::thread> t;
    for (long long i = 0; i < 7; ++i) t.emplace_back([=] { body((int)(n * i * i / 49), (int)(n * (i + 1) * (i + 1) / 49)); });
    for (auto &x : t) x.join();
}

int main() {
    std::mt19937 g(7);
    for (int n : {1, 2, 127, 128, 129, 255, 1000, 40000})
        for (int kind = 0; kind < 5; ++kind) {
            std::vector<int32_t> lab((size_t)n), labs, idx, want, widx;
            for (int v = 0; v < n; ++v) {
                const int32_t r = (int32_t)g();
                lab[(size_t)v] = kind == 0 ? 5 : kind == 1 ? r % 64 : kind == 2 ? r
                                 : kind == 3 ? (v % 3 == 0 ? INT_MIN : v % 3 == 1 ? INT_MAX : -1)
                                             : (r % 200) << 24;
            }
            by_sorting(lab, want, widx);
            for (long long most : {(long long)n, (long long)want.size(), (long long)want.size() - 1, 0ll}) {
                const bool fits = (long long)want.size() <= most;
                for (int how = 0; how < 3; ++how) {
                    if (how == 2) label_indices(lab.data(), n, most, labs, nullptr, [](int m, auto b) { threads(m, b); });
                    else if (how == 1) label_indices(lab.data(), n, most, labs, &idx, [](int m, auto b) { threads(m, b); });
                    else label_indices(lab.data(), n, most, labs, &idx, [](int m, auto b) { whole(m, b); });
                    if (fits ? labs != want || idx != widx : !labs.empty() || !idx.empty()) {
                        std::printf("n %d kind %d most %lld how %d wrong\n", n, kind, most, how);
                        return 1;
                    }
                }
            }
        }
    // 300,000 vertices, 200 labels: best of five each
    std::vector<int32_t> lab(300000), labs, idx;
    for (auto &x : lab) x = (int32_t)(g() % 200);
    double best[2] = {1e9, 1e9};
    for (int rep = 0; rep < 10; ++rep) {
        const auto t0 = std::chrono::steady_clock::now();
        if (rep & 1) by_sorting(lab, labs, idx);
        else label_indices(lab.data(), (int)lab.size(), 1 << 20, labs, &idx, [](int m, auto b) { whole(m, b); });
        const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        best[rep & 1] = std::min(best[rep & 1], ms);
    }
    std::printf("%.3f ms, by sorting %.3f ms\n", best[0], best[1]);
    return best[0] * 2 < best[1] ? 0 : 2;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_label_indices(tmp_path):
    with open(HOST_SRC) as f:
        text = f.read()
    a = text.index("struct LabelTable {")
    end = "\n}\n"
    b = text.index("void label_indices(", a)
    src = tmp_path / "labels.cpp"
    src.write_text(_HEAD + text[a:text.index(end, b) + len(end)] + _MAIN)
    exe = tmp_path / "labels"
    subprocess.run(["g++", "-std=c++20", "-O2", "-pthread", str(src), "-o", str(exe)], check=True, capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
