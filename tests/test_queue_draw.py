"""CPU check of the rule by which busy warps of the CSR search draw tickets for the frames they
hand out: the function is compiled here from the kernel source's own text, with the device's
atomics replaced by the host's, and run by many donor threads against few waiting consumers.
No donor may ever get a ticket that no consumer holds (so the queue's cells, however few, are
never oversubscribed), every ticket goes to one donor, and with donors left none stays undrawn."""
from __future__ import annotations

import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1705_09358_gb300", "csrc", "sge_kernels.cu")

_HEAD = r"""
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#define __device__
using std::min;
struct SearchCtl { unsigned long long *phead, *ptail; };
static unsigned long long load_relaxed(const unsigned long long *p) { return __atomic_load_n(p, __ATOMIC_RELAXED); }
static unsigned long long atomicCAS(unsigned long long *p, unsigned long long want, unsigned long long to) {
    __atomic_compare_exchange_n(p, &want, to, false, __ATOMIC_RELAXED, __ATOMIC_RELAXED);
    return want;
}
constexpr int DRAW_TRIES = 4;
"""

_MAIN = r"""
int main() {
    constexpr int DONORS = 10, ROUNDS = 120;
    for (int round = 0; round < ROUNDS; ++round) {
        alignas(128) unsigned long long head = 0;
        alignas(128) unsigned long long tail = 0;
        const int consumers = 1 + round % 50;
        SearchCtl C{&head, &tail};
        std::vector<std::atomic<int>> drawn(4 * consumers);
        for (auto &d : drawn) d = 0;
        std::atomic<int> bad{0}, done{0};
        std::vector<std::thread> ts;
        for (int d = 0; d < DONORS; ++d)
            ts.emplace_back([&, d] {
                for (int spin = 0; done.load() == 0 || load_relaxed(&tail) < load_relaxed(&head); ++spin) {
                    unsigned long long t = 0;
                    const int most = 1 + (d + spin) % 32, n = queue_draw(C, most, t);
                    if (n < 0 || n > most) bad++;
                    if (n > 0 && t + n > __atomic_load_n(&head, __ATOMIC_SEQ_CST)) bad++;   // nobody holds it
                    for (int i = 0; i < n; ++i)
                        if (t + i >= drawn.size() || drawn[t + i]++ != 0) bad++;
                }
            });
        // the consumers' tickets come in bursts, four laps of them
        for (int lap = 0; lap < 4; ++lap) {
            for (int i = 0; i < consumers; ++i) __atomic_fetch_add(&head, 1, __ATOMIC_SEQ_CST);
            if (round & 1) std::this_thread::yield();
        }
        done = 1;
        for (auto &t : ts) t.join();
        if (tail != head) bad++;
        for (auto &d : drawn) if (d != 1) bad++;
        if (bad) { std::printf("round %d: %d wrong, head %llu tail %llu\n", round, bad.load(), head, tail); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
"""


def _text() -> str:
    with open(SRC) as f:
        return f.read()


def _function(text: str, head: str) -> str:
    a = text.index(head)
    end = "\n}\n"
    return text[a:text.index(end, a) + len(end)]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_donors_draw_only_tickets_that_consumers_hold(tmp_path):
    src = tmp_path / "draw_check.cpp"
    src.write_text(_HEAD + _function(_text(), "__device__ int queue_draw(") + _MAIN)
    exe = tmp_path / "draw_check"
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", str(src), "-o", str(exe)], check=True,
                   capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


def test_csr_donors_draw_by_that_rule_alone():
    text = _text()
    # the producers' counter moves in the bounded rule and in the bitset search's claim only
    assert len(re.findall(r"atomic\w+\(C\.ptail", text)) == 2
    assert "atomicAdd(C.ptail" in _function(text, "__device__ long long queue_reserve(")
    kernel = text[text.index("k_search_csr(const JobDesc"):text.index("search: bitset kernel")]
    assert "push_children(" in kernel and "push_to_waiting(" in kernel and "push_frame(" not in kernel
    for name in ("__device__ unsigned push_children(", "__device__ bool push_to_waiting("):
        body = _function(text, name)
        assert "queue_draw(" in body and "queue_reserve(" not in body
