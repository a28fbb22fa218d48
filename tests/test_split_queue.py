"""CPU check of the rule by which the split's queue, which outlives a call, is cleared and marked:
compiled here from the library's own source text and run against buffers that fail to be allocated
or cleared at every point in turn.  A call that gets the queue must find no word in it that carries
the call's own mark, whatever failed before."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HOST_SRC = os.path.join(ROOT, "paper_1705_09358_gb300", "csrc", "sge_host.cpp")

_HEAD = r"""
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <vector>
enum cudaError_t { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
// a new block holds the marks 1 .. 1000 over and over, like a block that another queue has used
struct FakeBuf {
    void *p = nullptr;
    size_t cap = 0;
    bool fail = false;
    std::vector<unsigned long long> mem;
    cudaError_t ensure(size_t bytes) {
        if (p && bytes <= cap) return cudaSuccess;
        p = nullptr;
        cap = 0;
        if (fail) return cudaErrorMemoryAllocation;
        mem.assign(bytes / 8, 0);
        for (size_t i = 0; i < mem.size(); ++i) mem[i] = (unsigned long long)(1 + i % 1000) << 40;
        p = mem.data();
        cap = bytes;
        return cudaSuccess;
    }
    void drop() { p = nullptr; cap = 0; }
};
"""

_MAIN = r"""
int main() {
    constexpr int Q = 4096;
    // two calls with one failure each (none, list, entries, clearing), or the block dropped or grown before them
    for (int f1 = 0; f1 < 4; ++f1)
        for (int f2 = 0; f2 < 4; ++f2)
            for (int between = 0; between < 3; ++between) {
                FakeBuf entry, left;
                unsigned long long epoch = 0;
                for (int call = 0; call < 6; ++call) {
                    const int f = call == 1 ? f1 : call == 3 ? f2 : 0;
                    if (call == 3 && between == 1) entry.drop();
                    if ((call == 1 || call == 4) && f1 == 1) left.drop();
                    if (call == 1 && f1 == 2) entry.drop();
                    if (call == 3 && f2 == 1) left.drop();
                    if (call == 3 && f2 == 2) entry.drop();
                    if (call == 1 && f1 == 3) epoch = (1ull << 24) - 1;   // (the wrap clears as well)
                    left.fail = f == 1;
                    entry.fail = f == 2;
                    const int q = call >= 3 && between == 2 ? 2 * Q : Q;
                    const cudaError_t e = split_queue_ready(entry, (size_t)q * 8, left, 800, epoch, [&](void *p, size_t n) {
                        if (f == 3) return cudaErrorMemoryAllocation;
                        std::memset(p, 0, n);
                        return cudaSuccess;
                    });
                    if (e != cudaSuccess) continue;
                    if (epoch == 0 || epoch >= (1ull << 24)) { std::printf("mark %llu\n", epoch); return 1; }
                    for (int i = 0; i < q; ++i)
                        if (entry.mem[i] >> 40 == epoch) {
                            std::printf("word %d carries the mark of call %d (%d %d %d)\n", i, call, f1, f2, between);
                            return 1;
                        }
                    for (int i = 0; i < q; i += 2) entry.mem[i] = epoch << 40 | i;   // what a launch leaves
                }
            }
    // the first call ever fails after the entries were allocated
    for (int what = 1; what < 4; ++what) {
        FakeBuf entry, left;
        unsigned long long epoch = 0;
        left.fail = what == 1;
        entry.fail = what == 2;
        auto clear = [&](void *p, size_t n) {
            if (what == 3) return cudaErrorMemoryAllocation;
            std::memset(p, 0, n);
            return cudaSuccess;
        };
        if (split_queue_ready(entry, Q * 8, left, 800, epoch, clear) == cudaSuccess) { std::printf("no failure\n"); return 1; }
        left.fail = entry.fail = false;
        what = what == 3 ? 0 : what;
        if (split_queue_ready(entry, Q * 8, left, 800, epoch, clear) != cudaSuccess) { std::printf("stays failed\n"); return 1; }
        for (int i = 0; i < Q; ++i)
            if (entry.mem[i] >> 40 == epoch) { std::printf("uncleared word %d\n", i); return 1; }
        if (what == 0) break;
    }
    // every mark of a long run is new until the block is cleared again
    {
        FakeBuf entry, left;
        unsigned long long epoch = 0, last = 0;
        long long clears = 0;
        for (long long call = 0; call < (1ll << 24) + 100; ++call) {
            const long long before = clears;
            split_queue_ready(entry, 64, left, 64, epoch, [&](void *, size_t) { ++clears; return cudaSuccess; });
            if (clears == before ? epoch <= last : epoch == 0) { std::printf("mark repeated\n"); return 1; }
            last = epoch;
        }
        if (clears != 2) { std::printf("cleared %lld times\n", clears); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
"""


def _rule() -> str:
    with open(HOST_SRC) as f:
        text = f.read()
    a = text.index("template <class Buf, class Clear>")
    end = "\n}\n"
    return text[a:text.index(end, a) + len(end)]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_queue_never_holds_the_next_launches_mark(tmp_path):
    src = tmp_path / "queue_check.cpp"
    src.write_text(_HEAD + _rule() + _MAIN)
    exe = tmp_path / "queue_check"
    subprocess.run(["g++", "-std=c++17", "-O2", str(src), "-o", str(exe)], check=True, capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
