"""The table of remembered host queries (csrc/remembered.h), on the CPU: right
answers, no allocation (an entry point that promises to allocate nothing uses
it), failed queries not remembered, more keys than slots, several threads."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include <thread>
#include <initializer_list>
#include "remembered.h"

static std::atomic<int> allocations{0};
void* operator new(std::size_t n) { ++allocations; return std::malloc(n); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

static msc::Remembered table;
static int ask(int dev, long k, int threads, size_t smem, std::atomic<int>* queries, int fail = 0) {
    int out = -1;
    const int e = table.get(&out, dev, (const void*)k, threads, smem, [&](int* o) {
        ++*queries;
        *o = (int)(dev * 7 + k * 3 + threads + (int)smem);
        return fail;
    });
    return e ? -1000 - e : out;
}

int main() {
    std::atomic<int> q{0};
    const int a0 = allocations;
    int wrong = 0;
    if (ask(0, 5, 256, 64, &q, 2) != -1002 || ask(0, 5, 256, 64, &q, 2) != -1002 || q != 2) ++wrong;  // not remembered
    q = 0;
    for (int rep = 0; rep < 3; ++rep)
        for (int dev = 0; dev < 2; ++dev)
            for (long k = 1; k <= 20; ++k)
                for (size_t smem : {0ul, 1000ul, 98304ul})
                    wrong += ask(dev, k, 256, smem, &q) != (int)(dev * 7 + k * 3 + 256 + (int)smem);
    if (q != 120) ++wrong;  // each key asked once
    for (int rep = 0; rep < 2; ++rep)
        for (long k = 1000; k < 4000; ++k) wrong += ask(1, k, 128, 8, &q) != (int)(7 + k * 3 + 128 + 8);  // past the slots
    const int a1 = allocations;
    std::thread t[4];
    std::atomic<int> bad{0};
    static msc::Remembered fresh;
    for (int i = 0; i < 4; ++i)
        t[i] = std::thread([&, i] {
            for (int rep = 0; rep < 200; ++rep)
                for (long k = 1; k <= 50; ++k) {
                    int out = -1;
                    fresh.get(&out, i & 1, (const void*)k, 64, 0, [&](int* o) { *o = (int)(k * 2 + (i & 1)); return 0; });
                    if (out != (int)(k * 2 + (i & 1))) ++bad;
                }
        });
    for (auto& x : t) x.join();
    std::printf("%d %d %d\n", wrong, (int)bad, a1 - a0);
}
"""


def test_remembered(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2409_03771_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert out.split() == ["0", "0", "0"], out
