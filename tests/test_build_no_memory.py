"""The host Bi-CSR builder when memory runs out: whichever allocation fails, it
reports it (2) or builds the same graph without it; no thread is lost and the
process goes on."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_05895_gb300", "csrc")

HARNESS = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>
#include "mf_internal.h"
static std::atomic<long> left{-1};   // allocations until one fails; -1: none does
static std::atomic<long> count{0};
static void *get(std::size_t n) {
    count.fetch_add(1);
    if (left.load() >= 0 && left.fetch_sub(1) == 0) throw std::bad_alloc();
    void *p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void *operator new(std::size_t n) { return get(n); }
void *operator new[](std::size_t n) { return get(n); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete[](void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
void operator delete[](void *p, std::size_t) noexcept { std::free(p); }

int main() {
    // vertices 0..7 have edges to most others in falling order (rows the builder sorts by a bitmap)
    const int n = 8192;
    std::vector<int64_t> row(1, 0);
    std::vector<int32_t> col, cap;
    unsigned x = 1;
    for (int u = 0; u < n; ++u) {
        const int d = u < 8 ? 7000 : 4;
        for (int i = 0; i < d; ++i) {
            x = x * 1664525u + 1013904223u;
            col.push_back(u < 8 ? n - 1 - i : int(x >> 19));
            cap.push_back(int(x >> 24));
        }
        row.push_back(int64_t(col.size()));
    }
    mf::HostBiCSR want;
    if (mf::build_bicsr(n, int64_t(col.size()), row.data(), col.data(), cap.data(), 0, n - 1, true, &want)) return 3;
    const long all = 4 * count.load() + 64;
    int failed = 0, built = 0;
    for (long k = 0; k < all; ++k) {
        mf::HostBiCSR got;
        left.store(k);
        const int rc = mf::build_bicsr(n, int64_t(col.size()), row.data(), col.data(), cap.data(), 0, n - 1, true, &got);
        const bool hit = left.load() < 0;
        left.store(-1);
        if (rc == 2) { ++failed; continue; }
        if (rc != 0) return 4;
        ++built;
        if (got.arcs != want.arcs || got.cap_limit != want.cap_limit) return 5;
        for (int64_t a = 0; a < got.arcs; ++a)
            if (got.head[a] != want.head[a] || got.rev[a] != want.rev[a] || got.cap[a] != want.cap[a]) return 6;
        if (!hit && k > 8) break;   // every allocation has been failed once
    }
    std::printf("%d refused, %d built\n", failed, built);
    return failed > 10 ? 0 : 7;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_any_allocation_may_fail(tmp_path):
    src = tmp_path / "harness.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "harness")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, str(src), os.path.join(CSRC, "mf_build.cpp"),
                    "-o", exe], check=True, timeout=300)
    res = subprocess.run([exe], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, timeout=300)
    assert res.returncode == 0, res.stdout.decode(errors="replace")
