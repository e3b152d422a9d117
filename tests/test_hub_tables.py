"""Capacity, home slot and task shares of the hub tables, over every capacity up
to the largest (2^32 slots, for vertices of more than 2^30 edges): no size may
lose slots to 32-bit arithmetic.  The library's own functions, compiled for the
host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "internal.cuh"
#include <cstdio>

int main() {
    using namespace gsp;
    int bad = 0;
    auto expect = [&](bool ok, const char *what, uint64_t deg) {
        if (!ok && bad++ < 20) printf("%s: degree %llu\n", what, (unsigned long long)deg);
    };
    for (int lg = 13; lg < 36; lg++) {
        for (int d = -1; d <= 1; d++) {
            const uint64_t deg = (1ull << lg) + d;
            const uint64_t cap = hub_slots(deg);
            expect(cap && !(cap & (cap - 1)) && cap <= 1ull << 32, "a power of two up to 2^32", deg);
            expect(cap >= 2 * deg || cap == 1ull << 32, "two slots an edge", deg);
            const uint32_t mask = (uint32_t)(cap - 1);
            // homes are the hash's top bits: monotone, from the first slot to the last
            expect(hub_home(0u, mask) == 0 && hub_home(0xFFFFFFFFu, mask) == mask, "homes span the table", deg);
            uint32_t before = 0;
            for (uint64_t x = 0; x < 1ull << 32; x += 0x0123457ull) {
                const uint32_t h = hub_home((uint32_t)x, mask);
                expect(h <= mask && h >= before && h == (uint32_t)(((unsigned __int128)x * cap) >> 32), "home", deg);
                before = h;
            }
            expect(((mask + 1u) & mask) == 0, "the probe wraps to the first slot", deg);
            // the tasks' shares cover [0, cap) without gap, each in 32 bits
            const uint64_t n = (deg + HUB_CHUNK - 1) / HUB_CHUNK;
            expect(hub_share(cap, 0, n) == 0 && hub_share(cap, n, n) == cap, "shares cover the table", deg);
            for (uint64_t k = 0; k < n; k += 1 + n / 1000) {
                const uint64_t first = hub_share(cap, k, n), slots = hub_share(cap, k + 1, n) - first;
                expect(first <= mask && slots >= 1 && (uint32_t)slots == slots && first + slots <= cap, "share", deg);
            }
            const uint64_t last = hub_share(cap, n - 1, n);
            expect(last + (uint32_t)(hub_share(cap, n, n) - last) == cap, "the last share ends the table", deg);
        }
    }
    return bad != 0;
}
"""


def test_hub_table_arithmetic(tmp_path):
    from paper_2402_11454_gb300 import build
    src, exe = tmp_path / "hub.cu", tmp_path / "hub"
    src.write_text(PROGRAM)
    r = subprocess.run([build.NVCC, *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "--extended-lambda", "-O1",
                        "-I", build.CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
