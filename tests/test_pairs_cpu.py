"""The pair gathers stay inside the pair region and its pads whatever state a
packet is resumed in: pairs.cuh compiled for the host, on a region between two
guards."""
import os
import subprocess

import pytest

from paper_1709_10187_gb300 import build as B

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "pairs.cuh"
using namespace rddmc;

int main() {
    uint32_t seed = 12345u;
    auto rnd = [&]() { seed = seed * 1664525u + 1013904223u; return seed ^ (seed >> 13); };
    for (uint32_t n : {1u, 2u, 3u, 37u, 512u, 1u << 20}) {
        const uint32_t J = n < 37u ? 1u : 37u;
        // pad, pairs, pad: exactly what the walk may read
        char* mem = (char*)std::aligned_alloc(64, ((2 * kPairPad + 16ull * n) + 63) & ~63ull);
        for (uint64_t i = 0; i < 2 * kPairPad + 16ull * n; ++i) mem[i] = (char)rnd();
        const Pair* base = (const Pair*)(mem + kPairPad);
        // states of a table, of a cell in vacuum (class 0xffffffff), and anything
        std::vector<uint32_t> states = {0u, n - 1u, n, 0xffffffffu, 0x80000000u, 0x10000000u, 0x0fffffffu};
        for (uint32_t j = 0; j < J; ++j) states.push_back(0xffffffffu * J + j);
        for (int i = 0; i < 200; ++i) states.push_back(rnd());
        for (uint32_t s : states)
            for (int k = 0; k < 50; ++k) {
                const uint32_t o = pair_offset(s, 16u * (n - 1u));
                if (o % 16u || o > 16u * (n - 1u) || (s < n && o != 16u * s)) return 1;
                uint4 r = make_uint4(rnd(), rnd(), rnd(), rnd());
                if (k & 1) r = make_uint4(0u, 0u, 0u, 0u);           // always down
                if (k & 2) r = make_uint4(~0u, ~0u, ~0u, ~0u);       // always up
                const FourMoves m = walk_four(base, r, o);
                // the second gather's sixteen bytes lie inside the pads
                const long long b = (long long)m.o2 - 32;
                if (b < -kPairPad || b + 16 > 16ll * n + kPairPad) return 2;
            }
        std::free(mem);
    }
    std::puts("ok");
    return 0;
}
"""


def test_gathers_of_any_state_stay_inside_the_region(tmp_path):
    src = tmp_path / "pairs.cu"
    src.write_text(SRC)
    exe = str(tmp_path / "pairs")
    try:
        cc = B.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    r = subprocess.run([cc, "-std=c++17", "-O1", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), "-o", exe,
                        str(src)] + B.ARCH, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.returncode
