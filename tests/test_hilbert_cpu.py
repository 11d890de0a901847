"""The Hilbert table (four bit pairs of a key at a step) against the bit-by-bit curve, and the curve's
defining property: consecutive positions are neighbouring cells. The header is compiled for the
host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#define __device__
#define __forceinline__ inline
#include <cmath>
#include <cstdint>
#include <cstdio>
struct float4 { float x, y, z, w; };
static struct { unsigned x = 0; } threadIdx;
static struct { unsigned x = 1; } blockDim;
#include "hilbert.cuh"

static uint32_t bitwise(uint32_t x, uint32_t y)
{
    uint32_t d = 0;
    for (int b = 15; b >= 0; --b) {
        const uint32_t rx = (x >> b) & 1u, ry = (y >> b) & 1u;
        d = (d << 2) | ((3u * rx) ^ ry);
        const uint32_t flip = (rx & ~ry & 1u) ? 0xffffu : 0u;
        const uint32_t u = x ^ flip, v = y ^ flip;
        x = ry ? u : v;
        y = ry ? v : u;
    }
    return d;
}

int main()
{
    static uint16_t t[1024];
    aidw::load_hilbert_table(t);
    const float4 box{0.0f, 0.0f, 65535.0f, 65535.0f};
    for (uint32_t x = 0; x < 65536; x += 13)
        for (uint32_t y = x % 7; y < 65536; y += 11)
            if (aidw::hilbert_of(float(x), float(y), box, t) != bitwise(x, y))
                return 1;
    // The first 2^20 positions cover the 1,024 x 1,024 corner cells, each next to the last.
    static uint32_t at[1 << 20];
    for (uint32_t x = 0; x < 1024; ++x)
        for (uint32_t y = 0; y < 1024; ++y) {
            const uint32_t d = aidw::hilbert_of(float(x), float(y), box, t);
            if (d >> 20)
                return 2;
            at[d] = (x << 16) | y;
        }
    for (uint32_t d = 1; d < (1u << 20); ++d) {
        const int dx = int(at[d] >> 16) - int(at[d - 1] >> 16);
        const int dy = int(at[d] & 0xffff) - int(at[d - 1] & 0xffff);
        if (dx * dx + dy * dy != 1)
            return 3;
    }
    const float nan = NAN;
    if (aidw::hilbert_of(nan, nan, box, t) != bitwise(0, 0) ||
        aidw::hilbert_of(-1e30f, 1e30f, box, t) != bitwise(0, 65535))
        return 4;
    return 0;
}
"""


def test_table(tmp_path):
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(SRC)
    inc = os.path.join(ROOT, "paper_1511_02186_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-w", "-I", inc, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)]).returncode == 0
