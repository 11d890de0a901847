// Hilbert keys of points: the position along the Hilbert curve of order 16 of the cell a point falls
// into on a 65,536 x 65,536 grid. A run of points along the curve never jumps, so its bounding box is
// compact (a run of the Z-order curve may straddle two far quadrants). Against Z-order a query's
// walk visits 3 sub-tiles instead of 11 (1M uniform points, k = 10), and phase 1 takes, us, before /
// now: 257 x 300,007 30 / 15, 8,192 x 1M 57 / 27, 153,984 x 262,147 clustered 720 / 356, 1M x 1M
// (pruned scan with the ordering) 1,890 / 1,293; FP64 8,191 x 131,072 92 / 49.
//
// From the top bit down the curve is a walk of four states (whether the coordinates are swapped and
// whether they are complemented): a bit pair gives two bits of the position and the next state. Bit
// by bit that is about 200 integer instructions a key and bounds the kernel; a table takes four bit
// pairs at a step. Keys of 6,000,000 points: 66.5 us bit by bit, 25.6 with the table
// (Z-order 20.8).
#pragma once

#include <cstdint>

namespace aidw {

// By state (swap, complement), four bits of x and four of y: eight bits of the position in the low
// byte, the next state above.
struct HilbertTable {
    uint16_t e[1024];
};

constexpr HilbertTable hilbert_table()
{
    HilbertTable t{};
    for (unsigned i = 0; i < 1024; ++i) {
        unsigned swap = i >> 9, flip = (i >> 8) & 1u, pos = 0;
        for (int b = 3; b >= 0; --b) {
            const unsigned x = (i >> (4 + b)) & 1u, y = (i >> b) & 1u;
            const unsigned rx = (swap ? y : x) ^ flip, ry = (swap ? x : y) ^ flip;
            pos = (pos << 2) | ((3u * rx) ^ ry);
            flip ^= rx & (ry ^ 1u);
            swap ^= ry ^ 1u;
        }
        t.e[i] = static_cast<uint16_t>((swap << 9) | (flip << 8) | pos);
    }
    return t;
}

static __device__ const HilbertTable kHilbertTable = hilbert_table();

// A block's copy of the table; the caller synchronises before it is read.
__device__ __forceinline__ void load_hilbert_table(uint16_t (&t)[1024])
{
    const uint32_t *src = reinterpret_cast<const uint32_t *>(kHilbertTable.e);
    for (int i = threadIdx.x; i < 512; i += blockDim.x)
        reinterpret_cast<uint32_t *>(t)[i] = src[i];
}

// The key of (x, y) on the grid over `box` (xmin, ymin, xmax, ymax); points outside the box, or NaN,
// clamp to its edges.
__device__ __forceinline__ uint32_t hilbert_of(float x, float y, float4 box,
                                               const uint16_t (&t)[1024])
{
    const float sx = box.z > box.x ? 65535.0f / (box.z - box.x) : 0.0f;
    const float sy = box.w > box.y ? 65535.0f / (box.w - box.y) : 0.0f;
    const uint32_t cx =
        static_cast<uint32_t>(fminf(fmaxf((x - box.x) * sx, 0.0f), 65535.0f));
    const uint32_t cy =
        static_cast<uint32_t>(fminf(fmaxf((y - box.y) * sy, 0.0f), 65535.0f));
    uint32_t d = 0, state = 0;
#pragma unroll
    for (int b = 12; b >= 0; b -= 4) {
        const uint32_t e = t[state | (((cx >> b) & 15u) << 4) | ((cy >> b) & 15u)];
        d = (d << 8) | (e & 0xffu);
        state = e & 0x300u;
    }
    return d;
}

}  // namespace aidw
