// kns_shade.cuh -- the shading layout of a cell (every weight of its two MLPs, forward layers k-major, the
// layers the gradient runs back through row-major) and the tile rows of the shading kernel.
#pragma once

#include "kns_device.cuh"

namespace kns {

// layout of one cell (shared and global) and of a tile (floats, 16-byte aligned blocks)
template <class C>
struct SL {
    static constexpr int W = C::W, R0 = (C::INP + 31) / 32 * 32;  // encoding rows, padded to 32
    static constexpr int ST = 4096 / W, SRS = ST + 4;              // hits per tile (shade_hit_tile), row stride
    static constexpr int OPT = W / 8, SPT = ST / 32;               // outputs x hits per thread
    // forward, k-major
    static constexpr int T0 = 0, b0 = T0 + C::INP * W, HL = W * W + W;
    __host__ __device__ static constexpr int Tl(int l) { return b0 + W + (l - 1) * HL; }
    __host__ __device__ static constexpr int bl(int l) { return Tl(l) + W * W; }
    static constexpr int To = b0 + W + (C::H - 1) * HL, bo = To + W * 16;
    // reverse, row-major
    static constexpr int W0r = bo + 16;  // [W][R0]
    __host__ __device__ static constexpr int Wlr(int l) { return W0r + W * R0 + (l - 1) * W * W; }
    static constexpr int wd = W0r + W * R0 + (C::H - 1) * W * W;
    // colour, k-major
    static constexpr int C0t = wd + W, c0 = C0t + C::CINP * W, C1t = c0 + W, c1 = C1t + W * 4, END = c1 + 4;
    // tile rows
    static constexpr int A0 = 0;
    __host__ __device__ static constexpr int A(int l) { return R0 + (l - 1) * W; }
    static constexpr int Ud = R0 + C::H * W, U = Ud + 1, Hc = U + C::CINP, ROWS = Hc + W;
};

}  // namespace kns
