// kns_warp.cuh -- layer products of one warp on a tile of same-cell samples, the weights read straight from
// global memory (L1 and L2 keep the cell's rows; no staging and no barrier wider than the warp), the layer
// input x[k][0 .. P) from shared rows.  Every sum is its bias followed by one FMA per input in ascending
// order, formed as packed pairs of samples (fma.rn.f32x2), so it does not depend on the map.
//
// TileMap: lane (sg, ug) = (lane % 4, lane / 4) owns units 4 ug .. 4 ug + 3 (and 32 more for width 64) of a
// quarter of the samples: per input one float4 of a weight row, shared by the four sample groups, and S / 4
// float4s of samples feed 2 S packed FMAs.  A shared load of 16 bytes occupies the load unit two cycles even
// when all lanes read one address, so a lane per unit with broadcast samples stops at 55 FMA per cycle and
// SM, this map at 80 (4 samples a lane) and 90 (8).
// UnitMap: a lane per unit (or two); for one sample, where the weight rows are all there is to read.
#pragma once

#include "kns_device.cuh"

namespace kns {

template <int W_, int P_>
struct TileMap {
    static constexpr int W = W_, P = P_, NU = W / 8, S = P / 4;
    static_assert(W % 32 == 0 && S % 4 == 0, "tile shape");
    f32x2 acc[NU][S / 2];
    int u0, s0;  // first unit, first sample
    __device__ __forceinline__ explicit TileMap(int lane) : u0(4 * (lane >> 2)), s0(4 * (lane & 3)) {}
    __host__ __device__ static constexpr int unit(int i) { return (i & 3) + 32 * (i >> 2); }    // of u0
    __host__ __device__ static constexpr int sample(int j) { return (j & 3) + 16 * (j >> 2); }  // of s0
    __device__ __forceinline__ void bias(const float *b) {
#pragma unroll
        for (int h = 0; h < NU / 4; ++h) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(b + u0 + 32 * h));
            const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < S / 2; ++j) acc[4 * h + i][j] = f2_pack(vv[i], vv[i]);
        }
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int i = 0; i < NU; ++i)
#pragma unroll
            for (int j = 0; j < S / 2; ++j) acc[i][j] = 0ull;
    }
    // Weight rows are loaded two groups of G inputs ahead of their products; fetch() loads the first two
    // groups of a matrix, which mm() finds loaded, and mm() in turn fetches those of `next` (so that they
    // arrive while the sums are finished and stored).
    static constexpr int G = 4;
    float4 w[3][G * NU / 4];
    template <int B>
    __device__ __forceinline__ void fetch_to(const float *__restrict__ p, int ws) {
#pragma unroll
        for (int k = 0; k < G; ++k)
#pragma unroll
            for (int h = 0; h < NU / 4; ++h)
                w[B][k * (NU / 4) + h] = __ldg(reinterpret_cast<const float4 *>(p + k * ws + u0 + 32 * h));
    }
    __device__ __forceinline__ void fetch(const float *__restrict__ p, int ws) {
        fetch_to<0>(p, ws);
        fetch_to<1>(p + G * ws, ws);
    }
    template <int A, int B>
    __device__ __forceinline__ void move() {
#pragma unroll
        for (int i = 0; i < G * NU / 4; ++i) w[A][i] = w[B][i];
    }
    template <int B>
    __device__ __forceinline__ void products(const float *x, int xs) {
#pragma unroll
        for (int k = 0; k < G; ++k) {
            f32x2 t[S / 2];
#pragma unroll
            for (int j = 0; j < S / 4; ++j) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(x + k * xs + 16 * j);
                t[2 * j] = v.x;
                t[2 * j + 1] = v.y;
            }
#pragma unroll
            for (int h = 0; h < NU / 4; ++h) {
                const float4 v = w[B][k * (NU / 4) + h];
                const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f32x2 d = f2_pack(vv[i], vv[i]);
#pragma unroll
                    for (int j = 0; j < S / 2; ++j) acc[4 * h + i][j] = f2_fma(d, t[j], acc[4 * h + i][j]);
                }
            }
        }
    }
    // acc += sum_{k < K} w[k ws + unit] x[k xs + sample]
    template <int K>
    __device__ __forceinline__ void mm(const float *__restrict__ wk, int ws, const float *x, int xs,
                                       const float *__restrict__ next, int next_ws) {
        constexpr int NG = K / G;
        static_assert(K % G == 0 && NG >= 4, "layer input must be padded to 4");
        const float *xp = x + s0;
#pragma unroll 1
        for (int g = 0; g + 3 <= NG; g += 3) {
            if (g + 2 < NG) fetch_to<2>(wk + (g + 2) * G * ws, ws);
            products<0>(xp + g * G * xs, xs);
            if (g + 3 < NG) fetch_to<0>(wk + (g + 3) * G * ws, ws);
            else if (next) fetch_to<0>(next, next_ws);
            products<1>(xp + (g + 1) * G * xs, xs);
            if (g + 4 < NG) fetch_to<1>(wk + (g + 4) * G * ws, ws);
            else if (next) fetch_to<1>(next + (g + 4 - NG) * G * next_ws, next_ws);
            products<2>(xp + (g + 2) * G * xs, xs);
        }
        if constexpr (NG % 3 == 1) {  // buffer 0: the last group; 1: next's first
            if (next) fetch_to<2>(next + G * next_ws, next_ws);
            products<0>(xp + (NG - 1) * G * xs, xs);
            move<0, 1>();
            move<1, 2>();
        }
        if constexpr (NG % 3 == 2) {  // buffers 0 and 1: the last two groups
            if (next) fetch_to<2>(next, next_ws);
            products<0>(xp + (NG - 2) * G * xs, xs);
            if (next) fetch_to<0>(next + G * next_ws, next_ws);
            products<1>(xp + (NG - 1) * G * xs, xs);
            move<1, 0>();
            move<0, 2>();
        }
    }
    // The same with the weight rows in shared memory (16-byte aligned).
    template <int K>
    __device__ __forceinline__ void mm_shared(const float *wk, int ws, const float *x, int xs) {
        const float *xp = x + s0, *wp = wk + u0;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            f32x2 t[S / 2];
#pragma unroll
            for (int j = 0; j < S / 4; ++j) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(xp + k * xs + 16 * j);
                t[2 * j] = v.x;
                t[2 * j + 1] = v.y;
            }
#pragma unroll
            for (int h = 0; h < NU / 4; ++h) {
                const float4 v = *reinterpret_cast<const float4 *>(wp + k * ws + 32 * h);
                const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f32x2 d = f2_pack(vv[i], vv[i]);
#pragma unroll
                    for (int j = 0; j < S / 2; ++j) acc[4 * h + i][j] = f2_fma(d, t[j], acc[4 * h + i][j]);
                }
            }
        }
    }
    __device__ __forceinline__ void bias_shared(const float *b) {
#pragma unroll
        for (int h = 0; h < NU / 4; ++h) {
            const float4 v = *reinterpret_cast<const float4 *>(b + u0 + 32 * h);
            const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < S / 2; ++j) acc[4 * h + i][j] = f2_pack(vv[i], vv[i]);
        }
    }
    // rows[unit][sample] = f(sum, unit, sample)
    template <class F>
    __device__ __forceinline__ void store(float *rows, int xs, F f) const {
#pragma unroll
        for (int i = 0; i < NU; ++i) {
            const int u = u0 + unit(i);
#pragma unroll
            for (int j = 0; j < S; j += 4) {
                const int s = s0 + sample(j);
                float a, b, c, d;
                f2_unpack(acc[i][j / 2], a, b);
                f2_unpack(acc[i][j / 2 + 1], c, d);
                *reinterpret_cast<float4 *>(rows + u * xs + s) =
                    make_float4(f(a, u, s), f(b, u, s + 1), f(c, u, s + 2), f(d, u, s + 3));
            }
        }
    }
};

template <int W_>
struct UnitMap {
    static constexpr int W = W_, P = 1, NU = W / 32;
    static_assert(NU == 1 || NU == 2, "width must be 32 or 64");
    float acc[NU];
    int u0;
    __device__ __forceinline__ explicit UnitMap(int lane) : u0(NU * lane) {}
    static __device__ __forceinline__ void load(const float *p, float (&v)[NU]) {
        if constexpr (NU == 1) {
            v[0] = __ldg(p);
        } else {
            const float2 t = __ldg(reinterpret_cast<const float2 *>(p));
            v[0] = t.x;
            v[1] = t.y;
        }
    }
    __device__ __forceinline__ void bias(const float *b) { load(b + u0, acc); }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int u = 0; u < NU; ++u) acc[u] = 0.f;
    }
    __device__ __forceinline__ void fetch(const float *, int) {}
    template <int K>
    __device__ __forceinline__ void mm(const float *__restrict__ w, int ws, const float *x, int, const float *, int) {
        static_assert(K % 4 == 0, "layer input must be padded to 4");
        const float *wp = w + u0;
#pragma unroll 4
        for (int k = 0; k < K; k += 4) {
            const float4 t4 = *reinterpret_cast<const float4 *>(x + k);
            const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float v[NU];
                load(wp + (k + i) * ws, v);
#pragma unroll
                for (int u = 0; u < NU; ++u) acc[u] = fmaf(v[u], t[i], acc[u]);
            }
        }
    }
    template <class F>
    __device__ __forceinline__ void store(float *rows, int xs, F f) const {
#pragma unroll
        for (int u = 0; u < NU; ++u) rows[(u0 + u) * xs] = f(acc[u], u0 + u, 0);
    }
    // f(sum, index) of the lane's units
    template <class F>
    __device__ __forceinline__ void each(F f) const {
#pragma unroll
        for (int u = 0; u < NU; ++u) f(acc[u], u);
    }
};

// Starts bringing `bytes` (a multiple of 16) at p (16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Row stride (floats) of P samples: the stores of a warp's units fall into distinct banks.
__host__ __device__ constexpr int row_stride(int P) { return P == 1 ? 1 : P + 4; }

}  // namespace kns
