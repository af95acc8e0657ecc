// kns_train_tile.cu -- the grouped MLP kernels of the training step: SDF and colour MLPs of one cell
// evaluated, and differentiated, on warp tiles of same-cell records.
//
// A block takes a chunk (up to 4096 records of one cell, from the counting sort), stages the cell's weights in
// shared memory (forward layers k-major, backward layers row-major), and its warps walk the chunk in tiles of
// 32 records (16 for the sample centres), each on rows of its own: every dense layer, forward (A_l = act(W
// A_{l-1} + b)) and backward (D_l = (W^T D_{l+1}) . act'(A_l)), is a product of the warp's 8 x 4 lanes
// (kns_warp.cuh), so no barrier stands between layers, only around a chunk.  The weight gradient of a tile, dW_l =
// D_l A_{l-1}^T summed over its records, accumulates in the lanes' registers over the whole chunk, and the
// block adds its warps' sums to the global gradient once per chunk.
//
// What bounds them is the FP32 pipe and the loads that feed it.  Block tiles of 128 records (a barrier per layer;
// for each layer's weight gradient only the 72 threads that held its entries at work) took, per step of 65,536 rays
// x 96 samples and 16,384 eikonal points on a GB300: difference points forward 7.1 ms, centres forward 2.5,
// centres backward 10.6, difference points backward 28.6 ms; now 6.3, 2.2, 7.1 and 18.8 ms (the step 51.2 -> 36.6
// ms; 1,024 rays 3.0 -> 2.2 ms).  The forward kernel keeps the FP32 pipe 58 % busy; the backward ones have eight
// warps per SM (238 registers a thread for the difference points, 255 for the centres) and wait for the results of
// their own FMA chains, on shared loads and on instruction fetch: unrolling the weight-gradient
// loop twice costs 4.7 ms, five warps of 168 registers the same, loads a half step ahead 2.9 ms.
//
// Kernels: d at records (coarse samples and difference points); sample centres forward (d, z,
// colour); sample centres backward (colour and SDF, writes the difference points' upstream);
// difference points backward.  Model: Sec. 3.1 (Eq. 1-3) with the training loss of Sec. 3.2.2.
#include <cuda_runtime.h>
#include <stdint.h>

#include "kns_device.cuh"
#include "kns_kernels.h"
#include "kns_train.cuh"
#include "kns_warp.cuh"

namespace kns {
namespace {

using train::CHUNK;
using train::chunk_key;
using train::fd_normal;
using train::grid_for;
using train::load3;

constexpr int PE_L = 4;

// ------------------------------------------------------------------ canonical offsets in a cell
template <int H>
struct WL {
    static constexpr int HL = 32 * 32 + 32;
    static constexpr int cW0 = 0, cb0 = 27 * 32, cH = cb0 + 32;
    static constexpr int cWo = cH + (H - 1) * HL, cbo = cWo + 512, cC0 = cbo + 16;
    static constexpr int cc0 = cC0 + 33 * 32, cC1 = cc0 + 32, cc1 = cC1 + 96;
};

// ------------------------------------------------------------------ records on warps
// The kernels of the difference points and coarse samples (151 M records in a step of 2^18 rays) work on warp
// tiles: a warp takes 32 records of the chunk's cell through every layer on its own rows in shared memory
// (kns_warp.cuh's map: 8 records x 4 units a lane), with no barrier but those around the cell's weights,
// which the block's warps share.
constexpr int WT = 32;                 // records per warp tile
constexpr int WRS = row_stride(WT);    // row stride (floats)
constexpr int WTS = 36;                // row stride of transposed weights: the transposing stores conflict less

// weights of one cell in shared memory (floats): per layer T_l[k][o] (stride WTS) and b_l; the row-major
// hidden layers the deltas run back through; the d row and its bias
template <int H>
struct WW {
    static constexpr int K0 = 28;
    __host__ __device__ static constexpr int T(int l) { return l == 0 ? 0 : K0 * WTS + 32 + (l - 1) * (32 * WTS + 32); }
    __host__ __device__ static constexpr int b(int l) { return T(l) + (l == 0 ? K0 : 32) * WTS; }
    static constexpr int wo = T(H), bo = wo + 32, FEND = bo + 4;
    __host__ __device__ static constexpr int R(int l) { return FEND + (l - 1) * 1024; }
    static constexpr int END = FEND + (H - 1) * 1024;
};

// the cell's canonical SDF weights into sw (every thread of the block; nt threads)
template <int H, bool BACKWARD>
__device__ __forceinline__ void load_cell(const float *__restrict__ cw, float *sw, int nt) {
    using L = WL<H>;
    using S = WW<H>;
    const int tid = threadIdx.x;
    for (int j = tid; j < 27 * 32; j += nt) sw[S::T(0) + (j % 27) * WTS + j / 27] = __ldg(cw + L::cW0 + j);
    if (tid < 32) {
        sw[S::T(0) + 27 * WTS + tid] = 0.f;
        sw[S::b(0) + tid] = __ldg(cw + L::cb0 + tid);
        sw[S::wo + tid] = __ldg(cw + L::cWo + tid);
        if (tid == 0) sw[S::bo] = __ldg(cw + L::cbo);
    }
#pragma unroll
    for (int l = 1; l < H; ++l) {
        const float *src = cw + L::cH + (l - 1) * L::HL;
        for (int j = tid; j < 1024; j += nt) {
            const float v = __ldg(src + j);
            sw[S::T(l) + (j & 31) * WTS + (j >> 5)] = v;
            if (BACKWARD) sw[S::R(l) + j] = v;
        }
        if (tid < 32) sw[S::b(l) + tid] = __ldg(src + 1024 + tid);
    }
}

// encoding of record `lane` (Eq. 1) into column lane of rows E; row 27 is zero
__device__ __forceinline__ void encode_record(float *E, int lane, float x, float y, float z) {
    float in[28];
    encode3<PE_L>(x, y, z, in);
#pragma unroll
    for (int k = 0; k < 28; ++k) E[k * WRS + lane] = in[k];
}

// ------------------------------------------------------------------ forward: d at records
constexpr int FW = 8, FB = 3;  // warps per block, blocks per SM
template <int H>
__global__ void __launch_bounds__(32 * FW, FB) k_warp_eval_d(TrainArgs a, int k0, int k1, float *out) {
    using S = WW<H>;
    extern __shared__ float4 smem4[];
    float *sw = reinterpret_cast<float *>(smem4);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *rows = sw + S::FEND + warp * 32 * WRS;  // a layer overwrites its input
    const int c0 = a.chunk_off[k0], total = a.chunk_off[k1] - c0;
    auto act = [&](float v, int, int) { return softplus_f32(v, a.beta, a.inv_beta); };
    for (int ci = blockIdx.x; ci < total; ci += gridDim.x) {
        const int key = chunk_key(a.chunk_off, k0, k1, c0 + ci);
        const int j = c0 + ci - a.chunk_off[key];
        const int beg = a.off[key] + j * CHUNK, end = min(beg + CHUNK, a.off[key + 1]);
        __syncthreads();
        load_cell<H, false>(a.params + (int64_t)key * a.p_cell, sw, 32 * FW);
        __syncthreads();
        for (int tb = beg + WT * warp; tb < end; tb += WT * FW) {
            float4 r = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
            if (tb + lane < end) r = a.sorted[tb + lane];
            encode_record(rows, lane, r.x, r.y, r.z);
            __syncwarp();
            TileMap<32, WT> m(lane);
            m.bias_shared(sw + S::b(0));
            m.template mm_shared<28>(sw + S::T(0), WTS, rows, WRS);
            __syncwarp();  // every lane has read the input before it is overwritten
            m.store(rows, WRS, act);
            __syncwarp();
#pragma unroll 1
            for (int l = 1; l < H; ++l) {
                m.bias_shared(sw + S::b(l));
                m.template mm_shared<32>(sw + S::T(l), WTS, rows, WRS);
                __syncwarp();
                m.store(rows, WRS, act);
                __syncwarp();
            }
            float d = sw[S::bo];
#pragma unroll 8
            for (int k = 0; k < 32; ++k) d = fmaf(sw[S::wo + k], rows[k * WRS + lane], d);
            const int rec = __float_as_int(r.w);
            if (rec >= 0) out[rec] = d;
            __syncwarp();
        }
    }
}

// ------------------------------------------------------------------ backward of the difference points
// Per warp tile: the forward layers recomputed (rows E, A_1 .. A_H), then from the output back, each layer's
// weight gradient while its inputs are still in their rows and the deltas D_l over A_l.  The weight gradients
// of the whole chunk stay in registers -- lane (og, ig) = (lane / 8, lane % 8) owns outputs og + 4 i and inputs
// ig + 8 j of every layer, 12 loads of 16 bytes for 128 FMAs -- and are summed over the block's warps in shared
// memory and added to the global gradient once per chunk.
constexpr int BW = 4;  // warps per block, two blocks per SM: 238 registers, 101 of them gradient sums
template <int H>
struct WRows {
    __host__ __device__ static constexpr int A(int l) { return 32 * l; }  // A(0): the encoding
    static constexpr int G = 32 * (H + 1), ROWS = G + 1;                  // G: the upstream of d
};

// acc[i][j] += sum over the tile's records of D[og + 4 i] A[ig + 8 j]
__device__ __forceinline__ void fma44(const float4 &dv, const float4 (&xv)[4], float (&acc)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float s = acc[j];
        s = fmaf(dv.x, xv[j].x, s);
        s = fmaf(dv.y, xv[j].y, s);
        s = fmaf(dv.z, xv[j].z, s);
        s = fmaf(dv.w, xv[j].w, s);
        acc[j] = s;
    }
}
__device__ __forceinline__ void grad_tile32(const float *D, const float *A, float (&acc)[8][4], int lane) {
    const float *d = D + (lane >> 3) * WRS, *x = A + (lane & 7) * WRS;
#pragma unroll 1
    for (int r = 0; r < WT; r += 4) {
        float4 xv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) xv[j] = *reinterpret_cast<const float4 *>(x + 8 * j * WRS + r);
#pragma unroll
        for (int i = 0; i < 8; ++i) fma44(*reinterpret_cast<const float4 *>(d + 4 * i * WRS + r), xv, acc[i]);
    }
}
// sum over the tile's records of row `lane` of X times g (NULL: 1)
__device__ __forceinline__ float row_sum32(const float *X, const float *g, int lane) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < WT; r += 4) {
        const float4 x = *reinterpret_cast<const float4 *>(X + lane * WRS + r);
        if (g) {
            const float4 y = *reinterpret_cast<const float4 *>(g + r);
            s = fmaf(x.x, y.x, s);
            s = fmaf(x.y, y.y, s);
            s = fmaf(x.z, y.z, s);
            s = fmaf(x.w, y.w, s);
        } else {
            s += (x.x + x.y) + (x.z + x.w);
        }
    }
    return s;
}

template <int H>
__global__ void __launch_bounds__(32 * BW, 2) k_warp_fd_backward(TrainArgs a) {
    using L = WL<H>;
    using S = WW<H>;
    using R = WRows<H>;
    constexpr int NT = 32 * BW;
    static_assert(R::ROWS * WRS >= L::cbo + 1, "a warp's rows must hold its gradient");
    extern __shared__ float4 smem4[];
    float *sw = reinterpret_cast<float *>(smem4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *all = sw + S::END, *rows = all + warp * R::ROWS * WRS, *gr = rows + R::G * WRS;
    const int c0 = a.chunk_off[0], total = a.chunk_off[a.NC] - c0;
    auto act = [&](float v, int, int) { return softplus_f32(v, a.beta, a.inv_beta); };
    for (int ci = blockIdx.x; ci < total; ci += gridDim.x) {
        const int cell = chunk_key(a.chunk_off, 0, a.NC, c0 + ci);
        const int j = c0 + ci - a.chunk_off[cell];
        const int beg = a.off[cell] + j * CHUNK, end = min(beg + CHUNK, a.off[cell + 1]);
        __syncthreads();
        load_cell<H, true>(a.params + (int64_t)cell * a.p_cell, sw, NT);
#pragma unroll
        for (int k = 27; k < 32; ++k) rows[k * WRS + lane] = 0.f;  // inputs past the encoding
        __syncthreads();
        float dw[H][8][4], db[H], dwo = 0.f, dbo = 0.f;
#pragma unroll
        for (int l = 0; l < H; ++l) {
            db[l] = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) dw[l][i][k] = 0.f;
        }
        for (int tb = beg + WT * warp; tb < end; tb += WT * BW) {
            {
                float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
                float g = 0.f;
                if (tb + lane < end) {
                    r = a.sorted[tb + lane];
                    g = a.g_fd[__float_as_int(r.w)];
                }
                encode_record(rows, lane, r.x, r.y, r.z);
                gr[lane] = g;
                dbo += g;
            }
            __syncwarp();
            TileMap<32, WT> m(lane);
            m.bias_shared(sw + S::b(0));
            m.template mm_shared<28>(sw + S::T(0), WTS, rows, WRS);
            m.store(rows + R::A(1) * WRS, WRS, act);
            __syncwarp();
#pragma unroll 1
            for (int l = 1; l < H; ++l) {
                m.bias_shared(sw + S::b(l));
                m.template mm_shared<32>(sw + S::T(l), WTS, rows + R::A(l) * WRS, WRS);
                m.store(rows + R::A(l + 1) * WRS, WRS, act);
                __syncwarp();
            }
            dwo += row_sum32(rows + R::A(H) * WRS, gr, lane);
            __syncwarp();
            {  // D_H = w_o g . softplus'(A_H)
                float *own = rows + R::A(H) * WRS;
                m.zero();
                m.store(own, WRS, [&](float, int u, int s) {
                    return sw[S::wo + u] * gr[s] * dsoftplus_from_act(own[u * WRS + s], a.beta);
                });
            }
            __syncwarp();
#pragma unroll
            for (int l = H - 1; l >= 1; --l) {  // hidden layer l's weight gradient, then D_l over A_l
                const float *D = rows + R::A(l + 1) * WRS;
                float *own = rows + R::A(l) * WRS;
                grad_tile32(D, own, dw[l], lane);
                db[l] += row_sum32(D, nullptr, lane);
                m.zero();
                m.template mm_shared<32>(sw + S::R(l), 32, D, WRS);
                __syncwarp();  // A_l has been read
                m.store(own, WRS, [&](float v, int u, int s) { return v * dsoftplus_from_act(own[u * WRS + s], a.beta); });
                __syncwarp();
            }
            grad_tile32(rows + R::A(1) * WRS, rows, dw[0], lane);
            db[0] += row_sum32(rows + R::A(1) * WRS, nullptr, lane);
            __syncwarp();
        }
        // the chunk's gradient: each warp's in its rows, canonical order; then summed over the warps
        __syncwarp();
        const int og = lane >> 3, ig = lane & 7;
#pragma unroll
        for (int l = 0; l < H; ++l) {
            const int K = l == 0 ? 27 : 32, cW = l == 0 ? L::cW0 : L::cH + (l - 1) * L::HL;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (ig + 8 * k < K) rows[cW + (og + 4 * i) * K + ig + 8 * k] = dw[l][i][k];
            rows[cW + 32 * K + lane] = db[l];
        }
        rows[L::cWo + lane] = dwo;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dbo += __shfl_xor_sync(0xffffffffu, dbo, o);
        if (lane == 0) rows[L::cbo] = dbo;
        __syncthreads();
        const int nw = min(BW, (end - beg + WT - 1) / WT);  // warps that had a tile
        float *gcell = a.grad + (int64_t)cell * a.p_cell;
        for (int e = tid; e < L::cWo + 33; e += NT) {
            const int q = e < L::cWo + 32 ? e : L::cbo;
            float v = 0.f;
            for (int w = 0; w < nw; ++w) v += all[w * R::ROWS * WRS + q];
            if (v != 0.f) atomicAdd(gcell + q, v);
        }
    }
}

// ------------------------------------------------------------------ sample centres
// Sample centres run the colour MLP as well; their tiles are 16 records, so that the backward's eight warps of
// rows and the cell's weights fit in shared memory and its 156 accumulators in registers.
constexpr int CT = 16;                 // records per warp tile
constexpr int CRS = row_stride(CT);
constexpr int CFW = 8, CBW = 8;        // warps per block, forward and backward

// what the SDF layers of WW lack: the output layer's T_o[k][16] and biases, the colour layers C0[i][o] (rows
// past 33 zero) and C1[c][k], and for the backward W_o[o][k] and C0[o][i]
template <int H>
struct WC {
    static constexpr int To = WW<H>::END, bo = To + 512, C0 = bo + 16, c0 = C0 + 36 * WTS, C1 = c0 + 32, c1 = C1 + 96;
    static constexpr int FEND = c1 + 4, Wo = FEND, Cr = Wo + 512, END = Cr + 32 * WTS;
};
template <int H, bool BACKWARD>
__device__ __forceinline__ void load_centre_cell(const float *__restrict__ cw, float *sw, int nt) {
    using L = WL<H>;
    using S = WC<H>;
    const int tid = threadIdx.x;
    load_cell<H, BACKWARD>(cw, sw, nt);
    for (int j = tid; j < 512; j += nt) {
        const float v = __ldg(cw + L::cWo + j);
        sw[S::To + (j & 31) * 16 + (j >> 5)] = v;
        if (BACKWARD) sw[S::Wo + j] = v;
    }
    for (int j = tid; j < 33 * 32; j += nt) {
        const float v = __ldg(cw + L::cC0 + j);
        const int o = j / 33, i = j - 33 * o;
        sw[S::C0 + i * WTS + o] = v;
        if (BACKWARD) sw[S::Cr + o * WTS + i] = v;
    }
    for (int j = tid; j < 3 * WTS; j += nt) sw[S::C0 + 33 * WTS + j] = 0.f;
    if (tid < 16) sw[S::bo + tid] = __ldg(cw + L::cbo + tid);
    if (tid < 32) sw[S::c0 + tid] = __ldg(cw + L::cc0 + tid);
    if (tid < 96) sw[S::C1 + tid] = __ldg(cw + L::cC1 + tid);
    if (tid < 3) sw[S::c1 + tid] = __ldg(cw + L::cc1 + tid);
}

// rows of a warp: the encoding and A_1 .. A_H (32 each), the output row d, the colour inputs U (z, n, gamma(v),
// three zero rows), the upstream of d, the colour hidden layer -- whose rows 0 .. 14 become z's deltas
// (forward alone: one buffer, a layer overwrites its input)
template <int H, bool KEEP>
struct CR {
    __host__ __device__ static constexpr int A(int l) { return KEEP ? 32 * l : 0; }
    static constexpr int Ud = KEEP ? 32 * (H + 1) : 32, U = Ud + 1, Dout = U + 36, Hc = Dout + 1, Dc = Hc + 32, ROWS = Dc + 3;
    static constexpr int GRAD = (WL<H>::cc1 + 3 + 3) / 4 * 4;  // a warp's gradient is put in its rows at the end
    static constexpr int FLOATS = ROWS * CRS > GRAD ? ROWS * CRS : GRAD;
};

// A tile forward: lane j and lane j + 16 share record j (q < 0: padding).  Leaves the activations, d and z, the
// colour inputs and the colour hidden layer in the rows; returns the colour logits and the difference gradient's
// length in lanes 0 .. 15.
template <int H, bool KEEP>
__device__ __forceinline__ void centre_tile(const TrainArgs &a, const float *sw, float *rows, int lane, float4 r,
                                            long long q, float (&lg)[3], float &gn) {
    using W = WW<H>;
    using S = WC<H>;
    using R = CR<H, KEEP>;
    const int j = lane & 15, h = lane >> 4;
    {  // Eq. 1: half 0 x and frequencies 0, 1, half 1 frequencies 2, 3; the colour inputs n and gamma(v)
        const float p[3] = {r.x, r.y, r.z};
        if (h == 0) {
#pragma unroll
            for (int c = 0; c < 3; ++c) rows[c * CRS + j] = p[c];
            if (!KEEP) rows[27 * CRS + j] = 0.f;
            float n[3] = {0.f, 0.f, 0.f}, g[3];
            if (q >= 0) gn = fd_normal(a, q, g, n);
#pragma unroll
            for (int c = 0; c < 3; ++c) rows[(R::U + 15 + c) * CRS + j] = n[c];
        } else {
            float v[3] = {0.f, 0.f, 0.f}, e[16];
            if (q >= 0) load3(a.w + 3 * (q / a.S), v);
            encode3<2, 16>(v[0], v[1], v[2], e);
#pragma unroll
            for (int k = 0; k < 15; ++k) rows[(R::U + 18 + k) * CRS + j] = e[k];
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
            const int k = 2 * h + kk;
            const float f = (float)(1 << k);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float sn, cs;
                sincospif(f * p[c], &sn, &cs);
                rows[(3 + 6 * k + c) * CRS + j] = sn;
                rows[(6 + 6 * k + c) * CRS + j] = cs;
            }
        }
    }
    __syncwarp();
    auto act = [&](float v, int, int) { return softplus_f32(v, a.beta, a.inv_beta); };
    TileMap<32, CT> m(lane);
#pragma unroll
    for (int l = 0; l < H; ++l) {
        m.bias_shared(sw + W::b(l));
        if (l == 0) m.template mm_shared<28>(sw + W::T(0), WTS, rows, CRS);
        else m.template mm_shared<32>(sw + W::T(l), WTS, rows + R::A(l) * CRS, CRS);
        if (!KEEP) __syncwarp();
        m.store(rows + R::A(l + 1) * CRS, CRS, act);
        __syncwarp();
    }
    {  // the 16 outputs [d, z]: lane (h, o) output o of records 8 h .. 8 h + 7
        const float *X = rows + R::A(H) * CRS + 8 * h;
        float out[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) out[i] = sw[S::bo + j];
#pragma unroll 4
        for (int k = 0; k < 32; ++k) {
            const float w = sw[S::To + k * 16 + j];
            const float4 x = *reinterpret_cast<const float4 *>(X + k * CRS),
                         y = *reinterpret_cast<const float4 *>(X + k * CRS + 4);
            const float xa[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) out[i] = fmaf(w, xa[i], out[i]);
        }
        float *o = rows + (R::Ud + j) * CRS + 8 * h;  // d, then z in U's rows 0 .. 14
        *reinterpret_cast<float4 *>(o) = make_float4(out[0], out[1], out[2], out[3]);
        *reinterpret_cast<float4 *>(o + 4) = make_float4(out[4], out[5], out[6], out[7]);
    }
    __syncwarp();
    m.bias_shared(sw + S::c0);
    m.template mm_shared<36>(sw + S::C0, WTS, rows + R::U * CRS, CRS);
    m.store(rows + R::Hc * CRS, CRS, [](float v, int, int) { return fmaxf(v, 0.f); });
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 3; ++c) lg[c] = sw[S::c1 + c];
    if (h == 0) {
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const float x = rows[(R::Hc + k) * CRS + j];
#pragma unroll
            for (int c = 0; c < 3; ++c) lg[c] = fmaf(sw[S::C1 + 32 * c + k], x, lg[c]);
        }
    }
}

// the rows no tile writes and every tile reads: inputs past the encoding, colour inputs past 33
template <class R>
__device__ __forceinline__ void centre_zero_rows(float *rows, int lane) {
    for (int i = lane; i < 5 * CRS; i += 32) rows[27 * CRS + i] = 0.f;
    for (int i = lane; i < 3 * CRS; i += 32) rows[(R::U + 33) * CRS + i] = 0.f;
}

template <int H>
__global__ void __launch_bounds__(32 * CFW, 2) k_warp_centre_fwd(TrainArgs a) {
    using S = WC<H>;
    using R = CR<H, false>;
    extern __shared__ float4 smem4[];
    float *sw = reinterpret_cast<float *>(smem4);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *rows = sw + S::FEND + warp * R::ROWS * CRS;
    const int k0 = a.NC, k1 = 2 * a.NC;
    const int64_t nfd = 6 * (a.B * a.S + a.M);
    const int c0 = a.chunk_off[k0], total = a.chunk_off[k1] - c0;
    centre_zero_rows<R>(rows, lane);
    for (int ci = blockIdx.x; ci < total; ci += gridDim.x) {
        const int key = chunk_key(a.chunk_off, k0, k1, c0 + ci);
        const int j = c0 + ci - a.chunk_off[key];
        const int beg = a.off[key] + j * CHUNK, end = min(beg + CHUNK, a.off[key + 1]);
        __syncthreads();
        load_centre_cell<H, false>(a.params + (int64_t)(key - a.NC) * a.p_cell, sw, 32 * CFW);
        __syncthreads();
        for (int tb = beg + CT * warp; tb < end; tb += CT * CFW) {
            const int i = tb + (lane & 15);
            float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
            long long q = -1;
            if (i < end) {
                r = a.sorted[i];
                q = (long long)__float_as_int(r.w) - nfd;
            }
            float lg[3], gn;
            centre_tile<H, false>(a, sw, rows, lane, r, q, lg, gn);
            if (lane < 16 && q >= 0) {
                a.d_c[q] = rows[R::Ud * CRS + lane];
                a.rgb_c[3 * q] = sigmoid_f32(lg[0]);
                a.rgb_c[3 * q + 1] = sigmoid_f32(lg[1]);
                a.rgb_c[3 * q + 2] = sigmoid_f32(lg[2]);
            }
            __syncwarp();
        }
    }
}

// acc[i][j] += sum over the tile's records of D[og + 4 i] A[ig + 8 j], i < NI
template <int NI>
__device__ __forceinline__ void grad_tile16(const float *D, const float *A, float (&acc)[NI][4], int lane) {
    const float *d = D + (lane >> 3) * CRS, *x = A + (lane & 7) * CRS;
#pragma unroll 1
    for (int r = 0; r < CT; r += 4) {
        float4 xv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) xv[j] = *reinterpret_cast<const float4 *>(x + 8 * j * CRS + r);
#pragma unroll
        for (int i = 0; i < NI; ++i) fma44(*reinterpret_cast<const float4 *>(d + 4 * i * CRS + r), xv, acc[i]);
    }
}
// sum over the tile's records of x times y (y NULL: 1), rows of CT records
__device__ __forceinline__ float row_dot16(const float *x, const float *y) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < CT; r += 4) {
        const float4 u = *reinterpret_cast<const float4 *>(x + r);
        const float4 v = y ? *reinterpret_cast<const float4 *>(y + r) : make_float4(1.f, 1.f, 1.f, 1.f);
        s = fmaf(u.x, v.x, s);
        s = fmaf(u.y, v.y, s);
        s = fmaf(u.z, v.z, s);
        s = fmaf(u.w, v.w, s);
    }
    return s;
}

// Sample centres backward: the tile recomputed forward, the colour MLP's deltas, then the SDF's with upstream on d
// and z; writes the difference points' upstream.  Weight gradients stay in registers over the chunk as in
// k_warp_fd_backward: lane (og, ig) owns outputs og + 4 i and inputs ig + 8 j of every layer.
template <int H>
__global__ void __launch_bounds__(32 * CBW, 1) k_warp_centre_backward(TrainArgs a) {
    using L = WL<H>;
    using W = WW<H>;
    using S = WC<H>;
    using R = CR<H, true>;
    constexpr int NT = 32 * CBW;
    extern __shared__ float4 smem4[];
    float *sw = reinterpret_cast<float *>(smem4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *all = sw + S::END, *rows = all + warp * R::FLOATS;
    const int k0 = a.NC, k1 = 2 * a.NC;
    const int64_t nfd = 6 * (a.B * a.S + a.M);
    const int c0 = a.chunk_off[k0], total = a.chunk_off[k1] - c0;
    const float inv2h = 1.f / (2.f * a.h);
    for (int ci = blockIdx.x; ci < total; ci += gridDim.x) {
        const int key = chunk_key(a.chunk_off, k0, k1, c0 + ci);
        const int cell = key - k0;
        const int jc = c0 + ci - a.chunk_off[key];
        const int beg = a.off[key] + jc * CHUNK, end = min(beg + CHUNK, a.off[key + 1]);
        __syncthreads();
        load_centre_cell<H, true>(a.params + (int64_t)cell * a.p_cell, sw, NT);
        centre_zero_rows<R>(rows, lane);
        __syncthreads();
        float dw[H][8][4], dwo[4][4], dwc[8][4], db[H], dbo = 0.f, dbc0 = 0.f, dwc32 = 0.f, dc1[3], dbc1[3];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
                for (int l = 0; l < H; ++l) dw[l][i][k] = 0.f;
                dwc[i][k] = 0.f;
                if (i < 4) dwo[i][k] = 0.f;
            }
#pragma unroll
        for (int l = 0; l < H; ++l) db[l] = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) dc1[c] = dbc1[c] = 0.f;
        for (int tb = beg + CT * warp; tb < end; tb += CT * CBW) {
            const int i = tb + (lane & 15);
            float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
            long long q = -1;
            if (i < end) {
                r = a.sorted[i];
                q = (long long)__float_as_int(r.w) - nfd;
            }
            float lg[3], gn = 0.f, up[4] = {0.f, 0.f, 0.f, 0.f};
            if (lane < 16 && q >= 0) {  // the upstreams, on their way while the tile runs forward
#pragma unroll
                for (int c = 0; c < 3; ++c) up[c] = a.g_rgb[3 * q + c];
                up[3] = a.g_dc[q];
            }
            centre_tile<H, true>(a, sw, rows, lane, r, q, lg, gn);
            if (lane < 16) {  // logits -> colour delta; the upstream of d
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float rgb = sigmoid_f32(lg[c]);
                    const float dc = up[c] * rgb * (1.f - rgb);
                    rows[(R::Dc + c) * CRS + lane] = dc;
                    dbc1[c] += dc;
                }
                rows[R::Dout * CRS + lane] = up[3];
            }
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 3; ++c) dc1[c] += row_dot16(rows + (R::Hc + lane) * CRS, rows + (R::Dc + c) * CRS);
            __syncwarp();
            TileMap<32, CT> m(lane);
            {  // Dh = (Wc1^T Dc) . [Hc > 0] over Hc
                float *own = rows + R::Hc * CRS;
                const float *dc = rows + R::Dc * CRS;
                m.zero();
                m.store(own, CRS, [&](float, int u, int s) {
                    const float v = fmaf(sw[S::C1 + u], dc[s], fmaf(sw[S::C1 + 32 + u], dc[CRS + s],
                                                                   sw[S::C1 + 64 + u] * dc[2 * CRS + s]));
                    return own[u * CRS + s] > 0.f ? v : 0.f;
                });
            }
            __syncwarp();
            grad_tile16<8>(rows + R::Hc * CRS, rows + R::U * CRS, dwc, lane);
            dwc32 += row_dot16(rows + (R::Hc + lane) * CRS, rows + (R::U + 32) * CRS);
            dbc0 += row_dot16(rows + (R::Hc + lane) * CRS, nullptr);
            // input deltas over Dh: rows 0 .. 14 z's, 15 .. 17 the normal's
            m.zero();
            m.template mm_shared<32>(sw + S::Cr, WTS, rows + R::Hc * CRS, CRS);
            __syncwarp();
            m.store(rows + R::Hc * CRS, CRS, [](float v, int, int) { return v; });
            __syncwarp();
            if (lane < 16 && q >= 0) {  // the normal's delta to the difference records
                const float n[3] = {rows[(R::U + 15) * CRS + lane], rows[(R::U + 16) * CRS + lane],
                                    rows[(R::U + 17) * CRS + lane]};
                const float gx = rows[(R::Hc + 15) * CRS + lane], gy = rows[(R::Hc + 16) * CRS + lane],
                            gz = rows[(R::Hc + 17) * CRS + lane];
                const float nd = n[0] * gx + n[1] * gy + n[2] * gz;
                const float ig = gn > 0.f ? inv2h / gn : 0.f;
                const float dg[3] = {(gx - n[0] * nd) * ig, (gy - n[1] * nd) * ig, (gz - n[2] * nd) * ig};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    a.g_fd[6 * q + 2 * k] = dg[k];
                    a.g_fd[6 * q + 2 * k + 1] = -dg[k];
                }
            }
            // output layer: its gradient, then D_H = (Wo^T Dout) . softplus'(A_H) over A_H
            grad_tile16<4>(rows + R::Dout * CRS, rows + R::A(H) * CRS, dwo, lane);
            if (lane < 16) dbo += row_dot16(rows + (R::Dout + lane) * CRS, nullptr);
            {
                float *own = rows + R::A(H) * CRS;
                m.zero();
                m.template mm_shared<16>(sw + S::Wo, 32, rows + R::Dout * CRS, CRS);
                __syncwarp();
                m.store(own, CRS, [&](float v, int u, int s) { return v * dsoftplus_from_act(own[u * CRS + s], a.beta); });
            }
            __syncwarp();
#pragma unroll
            for (int l = H - 1; l >= 1; --l) {
                const float *D = rows + R::A(l + 1) * CRS;
                float *own = rows + R::A(l) * CRS;
                grad_tile16<8>(D, own, dw[l], lane);
                db[l] += row_dot16(D + lane * CRS, nullptr);
                m.zero();
                m.template mm_shared<32>(sw + W::R(l), 32, D, CRS);
                __syncwarp();
                m.store(own, CRS, [&](float v, int u, int s) { return v * dsoftplus_from_act(own[u * CRS + s], a.beta); });
                __syncwarp();
            }
            grad_tile16<8>(rows + R::A(1) * CRS, rows, dw[0], lane);
            db[0] += row_dot16(rows + (R::A(1) + lane) * CRS, nullptr);
            __syncwarp();
        }
        // the chunk's gradient: each warp's in its rows, canonical order; then summed over the warps
        const int og = lane >> 3, ig = lane & 7;
#pragma unroll
        for (int l = 0; l < H; ++l) {
            const int K = l == 0 ? 27 : 32, cW = l == 0 ? L::cW0 : L::cH + (l - 1) * L::HL;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (ig + 8 * k < K) rows[cW + (og + 4 * i) * K + ig + 8 * k] = dw[l][i][k];
            rows[cW + 32 * K + lane] = db[l];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (i < 4) rows[L::cWo + (og + 4 * i) * 32 + ig + 8 * k] = dwo[i][k];
                rows[L::cC0 + (og + 4 * i) * 33 + ig + 8 * k] = dwc[i][k];
            }
        if (lane < 16) rows[L::cbo + lane] = dbo;
        rows[L::cC0 + lane * 33 + 32] = dwc32;
        rows[L::cc0 + lane] = dbc0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            rows[L::cC1 + 32 * c + lane] = dc1[c];
            float v = dbc1[c];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) rows[L::cc1 + c] = v;
        }
        __syncthreads();
        const int nw = min(CBW, (end - beg + CT - 1) / CT);  // warps that had a tile
        float *gcell = a.grad + (int64_t)cell * a.p_cell;
        for (int e = tid; e < L::cc1 + 3; e += NT) {
            float v = 0.f;
            for (int w = 0; w < nw; ++w) v += all[w * R::FLOATS + e];
            if (v != 0.f) atomicAdd(gcell + e, v);
        }
    }
}

// ------------------------------------------------------------------ launchers
template <class F>
cudaError_t set_smem(F f, size_t bytes) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int H>
cudaError_t eval_d_h(const TrainArgs &a, int k0, int k1, float *out, int64_t chunks, int sm_count, cudaStream_t s) {
    const size_t sm = (WW<H>::FEND + FW * 32 * WRS) * sizeof(float);
    cudaError_t e = set_smem(k_warp_eval_d<H>, sm);
    if (e != cudaSuccess) return e;
    k_warp_eval_d<H><<<grid_for(sm_count, FB, chunks), 32 * FW, sm, s>>>(a, k0, k1, out);
    return cudaGetLastError();
}

template <int H>
cudaError_t centre_fwd_h(const TrainArgs &a, int64_t chunks, int sm_count, cudaStream_t s) {
    const size_t sm = (WC<H>::FEND + CFW * CR<H, false>::ROWS * CRS) * sizeof(float);
    cudaError_t e = set_smem(k_warp_centre_fwd<H>, sm);
    if (e != cudaSuccess) return e;
    k_warp_centre_fwd<H><<<grid_for(sm_count, 2, chunks), 32 * CFW, sm, s>>>(a);
    return cudaGetLastError();
}

template <int H>
cudaError_t centre_backward_h(const TrainArgs &a, int64_t chunks, int sm_count, cudaStream_t s) {
    const size_t sm = (WC<H>::END + CBW * CR<H, true>::FLOATS) * sizeof(float);
    cudaError_t e = set_smem(k_warp_centre_backward<H>, sm);
    if (e != cudaSuccess) return e;
    k_warp_centre_backward<H><<<grid_for(sm_count, 1, chunks), 32 * CBW, sm, s>>>(a);
    return cudaGetLastError();
}

template <int H>
cudaError_t fd_backward_h(const TrainArgs &a, int64_t chunks, int sm_count, cudaStream_t s) {
    const size_t sm = (WW<H>::END + BW * WRows<H>::ROWS * WRS) * sizeof(float);
    cudaError_t e = set_smem(k_warp_fd_backward<H>, sm);
    if (e != cudaSuccess) return e;
    k_warp_fd_backward<H><<<grid_for(sm_count, 2, chunks), 32 * BW, sm, s>>>(a);
    return cudaGetLastError();
}

int64_t fd_chunks(const TrainArgs &a) { return 6 * (a.B * a.S + a.M) / CHUNK + a.NC + 1; }
int64_t centre_chunks(const TrainArgs &a) { return a.B * a.S / CHUNK + a.NC + 1; }

}  // namespace

cudaError_t train_coarse_eval(const TrainArgs &a, int sm_count, cudaStream_t s) {
    const int64_t chunks = a.B * a.Ns / CHUNK + a.NC + 1;
    return a.H == 3 ? eval_d_h<3>(a, 0, a.NC, a.d_coarse, chunks, sm_count, s)
                    : eval_d_h<2>(a, 0, a.NC, a.d_coarse, chunks, sm_count, s);
}

cudaError_t train_fd_forward(const TrainArgs &a, int sm_count, cudaStream_t s) {
    return a.H == 3 ? eval_d_h<3>(a, 0, a.NC, a.d_fd, fd_chunks(a), sm_count, s)
                    : eval_d_h<2>(a, 0, a.NC, a.d_fd, fd_chunks(a), sm_count, s);
}

cudaError_t train_centre_forward(const TrainArgs &a, int sm_count, cudaStream_t s) {
    return a.H == 3 ? centre_fwd_h<3>(a, centre_chunks(a), sm_count, s)
                    : centre_fwd_h<2>(a, centre_chunks(a), sm_count, s);
}

cudaError_t train_centre_backward(const TrainArgs &a, int sm_count, cudaStream_t s) {
    return a.H == 3 ? centre_backward_h<3>(a, centre_chunks(a), sm_count, s)
                    : centre_backward_h<2>(a, centre_chunks(a), sm_count, s);
}

cudaError_t train_fd_backward(const TrainArgs &a, int sm_count, cudaStream_t s) {
    return a.H == 3 ? fd_backward_h<3>(a, fd_chunks(a), sm_count, s)
                    : fd_backward_h<2>(a, fd_chunks(a), sm_count, s);
}

}  // namespace kns
