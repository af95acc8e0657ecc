// kns_points.cu -- the batch field query (the vectorised per-cell MLP query of Sec. 3.3): d, the feature z
// and the analytic gradient of the SDF MLP of cell m(x) at each point, on warp tiles of same-cell points.
// kns:instantiate (compiled once per grid configuration)
//
// A warp takes a tile of up to P points of one cell and runs the MLP forward, and backward from the d row
// (in place), with the weights read from the cell's shading layout in global memory
// (kns_warp.cuh): 85 KB per tile at width 64, so what bounds a large batch is the latency and the number of
// those reads.  Batches of a few points per cell and more are therefore grouped first -- a count per cell, a
// segment per non-empty cell (segments in any order, so no scan across blocks), a scatter of (point, id) --
// and evaluated in tiles of 16 points, each tile's weights on their way to L2 while the warp's previous tile
// runs.  Smaller batches take one point per warp, ungrouped: nothing is gained by grouping when the cells
// hold about one point each.  A thread per point, each reading its own cell's weights, was what this
// replaced: 1,000,003 random points of 32^3 cells of width 64 took 52 ms, now 2.0 ms (2.9 GB of weights
// once from memory: 0.43 ms at 6.8 TB/s; 12 warps per SM, 60 % of their time waiting for weight rows); 4,096
// points of 16^3 cells of width 32 took 115 us, now 21 us (one wave of warps).
#include <algorithm>

#include "kns_shade.cuh"
#include "kns_warp.cuh"
#include "kns_wave.cuh"

namespace kns {
namespace {

constexpr int PWARPS = 4;  // warps per block

// softplus_beta'(s) = sigmoid(beta s), from the exponential softplus_f32 takes
__device__ __forceinline__ float dsoftplus(float s, float beta) {
    const float e = __expf(-beta * fabsf(s)), r = __fdividef(1.f, 1.f + e);
    return s < 0.f ? e * r : r;
}

// shared rows of a warp: the encoding, A_1 .. A_H, and rows for W_0^T D_1 beyond those of A_2 .. A_H.  The gradient takes
// softplus' from the sums, not from the activations as shading does: softplus_f32 rounds to zero where softplus' is below
// 6e-8.  Either they lie in the layer's own rows, and its activations in the rows of the next layer (the last one's in its
// own): `shifted`; or, for one point of width 32, a lane keeps its units' in registers.  (One point is bound by the
// weight rows on their way, and so by how the compiler orders their loads: shifted, a query of width 32 for d alone
// takes 17 us instead of 11 (64 points of a 16^3 grid); in registers, one of width 64 takes 52 us instead of 38.)
template <class C>
struct PL {
    __host__ __device__ static constexpr int A(int l) { return C::INP + (l - 1) * C::W; }
    __host__ __device__ static constexpr int act(int l, bool shifted) { return shifted && l < C::H ? A(l + 1) : A(l); }
    static constexpr int G = C::INP + C::W;  // W_0^T D_1 over A_2 .. A_H, dead by then
    static constexpr int R0 = SL<C>::R0;
    static constexpr int ROWS = G + ((C::H - 1) * C::W > R0 ? (C::H - 1) * C::W : R0);
};

// The tile's points are in lanes 0 .. P - 1 (px, py, pz; id < 0: padding); M maps layers of width W to the
// lanes, ME the encoding's gradient; GRAD: with the gradient, where the caller wants it (in a tile always; a branch between
// its layers would keep the next layer's first weight rows from being loaded ahead of it).
template <class C, class M, class ME, bool GRAD>
__device__ __forceinline__ void points_tile(const GridView &g, const float *__restrict__ cw, float *rows, int lane,
                                            float px, float py, float pz, int64_t id, float *sdf, float *feat,
                                            float *grad) {
    using L = SL<C>;
    using R = PL<C>;
    constexpr int P = M::P, RS = row_stride(P), W = C::W;
    constexpr bool SHIFT = GRAD && (P > 1 || W == 64);
    float slope[C::H][P == 1 ? M::NU : 1];  // one point: softplus' of the lane's units
    if (lane < P) {  // Eq. 1, one lane per point
        float in[C::INP];
        encode3<C::L>(px, py, pz, in);
#pragma unroll
        for (int k = 0; k < C::INP; ++k) rows[k * RS + lane] = in[k];
    }
    __syncwarp();
    M m(lane);
    m.fetch(cw + L::T0, W);
    auto act = [&](float v, int, int) { return softplus_f32(v, g.beta, g.inv_beta); };
    auto dact = [&](float v, int, int) { return dsoftplus(v, g.beta); };
    m.bias(cw + L::b0);
    m.template mm<C::INP>(cw + L::T0, W, rows, RS, cw + L::Tl(1), W);
    m.store(rows + R::act(1, SHIFT) * RS, RS, act);
    if constexpr (SHIFT) m.store(rows + R::A(1) * RS, RS, dact);
    if constexpr (P == 1) m.each([&](float v, int i) { slope[0][i] = dsoftplus(v, g.beta); });
    __syncwarp();
#pragma unroll
    for (int l = 2; l <= C::H; ++l) {
        m.bias(cw + L::bl(l - 1));
        m.template mm<W>(cw + L::Tl(l - 1), W, rows + R::act(l - 1, SHIFT) * RS, RS,
                         l < C::H ? cw + L::Tl(l) : cw + L::Wlr(C::H - 1), W);
        if constexpr (SHIFT) __syncwarp();  // every lane has read the input, whose rows are written next
        m.store(rows + R::act(l, SHIFT) * RS, RS, act);
        if (SHIFT && l < C::H) m.store(rows + R::A(l) * RS, RS, dact);
        if constexpr (P == 1) m.each([&](float v, int i) { slope[l - 1][i] = dsoftplus(v, g.beta); });
        __syncwarp();
    }
    if (feat) {  // the 16 outputs [d, z]: lane l < 16 output l of the first half of the points, lane l + 16 of the second
        constexpr int PH = P == 1 ? 1 : P / 2;
        const int o = lane & 15, j0 = P == 1 ? 0 : (lane >> 4) * PH;
        const float *X = rows + R::A(C::H) * RS + j0;
        float out[PH];
#pragma unroll
        for (int j = 0; j < PH; ++j) out[j] = __ldg(cw + L::bo + o);
#pragma unroll 8
        for (int k = 0; k < W; ++k) {
            const float w = __ldg(cw + L::To + k * 16 + o);
#pragma unroll
            for (int j = 0; j < PH; ++j) out[j] = fmaf(w, X[k * RS + j], out[j]);
        }
#pragma unroll
        for (int j = 0; j < PH; ++j) {
            const int64_t q = __shfl_sync(FULL, id, j0 + j);
            if (q < 0 || (P == 1 && lane >= 16)) continue;
            if (o == 0) sdf[q] = out[j];
            else feat[q * FEAT + o - 1] = out[j];
        }
    } else if (lane < P && id >= 0) {  // d alone
        float d = __ldg(cw + L::bo);
#pragma unroll 8
        for (int k = 0; k < W; k += 4) {
            const float4 w = __ldg(reinterpret_cast<const float4 *>(cw + L::wd + k));
            const float *h = rows + (R::A(C::H) + k) * RS + lane;
            d = fmaf(w.x, h[0], d);
            d = fmaf(w.y, h[RS], d);
            d = fmaf(w.z, h[2 * RS], d);
            d = fmaf(w.w, h[3 * RS], d);
        }
        sdf[id] = d;
    }
    __syncwarp();
    if (!GRAD || !grad) return;
    // D_H = w_d . softplus', over A_H
    m.store(rows + R::A(C::H) * RS, RS, [&](float v, int u, int) {
        if constexpr (P == 1 && !SHIFT) return __ldg(cw + L::wd + u) * slope[C::H - 1][u - m.u0];
        else return __ldg(cw + L::wd + u) * dsoftplus(v, g.beta);
    });
    __syncwarp();
#pragma unroll
    for (int l = C::H - 1; l >= 1; --l) {  // D_l = (W_l^T D_{l+1}) . softplus', over the latter
        m.zero();
        m.template mm<W>(cw + L::Wlr(l), W, rows + R::A(l + 1) * RS, RS, l > 1 ? cw + L::Wlr(l - 1) : nullptr, W);
        float *own = rows + R::A(l) * RS;
        m.store(own, RS, [&](float v, int u, int s) {
            if constexpr (P == 1 && !SHIFT) return v * slope[l - 1][u - m.u0];
            else return v * own[u * RS + s];
        });
        __syncwarp();
    }
    ME e(lane);
    e.fetch(cw + L::W0r, R::R0);
    e.zero();
    e.template mm<W>(cw + L::W0r, R::R0, rows + R::A(1) * RS, RS, nullptr, 0);
    e.store(rows + R::G * RS, RS, [](float v, int, int) { return v; });
    __syncwarp();
    // through the encoding: d sin(f p)/dp = f cos(f p), d cos(f p)/dp = -f sin(f p)
    for (int i = lane; i < 3 * P; i += 32) {
        const int j = i % P, c = i / P;
        const float *in = rows + j, *d = rows + R::G * RS + j;
        float gc = d[c * RS];
#pragma unroll
        for (int k = 0; k < C::L; ++k) {
            const float f = 3.14159265358979323846f * (float)(1 << k);
            gc = fmaf(d[(3 + 6 * k + c) * RS] * f, in[(6 + 6 * k + c) * RS], gc);
            gc = fmaf(-d[(6 + 6 * k + c) * RS] * f, in[(3 + 6 * k + c) * RS], gc);
        }
        rows[(R::A(1) + c) * RS + j] = gc;  // D_1 is dead: nothing reads it below
    }
    __syncwarp();
    if (lane < P && id >= 0)
#pragma unroll
        for (int c = 0; c < 3; ++c) grad[3 * id + c] = rows[(R::A(1) + c) * RS + lane];
    __syncwarp();
}

// One point per warp, in the order given.
template <class C, bool GRAD>
__global__ void __launch_bounds__(32 * PWARPS) points_direct_kernel(GridView g, const float *__restrict__ pts, int64_t n,
                                                                     float *sdf, float *feat, float *grad) {
    extern __shared__ __align__(16) float psm[];
    constexpr int RS = row_stride(1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *rows = psm + warp * PL<C>::ROWS * RS;
    const int64_t q = (int64_t)blockIdx.x * PWARPS + warp;
    if (q >= n) return;
    const float x = __ldg(pts + 3 * q), y = __ldg(pts + 3 * q + 1), z = __ldg(pts + 3 * q + 2);
    const int cell = cell_of(g, x, y, z);
    points_tile<C, UnitMap<C::W>, UnitMap<PL<C>::R0>, GRAD>(g, g.ws + (int64_t)cell * g.ws_stride, rows, lane, x, y, z,
                                                            lane == 0 ? q : -1, sdf, feat, grad);
}

// registers for as many blocks per SM as shared memory holds
template <class C, int P, bool GRAD>
__global__ void __launch_bounds__(32 * PWARPS, C::W == 32 ? 5 : 3) points_tile_kernel(GridView g, PointsScratch s, float *sdf,
                                                                                      float *feat, float *grad) {
    extern __shared__ __align__(16) float psm[];
    constexpr int RS = row_stride(P);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *rows = psm + warp * PL<C>::ROWS * RS;
    const int n_tiles = s.ctl[1];
    for (int t = blockIdx.x * PWARPS + warp; t < n_tiles; t += gridDim.x * PWARPS) {
        const int4 d = s.tiles[t];  // cell, first sorted point, points
        const int tn = t + gridDim.x * PWARPS;  // the next tile's weights start for L2 while this one runs
        if (lane == 0 && tn < n_tiles) {
            const int c = s.tiles[tn].x;
            prefetch_l2(g.ws + (int64_t)c * g.ws_stride, (GRAD ? SL<C>::C0t : SL<C>::W0r) * (int)sizeof(float));
        }
        float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
        int64_t id = -1;
        if (lane < d.z) {
            p = s.sorted[d.y + lane];
            id = __float_as_int(p.w);
        }
        points_tile<C, TileMap<C::W, P>, TileMap<PL<C>::R0, P>, GRAD>(g, g.ws + (int64_t)d.x * g.ws_stride, rows, lane, p.x,
                                                                      p.y, p.z, id, sdf, feat, grad);
    }
}

template <class C, int P, bool GRAD>
cudaError_t launch_tiles(const GridView &g, const PointsScratch &sc, int64_t n, float *sdf, float *feat, float *grad,
                         int sm_count, cudaStream_t s) {
    constexpr int smem = PWARPS * PL<C>::ROWS * row_stride(P) * (int)sizeof(float);
    static_assert(smem <= 200 * 1024, "point tiles do not fit in shared memory");
    static PerDevice per_sm;
    int nb = 0;
    cudaError_t e = resident_blocks(points_tile_kernel<C, P, GRAD>, 32 * PWARPS, smem, per_sm, nb);
    if (e != cudaSuccess) return e;
    const int64_t most = (n / P + g.ncl + PWARPS) / PWARPS;  // blocks that could have a tile
    points_tile_kernel<C, P, GRAD><<<(unsigned)std::min<int64_t>((int64_t)sm_count * nb, most), 32 * PWARPS, smem, s>>>(
        g, sc, sdf, feat, grad);
    return cudaGetLastError();
}

}  // namespace

template <class C>
cudaError_t launch_points_direct_cfg(const GridView &g, const float *pts, int64_t n, float *sdf, float *feat,
                                     float *grad, cudaStream_t s) {
    constexpr int smem = PWARPS * PL<C>::ROWS * row_stride(1) * (int)sizeof(float);
    // width 32 has one kernel for both (compiled for d alone, it has fewer loads under way)
    auto kernel = grad || C::W == 32 ? points_direct_kernel<C, true> : points_direct_kernel<C, C::W == 32>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kernel<<<(unsigned)((n + PWARPS - 1) / PWARPS), 32 * PWARPS, smem, s>>>(g, pts, n, sdf, feat, grad);
    return cudaGetLastError();
}

template <class C>
cudaError_t launch_points_tiles_cfg(const GridView &g, const PointsScratch &sc, int64_t n, float *sdf, float *feat,
                                    float *grad, int sm_count, cudaStream_t s) {
    return grad ? launch_tiles<C, kPointsTile, true>(g, sc, n, sdf, feat, grad, sm_count, s)
                : launch_tiles<C, kPointsTile, false>(g, sc, n, sdf, feat, grad, sm_count, s);
}

#ifdef KNS_W
using InstCfg = Cfg<KNS_W, KNS_H, KNS_L, KNS_LD>;
template cudaError_t launch_points_direct_cfg<InstCfg>(const GridView &, const float *, int64_t, float *, float *,
                                                       float *, cudaStream_t);
template cudaError_t launch_points_tiles_cfg<InstCfg>(const GridView &, const PointsScratch &, int64_t, float *,
                                                      float *, float *, int, cudaStream_t);
#endif

}  // namespace kns
