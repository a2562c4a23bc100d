// FP32 2D adjoint step on register tiles (the maps of adjoint2d.cu, the tiles of
// tile2d.cu): one launch per set and step, even n_x (odd n_x stays on the staged
// kernels: another order of the FP32 sums moves dL/dtheta in its seventh digit).  A warp holds 8 rows of 64
// columns; u = Ebar - C_b Bbar, the M sweeps of the forward tile give w, and the
// rows of w at the warps' borders go through shared memory once for the
// transposed Faraday update and the filter of jbar.  M + 1 barriers a step
// against one per row of the row pipeline, which stays the faster one on grids
// beyond twice the L2.  1024^2, m = 4, p = 3, us per launch against the row
// pipeline: TE 12.3 against 24.5, TM with jbar_z 14.1 against 25.2.
#include <cuda_runtime.h>
#include <math.h>

#include "fused2d.h"
#include "tile2d.cuh"

namespace fmx {
namespace {

using namespace tile2d;

// Reach of a tile's outputs.  w is needed WL rows (columns) before the tile and
// WH after its last: Faraday one after, TM's averages one before and after,
// jbar's filter P on either side; every sweep takes one more on either side
// and u one more of Bbar before.
template <int POL, int M, int P, bool HJB>
struct AdjHalo {
    static constexpr int PF = HJB ? P : 0;
    static constexpr int WL = PF > (POL == TM ? 1 : 0) ? PF : (POL == TM ? 1 : 0);
    static constexpr int WH = PF > 1 ? PF : 1;
    static constexpr int HY = WL + M;                      // rows below the tile
    static constexpr int HC = (WL + M + 1 + 1) / 2 * 2;    // columns left of the tile (even)
    static constexpr int TWX = (64 - HC - WH - M) / 2 * 2;  // columns and rows a tile can write
    static constexpr int THX = R * NW - HY - WH - M;
    static_assert(TWX >= 2 && THX >= 1 && R >= P, "halo larger than the tile");
};

template <int POL, int M, int P, bool HJB>
__device__ __forceinline__ void adj_tile(const Adj2dArgs<float> &a, const Geo &g, const Coef2 &c, int tw, int th, int x0,
                                         int y0, int zero, float2 *sm) {
    using H = AdjHalo<POL, M, P, HJB>;
    constexpr int HY = H::HY, HC = H::HC, NC = POL == TE ? 2 : 1;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    float2 *s_row = sm + lane;
    float2 *s_pub = sm + NC * R * NW * 32 + lane;
    auto pub = [&](int buf, int slot, int w) -> float2 & { return s_pub[((buf * 3 + slot) * NW + w) * 32]; };
    auto row = [&](int q, int r) -> float2 & { return s_row[(q * R * NW + r) * 32]; };
    const int cg = x0 - HC + 2 * lane;
    int xc = cg % g.nx;
    if (xc < 0) xc += g.nx;
    const bool xout = 2 * lane >= HC && 2 * lane < HC + tw && cg < g.nx;
    const int ry = wp * R - HY;  // first own row, relative to the tile's first
    const int pitch = (int)g.pitch, plane = g.ny * pitch;
    int yw = (y0 + ry) % g.ny;
    if (yw < 0) yw += g.ny;
    const int orow0 = yw * pitch + xc + zero;
    auto need = [&](int lo, int hi) { return ry <= hi && ry + R - 1 >= lo; };
    auto next_row = [&](int &o) {
        o += pitch;
        if (o >= plane) o -= plane;
    };
    auto ld = [&](const float *p, int o) { return ld2(p + o); };
    auto st = [&](float *p, int o, f2 v) { *reinterpret_cast<float2 *>(p + o) = v; };
    const float *inE0 = POL == TE ? a.Eb[0] : a.Eb[2], *inE1 = a.Eb[1];
    const float *inB0 = POL == TE ? a.Bb[2] : a.Bb[0], *inB1 = a.Bb[1];
    float *oE0 = POL == TE ? a.Ebo[0] : a.Ebo[2], *oE1 = a.Ebo[1];
    float *oB0 = POL == TE ? a.Bbo[2] : a.Bbo[0], *oB1 = a.Bbo[1];
    float *oJ0 = POL == TE ? a.Jbo[0] : a.Jbo[2], *oJ1 = a.Jbo[1];
    const f2 z2 = mk(0.f, 0.f);
    const int oown = (y0 + ry) * pitch + xc;  // output offset of the first own row (used for rows of the tile)

    // ---------------- u = Ebar - C_b Bbar ----------------
    f2 d[NC][R];
    if (need(-HY, th - 1 + H::WH + M)) {
        int o = orow0 - pitch;  // the row below
        if (yw == 0) o += plane;
        f2 bp = ld(inB0, o);  // TE: Bbar_z, TM: Bbar_x of the row below
        o = orow0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const f2 e0 = ld(inE0, o), b0 = ld(inB0, o);
            if constexpr (POL == TE) {
                const f2 e1 = ld(inE1, o);
                d[0][j] = fma(c.ky, fma(b0, m1(), bp), e0);
                d[NC - 1][j] = fma(c.kx, mk(b0.x - up1(b0.y), b0.y - b0.x), e1);
            } else {
                const f2 b1 = ld(inB1, o);
                const f2 dxby = mk(b1.x - up1(b1.y), b1.y - b1.x);
                d[0][j] = fma(mul(c.kx, dxby), m1(), fma(c.ky, fma(bp, m1(), b0), e0));
            }
            bp = b0;
            next_row(o);
        }
    } else {
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int q = 0; q < NC; ++q) d[q][j] = z2;
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
        if (ry + j >= 0 && ry + j < th && xout) {
            st(oE0, oown + j * pitch, d[0][j]);
            if constexpr (POL == TE) st(oE1, oown + j * pitch, d[NC - 1][j]);
        }
    }
    // ---------------- w = sum_{s<=M} A^s u ----------------
    const int wb = wp > 0 ? wp - 1 : 0, wa = wp < NW - 1 ? wp + 1 : wp;
    sweeps<POL, M>(d, c, wp, wb, wa, row, pub,
                   [&](int s) { return need(-H::WL - (M - s), th - 1 + H::WH + (M - s)); });
    // the border rows of w (the shared rows are the warp's own until here)
    constexpr int BR = H::PF > 1 ? H::PF : 1;
#pragma unroll
    for (int j = 0; j < R; ++j)
        if (j < BR || j >= R - BR)
#pragma unroll
            for (int q = 0; q < NC; ++q) row(q, wp * R + j) = d[q][j];
    __syncthreads();
    if (!need(0, th - 1)) return;
    auto w = [&](int q, int r) -> f2 {  // row wp R + r; r in [-BR, R - 1 + BR]
        if (r >= 0 && r < R) return d[q][r];
        const int k = wp * R + r;
        return row(q, k < 0 ? 0 : (k > R * NW - 1 ? R * NW - 1 : k));
    };
    // ---------------- Bbar += S C_f w ----------------
    {
        int o = orow0;
        [[maybe_unused]] auto cyf = [&](f2 v) { return fma(c.kx, mk(v.x - v.y, v.y - dn1(v.x)), z2); };
        [[maybe_unused]] f2 cym = z2, cy0 = z2;
        if constexpr (POL == TM) {
            cym = cyf(w(0, -1));
            cy0 = cyf(w(0, 0));
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const f2 b0 = ld(inB0, o), w0 = w(0, j), wn = w(0, j + 1);
            const bool out = ry + j >= 0 && ry + j < th && xout;
            if constexpr (POL == TE) {
                const f2 wy = w(NC - 1, j);
                const f2 dxwy = mk(wy.y - wy.x, dn1(wy.x) - wy.y), dywx = fma(w0, m1(), wn);
                const f2 bo = fma(c.kx, dxwy, fma(mul(c.ky, dywx), m1(), b0));
                if (out) st(oB0, oown + j * pitch, bo);
            } else {
                const f2 b1 = ld(inB1, o);
                const f2 cx = fma(c.ky, fma(w0, m1(), wn), z2), cyp = cyf(wn);
                const f2 bxo = fma(c6(), fma(cx, m2(), xsum(cx, up1(cx.y), dn1(cx.x))), add(b0, cx));
                const f2 byo = fma(c6(), fma(cy0, m2(), add(cyp, cym)), add(b1, cy0));
                if (out) {
                    st(oB0, oown + j * pitch, bxo);
                    st(oB1, oown + j * pitch, byo);
                }
                cym = cy0;
                cy0 = cyp;
            }
            next_row(o);
        }
    }
    // ---------------- jbar = -q F w ----------------
    if constexpr (HJB) {
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            float *oj = q == 0 ? oJ0 : oJ1;
            f2 v[2 * P + 1];
#pragma unroll
            for (int k = 0; k < 2 * P; ++k) v[k + 1] = w(q, k - P);
#pragma unroll
            for (int j = 0; j < R; ++j) {
#pragma unroll
                for (int k = 0; k < 2 * P; ++k) v[k] = v[k + 1];
                v[2 * P] = w(q, j + P);
                f2 f = binom_taps<P>(v);
                if constexpr (P > 0) f = binom_x<P>(f);
                const f2 jb = mul(c.qf, fma(f, m1(), z2));
                if (oj && ry + j >= 0 && ry + j < th && xout) st(oj, oown + j * pitch, jb);
            }
        }
    }
}

template <int POL, int M, int P, bool HJB>
__global__ void __launch_bounds__(32 * NW, 2) k_adj_tile2d(Adj2dArgs<float> a, Geo g, Coef2 c, Tile2dGeo t) {
    extern __shared__ __align__(16) float2 tsm[];
    const int zero = dependency_wait();
    const int x0 = (int)(blockIdx.x % t.ntx) * t.tw, y0 = (int)(blockIdx.x / t.ntx) * t.th;
    const int th = min(t.th, g.ny - y0);
    adj_tile<POL, M, P, HJB>(a, g, c, t.tw, th, x0, y0, zero, tsm);
}

}  // namespace

template <int POL, int M, int P, bool HJB>
void launch_adj_tile2d(const Geo &g, const Coef2 &c, const Adj2dArgs<float> &a, cudaStream_t s) {
    using H = AdjHalo<POL, M, P, HJB>;
    constexpr size_t smem = (size_t)((POL == TE ? 2 : 1) * R * NW + 6 * NW) * 32 * sizeof(float2);
    auto k = k_adj_tile2d<POL, M, P, HJB>;
    static const bool attr =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
    (void)attr;  // a failure shows up in the launch
    const Tile2dGeo t = cover(g.nx, g.ny, H::TWX, H::THX);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(t.ntx * t.nty);
    cfg.blockDim = dim3(32 * NW);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k, a, g, c, t);
}

#define FMX_ADJ_TILE(POL, M, P, HJB) \
    template void launch_adj_tile2d<POL, M, P, HJB>(const Geo &, const Coef2 &, const Adj2dArgs<float> &, cudaStream_t);
#define FMX_ADJ_TILE_P(M, P) \
    FMX_ADJ_TILE(TE, M, P, false) FMX_ADJ_TILE(TE, M, P, true) FMX_ADJ_TILE(TM, M, P, false) FMX_ADJ_TILE(TM, M, P, true)
#define FMX_ADJ_TILE_M(M) FMX_ADJ_TILE_P(M, 0) FMX_ADJ_TILE_P(M, 1) FMX_ADJ_TILE_P(M, 2) FMX_ADJ_TILE_P(M, 3)
FMX_ADJ_TILE_M(0)
FMX_ADJ_TILE_M(1)
FMX_ADJ_TILE_M(2)
FMX_ADJ_TILE_M(3)
FMX_ADJ_TILE_M(4)

}  // namespace fmx
