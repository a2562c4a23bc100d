// FP32 2D step on register tiles (Sec. 2.2.2, TE set Ex, Ey, Bz; jx, jy and TM
// set Ez, Bx, By; jz apart, as in fused2d_pol.cu): one launch per step, one
// CTA per tile and set.
//
// A warp spans the tile's width: 32 lanes x 2 columns, with the x-halo of the
// whole step inside those 64 columns, so every x-neighbour is a warp shuffle.
// A warp holds R consecutive rows in registers and the CTA's NW warps stack
// up to R NW rows, the y-halo among them; a stage (current filter, source,
// one sweep, the E and Faraday update) works on all rows at once and hands
// only the rows at the warps' borders on through shared memory, one barrier
// per stage.  Columns and rows whose neighbours lie outside the tile go wrong
// by one per stage and are the halo.
//
// Against the row pipeline (pol_tile.cuh: a barrier per row, 50 rows deep
// before the first output of a segment is complete) a step has M + 2 barriers
// in all, and neither shared-memory neighbour loads nor ring addresses.
#include <cuda_runtime.h>
#include <math.h>

#include "fused2d.h"
#include "pol_tile.cuh"
#include "tile2d.cuh"

namespace fmx {
namespace {

using namespace tile2d;

// Grids of at most this many cells run both sets in one launch on the grid's
// own stream: the tiles of both (48 x 49 columns and rows at m = 4, p = 3; 200 at
// 443^2) are one wave of at most two CTAs per SM, and a step is not worth a second
// stream's fork and join.
constexpr double kTileOneLaunchCells = 192.0 * 1024.0;

template <int M, int P, bool HJ>
struct TileHalo {
    static constexpr int PX = (HJ && P > 1) ? P : 1;
    static constexpr int HY = M + PX;               // rows below the tile; HY + 1 above
    static constexpr int HC = (M + PX + 1) / 2 * 2;  // columns left of the tile (even) and right of it
};

template <int POL, int M, int P, bool HJ, bool SEAM>
__device__ __forceinline__ void tile_step(const Fused2dArgs<float> &a, const Geo &g, const Coef2 &c, int tw, int th,
                                          int x0, int y0, int zero, float2 *sm) {
    using H = TileHalo<M, P, HJ>;
    constexpr int HY = H::HY, HC = H::HC, NC = POL == TE ? 2 : 1, NB = POL == TE ? 1 : 2;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    // shared memory, one float2 per lane: rows [NC][R NW] (the raw current,
    // then dE'), border rows [2][3][NW]
    float2 *s_row = sm + lane;
    float2 *s_pub = sm + NC * R * NW * 32 + lane;
    auto pub = [&](int buf, int slot, int w) -> float2 & { return s_pub[((buf * 3 + slot) * NW + w) * 32]; };
    auto row = [&](int q, int r) -> float2 & { return s_row[(q * R * NW + r) * 32]; };

    const int cg = x0 - HC + 2 * lane;
    int xc = cg % g.nx;
    if (xc < 0) xc += g.nx;
    [[maybe_unused]] int dxc = 1;
    [[maybe_unused]] bool xlast = false;
    if constexpr (SEAM) {
        dxc = xc + 1 == g.nx ? 1 - g.nx : 1;
        xlast = cg + 1 >= g.nx;
    }
    const bool xout = 2 * lane >= HC && 2 * lane < HC + tw && cg < g.nx;
    const int ry = wp * R - HY;  // first own row, relative to the tile's first
    const int pitch = (int)g.pitch, plane = g.ny * pitch;
    int yw = (y0 + ry) % g.ny;
    if (yw < 0) yw += g.ny;
    const int orow0 = yw * pitch + xc + zero;
    // own rows overlap the tile rows lo .. hi
    auto need = [&](int lo, int hi) { return ry <= hi && ry + R - 1 >= lo; };
    auto ld = [&](const float *p, int o) {
        if constexpr (SEAM) return mk(tile2d::ld(p + o), tile2d::ld(p + o + dxc));
        else return ld2(p + o);
    };
    auto st = [&](float *p, int o, f2 v) {
        if constexpr (SEAM) {
            p[o] = v.x;
            if (!xlast) p[o + 1] = v.y;
        } else {
            *reinterpret_cast<float2 *>(p + o) = v;
        }
    };
    const float *inB0 = POL == TE ? a.B[2] : a.B[0], *inB1 = a.B[1];
    const float *inE0 = POL == TE ? a.E[0] : a.E[2], *inE1 = a.E[1];
    const f2 z2 = mk(0.f, 0.f);

    // ---------------- inputs: B and j of the own rows ----------------
    f2 d[NC][R];  // the current, then dE' and dE of the own rows
    f2 b[NB][R];
    {
        int o = orow0;
        const bool in = need(-HY, th + HY);
#pragma unroll
        for (int j = 0; j < R; ++j) {
            b[0][j] = in ? ld(inB0, o) : z2;
            if constexpr (POL == TM) b[1][j] = in ? ld(inB1, o) : z2;
            if constexpr (HJ) {
                d[0][j] = in ? ld(POL == TE ? a.J[0] : a.J[2], o) : z2;
                if constexpr (POL == TE) d[1][j] = in ? ld(a.J[1], o) : z2;
            }
            o += pitch;
            if (o >= plane) o -= plane;
        }
    }
    // ---------------- source ----------------
    if constexpr (HJ && P > 0) {
#pragma unroll
        for (int q = 0; q < NC; ++q)
#pragma unroll
            for (int j = 0; j < R; ++j) row(q, wp * R + j) = d[q][j];
    }
    pub(1, 0, wp) = b[0][R - 1];
    if constexpr (POL == TM) {
        pub(1, 1, wp) = b[1][R - 1];
        pub(1, 2, wp) = b[1][0];
    }
    __syncthreads();
    const int wb = wp > 0 ? wp - 1 : 0, wa = wp < NW - 1 ? wp + 1 : wp;  // warps below and above (at the edges: garbage rows)
    if (need(-M, th + M)) {
        if constexpr (HJ && P > 0) {
#pragma unroll
            for (int q = 0; q < NC; ++q) {
                // y binomial over rows j-P .. j+P (a rolling window), then the
                // x binomial; weights unnormalised, 1/4^2P folded into qf
                f2 w[2 * P + 1];
                auto jrow = [&](int r) {  // own row wp R + r
                    const int k = wp * R + r;
                    return (r >= 0 && r < R) ? d[q][r] : row(q, k < 0 ? 0 : (k > R * NW - 1 ? R * NW - 1 : k));
                };
#pragma unroll
                for (int k = 0; k < 2 * P; ++k) w[k + 1] = jrow(k - P);
                f2 f[R];
#pragma unroll
                for (int j = 0; j < R; ++j) {
#pragma unroll
                    for (int k = 0; k < 2 * P; ++k) w[k] = w[k + 1];
                    w[2 * P] = jrow(j + P);
                    f[j] = binom_taps<P>(w);
                }
#pragma unroll
                for (int j = 0; j < R; ++j) d[q][j] = binom_x<P>(f[j]);
            }
        }
        if constexpr (POL == TE) {
            f2 bp = pub(1, 0, wb);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const f2 bz = b[0][j];
                const float bzl = up1(bz.y);
                f2 d0 = mul(c.ky, sub(bz, bp));
                f2 d1 = mul(c.kx, mk(bzl - bz.x, bz.x - bz.y));
                if constexpr (HJ) {
                    d0 = fma(c.qf, fma(d[0][j], m1(), z2), d0);
                    d1 = fma(c.qf, fma(d[1][j], m1(), z2), d1);
                }
                d[0][j] = d0;
                d[1][j] = d1;
                bp = bz;
            }
        } else {
            auto alpha_x = [&](f2 v) { return fma(c6(), fma(v, m2(), xsum(v, up1(v.y), dn1(v.x))), v); };
            f2 axp = alpha_x(pub(1, 0, wb));
            f2 byp = pub(1, 1, wb);
            const f2 bya = pub(1, 2, wa);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const f2 ax = alpha_x(b[0][j]);
                const f2 by0 = b[1][j], byn = j < R - 1 ? b[1][j + 1] : bya;
                const f2 ay = fma(c6(), fma(by0, m2(), add(byn, byp)), by0);
                const float ayl = up1(ay.y);
                f2 d0 = fma(c.kx, mk(ay.x - ayl, ay.y - ay.x), mul(fma(c.ky, sub(ax, axp), z2), m1()));
                if constexpr (HJ) d0 = fma(c.qf, fma(d[0][j], m1(), z2), d0);
                d[0][j] = d0;
                axp = ax;
                byp = by0;
            }
        }
    }
    // ---------------- sweeps ----------------
    sweeps<POL, M>(d, c, wp, wb, wa, row, pub, [&](int s) { return need(s - M, th + M - s); });
    f2 e[NC][R], bf[NB][R];  // E^n of the own rows; B again for the Faraday update
    // ---------------- E and Faraday updates ----------------
    const bool act = need(0, th);
    {
        int o = orow0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
            if (act) {
                e[0][j] = ld(inE0, o);
                if constexpr (POL == TE) e[1][j] = ld(inE1, o);
                bf[0][j] = ld(inB0, o);
                if constexpr (POL == TM) bf[1][j] = ld(inB1, o);
            } else {
                e[0][j] = bf[0][j] = z2;
                if constexpr (POL == TE) e[1][j] = z2;
                if constexpr (POL == TM) bf[1][j] = z2;
            }
            o += pitch;
            if (o >= plane) o -= plane;
        }
    }
#pragma unroll
    for (int j = 0; j < R; ++j)
#pragma unroll
        for (int q = 0; q < NC; ++q) d[q][j] = add(e[q][j], d[q][j]);
    constexpr int EB = M & 1;  // the buffer the last sweep did not read
    pub(EB, 1, wp) = d[0][0];
    __syncthreads();
    if (!act) return;
    const f2 ea = pub(EB, 1, wa);
    float *oE0 = POL == TE ? a.Eo[0] : a.Eo[2], *oE1 = a.Eo[1];
    float *oB0 = POL == TE ? a.Bo[2] : a.Bo[0], *oB1 = a.Bo[1];
    const int o0 = (y0 + ry) * pitch + xc;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const f2 e0 = d[0][j], en = j < R - 1 ? d[0][j + 1] : ea;
        const float er = dn1(POL == TE ? d[NC - 1][j].x : e0.x);
        f2 bo0, bo1 = z2;
        if constexpr (POL == TE) {
            // Bz -= kx (Ey[i+1] - Ey[i]) - ky (Ex[j+1] - Ex[j])
            const f2 ey = d[1][j];
            bo0 = fma(c.ky, sub(en, e0), fma(fma(c.kx, mk(ey.y - ey.x, er - ey.y), z2), m1(), bf[0][j]));
        } else {
            // Bx -= ky (Ez[j+1] - Ez[j]);  By += kx (Ez[i+1] - Ez[i])
            bo0 = fma(fma(c.ky, sub(en, e0), z2), m1(), bf[0][j]);
            bo1 = fma(c.kx, mk(e0.y - e0.x, er - e0.y), bf[1][j]);
        }
        const int r = ry + j;
        if (r >= 0 && r < th && xout) {
            const int o = o0 + j * pitch;
            st(oE0, o, e0);
            if constexpr (POL == TE) st(oE1, o, d[1][j]);
            st(oB0, o, bo0);
            if constexpr (POL == TM) st(oB1, o, bo1);
        }
    }
}

// SET: the TE or the TM set, or BOTH (blockIdx.y picks it)
constexpr int BOTH = 2;

template <int SET, int M, int P, bool HJ>
__global__ void __launch_bounds__(32 * NW, 2) k_tile2d(Fused2dArgs<float> a, Geo g, Coef2 c, Tile2dGeo t) {
    extern __shared__ __align__(16) float2 tsm[];
    const int zero = dependency_wait();
    const int x0 = (int)(blockIdx.x % t.ntx) * t.tw, y0 = (int)(blockIdx.x / t.ntx) * t.th;
    const int th = min(t.th, g.ny - y0);
    constexpr int HC = TileHalo<M, P, HJ>::HC;
    const bool seam = (g.nx & 1) && (x0 < HC || x0 - HC + 64 > g.nx);
    const bool tm = SET == TM || (SET == BOTH && blockIdx.y == 1);
    if (SET != TM && !tm) {
        if (!seam) tile_step<TE, M, P, HJ, false>(a, g, c, t.tw, th, x0, y0, zero, tsm);
        else tile_step<TE, M, P, HJ, true>(a, g, c, t.tw, th, x0, y0, zero, tsm);
    }
    if (SET != TE && tm) {
        if (!seam) tile_step<TM, M, P, HJ, false>(a, g, c, t.tw, th, x0, y0, zero, tsm);
        else tile_step<TM, M, P, HJ, true>(a, g, c, t.tw, th, x0, y0, zero, tsm);
    }
}

}  // namespace

template <int SET, int M, int P, bool HJ>
void launch_tile2d(const Geo &g, const Coef2 &c, const Fused2dArgs<float> &a, cudaStream_t s) {
    constexpr size_t smem = (size_t)((SET == TM ? 1 : 2) * R * NW + 6 * NW) * 32 * sizeof(float2);
    auto k = k_tile2d<SET, M, P, HJ>;
    static const bool attr =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess;
    (void)attr;  // a failure shows up in the launch
    // what the halo leaves of 64 columns and R NW rows
    using H = TileHalo<M, P, HJ>;
    constexpr int TWX = (63 - H::HC - M - H::PX) / 2 * 2, THX = R * NW - 2 * H::HY - 1;
    static_assert(TWX >= 2 && THX >= 1 && R >= P, "halo larger than the tile");
    const Tile2dGeo t = cover(g.nx, g.ny, TWX, THX);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(t.ntx * t.nty, SET == BOTH ? 2 : 1);
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

#define FMX_TILE_S(SET, M, P, HJ) \
    template void launch_tile2d<SET, M, P, HJ>(const Geo &, const Coef2 &, const Fused2dArgs<float> &, cudaStream_t);
#define FMX_TILE_MP(M, P, HJ) FMX_TILE_S(TE, M, P, HJ) FMX_TILE_S(TM, M, P, HJ) FMX_TILE_S(BOTH, M, P, HJ)
#define FMX_TILE_M(M) \
    FMX_TILE_MP(M, 0, false) FMX_TILE_MP(M, 0, true) FMX_TILE_MP(M, 1, true) FMX_TILE_MP(M, 2, true) FMX_TILE_MP(M, 3, true)
FMX_TILE_M(0)
FMX_TILE_M(1)
FMX_TILE_M(2)
FMX_TILE_M(3)
FMX_TILE_M(4)

// Sizes: us per step against the row pipeline (m = 4, p = 3 / vacuum, back to back
// steps): 64^2 5.2 / 4.2 against 16.8 / 12.4, 512^2 8.8 / 6.7 against 22.9 / 18.5,
// 1024^2 18.2 / 13.0 against 30.8 / 22.6, 1400^2 37.8 / 25.7 against 47.2 / 32.6,
// 2048^2 78.6 / 58.3 against 82.2 / 59.1, 4096^2 315 / 233 against 234 / 165.  The
// tiles recompute 1.75 cells per cell (p = 3), the row pipeline 1.22 on a grid
// large enough for long segments whose rows it can prefetch from HBM, so the line
// lies where a step's 60 bytes per cell (48 without a current, where the two meet
// a little earlier) reach twice the L2.
// Wide grids of few rows: a tile holds 64 rows of warps however few it needs, and
// with several waves of such tiles the row pipeline is ahead while one segment of
// it takes the whole height (about its 3m + 2p + 8 warm-up rows).  Tiles against
// rows, n_x = 50000, m = 4, p = 3: 8 rows 26.4 / 21.8, 24 rows 34.0 / 29.9, 28 rows
// 37.0 / 40.7; vacuum 20 rows 22.6 / 20.5, 28 rows 26.8 / 25.8; m = 1, p = 0: 8 rows
// 14.5 / 9.0, 20 rows 15.9 / 14.5, 24 rows 16.4 / 18.2; n_x = 400000, m = 4, p = 3, 8 rows
// 242 / 121; n_x = 20001, 8 rows 13.7 / 21.8.  So from `wide` tiles per SM on; 4, and
// 8 for the adjoint (us per step of both sets and jbar, m = 4, p = 3, 8 rows: n_x =
// 50000 78.7 / 84.4, 100000 96.8 / 92.7, 400000 252 / 208).
int fused2d_tiles(const Geo &g, int m, int passes, int wide) {
    static const long long l2 = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev) == cudaSuccess && v > 0 ? (long long)v : 1LL << 27;
    }();
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 1;
    }();
    const double cells = (double)g.nx * (double)g.ny;
    if (60.0 * cells > 2.0 * (double)l2) return 0;
    const int warm = 3 * m + 2 * passes + 8;
    if (g.nx >= 48LL * wide * sms && g.ny <= (warm > 20 ? warm : 20)) return 0;
    return cells <= kTileOneLaunchCells ? 1 : 2;
}

}  // namespace fmx
