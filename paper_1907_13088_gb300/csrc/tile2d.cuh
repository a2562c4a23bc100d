// Register tiles of the FP32 2D step (tile2d.cu) and of its adjoint
// (adj_tile2d.cu): a warp's 64 columns x R rows and what both directions do on
// them.  Internal.
#pragma once

#include <cuda_runtime.h>

#include "pair2.cuh"

namespace fmx {
namespace tile2d {

using namespace pair2;

constexpr unsigned FULL = 0xffffffffu;
constexpr int R = 8, NW = 8;  // rows per warp, warps per CTA

__device__ __forceinline__ float up1(float v) { return __shfl_up_sync(FULL, v, 1); }
__device__ __forceinline__ float dn1(float v) { return __shfl_down_sync(FULL, v, 1); }
__device__ __forceinline__ f2 sub(f2 a, f2 b) { return fma(b, m1(), a); }

// The kernels are launched while the one before them in the stream still runs
// (programmatic dependent launch): nothing is read or written before that one is
// done, and the next may come up from here on.  Returns a zero that the compiler
// does not know, to go into the load addresses: ld and ld2 may move freely, but
// not ahead of the wait.  (Not __ldg: the kernel before may write these arrays
// while this one is already resident, which the read-only path does not allow and
// the wait does not order.  Plain loads cannot move past the shared-memory stores
// and spill 12 to 72 bytes.)  What they read must not be written by the kernel.
__device__ __forceinline__ int dependency_wait() {
    int zero;
    asm volatile("griddepcontrol.wait;\n\tmov.s32 %0, 0;" : "=r"(zero)::"memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    return zero;
}
__device__ __forceinline__ float ld(const float *p) {
    float v;
    asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ f2 ld2(const float *p) {
    f2 v;
    asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

// columns 2t-1 and 2t+2 beside the own pair: f[i-1] + f[i+1]
__device__ __forceinline__ f2 xsum(f2 v, float l, float r) { return mk(l + v.y, v.x + r); }

// unnormalised (2P+1)-tap binomial along x of a warp's columns, the taps
// folded in the order of binom_taps
template <int P>
__device__ __forceinline__ f2 binom_x(f2 v) {
    float col[2 * P + 2];  // columns 2t-P .. 2t+1+P
#pragma unroll
    for (int i = 0; i < 2 * P + 2; ++i) {
        const int off = i - P, pr = off >= 0 ? off / 2 : -((1 - off) / 2);  // pair t + pr
        const float w = (off - 2 * pr) ? v.y : v.x;
        col[i] = pr == 0 ? w : (pr < 0 ? __shfl_up_sync(FULL, w, -pr) : __shfl_down_sync(FULL, w, pr));
    }
    f2 acc = mk(col[0] + col[2 * P], col[1] + col[2 * P + 1]);
#pragma unroll
    for (int k = 1; k < P; ++k) acc = fma(cst(binom2(P, k)), mk(col[k] + col[2 * P - k], col[k + 1] + col[2 * P + 1 - k]), acc);
    return fma(cst(binom2(P, P)), v, acc);
}

struct Tile2dGeo {
    int tw, th, ntx, nty;  // columns and rows a tile writes, tiles along x and y
};

// tiles of equal size that cover n_x x n_y, none larger than twx x thx (twx even)
inline Tile2dGeo cover(int nx, int ny, int twx, int thx) {
    Tile2dGeo t;
    t.ntx = (nx + twx - 1) / twx;
    t.tw = ((nx + t.ntx - 1) / t.ntx + 1) / 2 * 2;
    t.ntx = (nx + t.tw - 1) / t.tw;
    t.nty = (ny + thx - 1) / thx;
    t.th = (ny + t.nty - 1) / t.nty;
    t.nty = (ny + t.th - 1) / t.th;
    return t;
}

// The sweeps of Algorithm 1 on the tile: d holds dE' of the own rows and
// receives dE_(M).  row(q, r): the CTA's shared-memory rows (own rows keep dE');
// pub(buf, slot, warp): border rows, two sets; wb, wa: the warps below and above;
// need(s): the warp's rows are needed after sweep s.  One barrier per sweep.
template <int POL, int M, typename Row, typename Pub, typename Need>
__device__ __forceinline__ void sweeps(f2 (&d)[POL == TE ? 2 : 1][R], const Coef2 &c, int wp, int wb, int wa,
                                       const Row &row, const Pub &pub, const Need &need) {
    constexpr int NC = POL == TE ? 2 : 1;
    auto publish = [&](int buf) {
        pub(buf, 0, wp) = d[0][R - 1];
        pub(buf, 1, wp) = d[0][0];
        if constexpr (POL == TE) pub(buf, 2, wp) = d[1][R - 1];
    };
#pragma unroll
    for (int s = 1; s <= M; ++s) {
        const int buf = (s - 1) & 1;
        publish(buf);
        __syncthreads();
        if (s == 1) {
            // the raw current is consumed: its rows now keep dE' (own rows only)
#pragma unroll
            for (int q = 0; q < NC; ++q)
#pragma unroll
                for (int j = 0; j < R; ++j) row(q, wp * R + j) = d[q][j];
        }
        if (!need(s)) continue;
        if constexpr (POL == TE) {
            // h = Dbar_x Ex, gy = Dbar_y Ey
            auto dx = [&](f2 v) { return mk(v.x - up1(v.y), v.y - v.x); };
            f2 xp = pub(buf, 0, wb), yp = pub(buf, 2, wb), h = dx(d[0][0]);
            const f2 xa = pub(buf, 1, wa);
            float eyrp = dn1(yp.x);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const f2 x = d[0][j], y = d[1][j], xn = j < R - 1 ? d[0][j + 1] : xa;
                const f2 dp0 = s == 1 ? x : row(0, wp * R + j), dp1 = s == 1 ? y : row(1, wp * R + j);
                const float eyl = up1(y.y), eyr = dn1(y.x);
                const f2 gy = sub(y, yp), hn = dx(xn);
                f2 o0 = fma(c.ay, fma(x, m2(), add(xn, xp)), dp0);
                o0 = fma(c.bxy, mk(gy.y - gy.x, (eyr - eyrp) - gy.y), o0);
                f2 o1 = fma(c.ax, fma(y, m2(), xsum(y, eyl, eyr)), dp1);
                o1 = fma(c.bxy, sub(hn, h), o1);
                d[0][j] = o0;
                d[1][j] = o1;
                xp = x;
                yp = y;
                h = hn;
                eyrp = eyr;
            }
        } else {
            auto dxx = [&](f2 v) { return fma(v, m2(), xsum(v, up1(v.y), dn1(v.x))); };
            f2 zp = pub(buf, 0, wb), Dp = dxx(zp), D = dxx(d[0][0]);
            const f2 za = pub(buf, 1, wa);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                const f2 z = d[0][j], zn = j < R - 1 ? d[0][j + 1] : za;
                const f2 dp0 = s == 1 ? z : row(0, wp * R + j);
                const f2 Dn = dxx(zn);
                f2 o0 = fma(c.ax, D, dp0);
                o0 = fma(c.ay, fma(z, m2(), add(zn, zp)), o0);
                d[0][j] = fma(c.axy, fma(D, m2(), add(Dn, Dp)), o0);
                zp = z;
                Dp = D;
                D = Dn;
            }
        }
    }
}

}  // namespace tile2d
}  // namespace fmx
