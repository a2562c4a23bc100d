// Staged engine: one kernel per stage of the step, every intermediate in
// global memory.  General path: 1D/2D/3D, FP32/FP64, fixed or
// residual-controlled iteration, current or field filtering.  Each kernel
// is a plain one-thread-per-cell periodic stencil; the fused 2D engine
// (fused2d.cu) is the throughput path.
//
// Stencils (paper arXiv:1907.13088):
//   Dbar_a f: forward f[+1] - f[0] when f sits on an integer position along
//     a, backward f[0] - f[-1] when it sits half a cell off (Sec. 2);
//   alpha_a f = f + (1/6) Dbar_aa f (the (1/6, 2/3, 1/6) stencil);
//   source: Eqs. ampere_aux_x..z; A: Eqs. matrixA_1st..matrixA_last;
//   Faraday: Eqs. faraday_x..z.  Inactive axes (2D, 1D) drop every term
//   that differentiates along them and alpha becomes 1 (Secs. 2.2.2-2.2.3).
#include <cuda_runtime.h>

#include <type_traits>

#include "fmx_internal.h"
#include "stencil.cuh"

namespace fmx {
namespace {

constexpr int BX = 32, BY = 8;

__device__ __forceinline__ bool cell(const Geo &g, Pos &p, int64_t &idx) {
    p.i = blockIdx.x * BX + threadIdx.x;
    p.j = blockIdx.y * BY + threadIdx.y;
    p.k = blockIdx.z;
    idx = (int64_t)p.k * g.plane + (int64_t)p.j * g.pitch + p.i;
    return p.i < g.nx && p.j < g.ny;
}

__device__ __forceinline__ int64_t block_slot() {
    return (int64_t)blockIdx.x + (int64_t)gridDim.x * ((int64_t)blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
}

// FP64 block sum of v (all threads call), thread 0 writes out[block_slot()]
__device__ __forceinline__ void block_sum_to(double v, double *out) {
    __shared__ double red[BX * BY / 32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int t = threadIdx.y * BX + threadIdx.x;
    if ((t & 31) == 0) red[t >> 5] = v;
    __syncthreads();
    if (t == 0) {
        double s = 0.0;
        for (int w = 0; w < BX * BY / 32; ++w) s += red[w];
        out[block_slot()] = s;
    }
}

template <typename T>
__global__ void k_filter_pass(Geo g, const T *__restrict__ in, T *__restrict__ out, int axis) {
    Pos p;
    int64_t idx;
    if (!cell(g, p, idx)) return;
    Field<T, T> f{in, g};
    int dx, dy, dz;
    unit(axis, 1, dx, dy, dz);
    out[idx] = T(0.25) * f(p, -dx, -dy, -dz) + T(0.5) * f(p, 0, 0, 0) + T(0.25) * f(p, dx, dy, dz);
}

// Binomial filter of several components at once, P passes along every axis in
// two launches.  The P passes of one axis are its (2P+1)-tap binomial, and P = 1
// rounds as the single passes do.  2D: in place, tile by tile (below).  1D and 3D:
// the x (3D: x and y) taps from the fields into scratch, the last axis' taps back
// (1D: copied back).
struct FilterSet {
    const void *in[6];
    void *out[6];
};
template <int P>
__host__ __device__ constexpr double filter_w(int k) {
    double c = 1.0;
    for (int i = 0; i < k; ++i) c = c * (2 * P - i) / (i + 1);
    for (int i = 0; i < P; ++i) c /= 4.0;
    return c;
}
template <typename T, int P>
__device__ __forceinline__ T filter_taps(const T *v) {
    T s = T(filter_w<P>(0)) * v[0];
#pragma unroll
    for (int k = 1; k < 2 * P + 1; ++k) s += T(filter_w<P>(k)) * v[k];
    return s;
}

// 2D, in place: a CTA holds a tile of at most 64 x 64 cells in shared memory, with
// a halo of P cells that the launch before it saved in ring (a tile's cells are
// written by its own CTA only, once all of them are loaded).  So the filter takes
// the workspace's one spare component array and none of the caller's others.  A
// grid of one tile is its own halo: one launch, ring = nullptr.
// Each cell is read and written once, and the halos (P = 1: 6%).  FP32 is bound by
// issue (72%): 1536 x 1200, E and B, P = 1: 12 + 22 us launched cold, 27 warm (two passes
// through a second array 35 + 33, one launch per component, axis and pass 12 x 10).
// FP64 is bound by its 2 (2P + 1) operations per cell, which is why the x taps are
// evaluated once per row of the tile (9% more rows than cells at P = 3) and small
// grids are cut into smaller tiles, over more SMs (same grid, P = 2: 258 us with the
// x taps of a row evaluated by each group of rows, 239 now).
// ring_size is how much of it a tile of a component takes, ring_cell the cell of
// its element e: P rows below and above with their corners, then P columns left
// and right.
constexpr int FT = 64, FNT = 256;  // tile, threads
__host__ __device__ constexpr int ring_size(int P, int tw, int th) { return 2 * P * (tw + 2 * P) + 2 * P * th; }
template <int P>
__device__ __forceinline__ void ring_cell(int e, int tw, int th, int &col, int &row) {
    const int w = tw + 2 * P;
    if (e < 2 * P * w) {
        const int r = e / w;
        col = e % w - P;
        row = r < P ? r - P : th + r - P;
    } else {
        e -= 2 * P * w;
        const int k = e % (2 * P);
        col = k < P ? k - P : tw + k - P;
        row = e / (2 * P);
    }
}
struct FilterTiles {
    int tw, th, ntx, h;  // tile, tiles along x, ring elements per tile
};
template <typename T>
__device__ __forceinline__ T wrapped(const Geo &g, const T *in, int x, int y) {
    while (x < 0) x += g.nx;
    while (x >= g.nx) x -= g.nx;
    while (y < 0) y += g.ny;
    while (y >= g.ny) y -= g.ny;
    return in[(int64_t)y * g.pitch + x];
}
template <typename T, int P>
__global__ void __launch_bounds__(FNT) k_filter_halo(Geo g, const __grid_constant__ FilterSet f, FilterTiles t, T *ring) {
    const T *in = (const T *)f.in[blockIdx.y];
    const int x0 = (int)(blockIdx.x % t.ntx) * t.tw, y0 = (int)(blockIdx.x / t.ntx) * t.th;
    const int tw = min(t.tw, g.nx - x0), th = min(t.th, g.ny - y0);
    T *out = ring + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * t.h;
    for (int e = threadIdx.x; e < ring_size(P, tw, th); e += blockDim.x) {
        int col, row;
        ring_cell<P>(e, tw, th, col, row);
        out[e] = wrapped(g, in, x0 + col, y0 + row);
    }
}
template <typename T, int P>
__global__ void __launch_bounds__(FNT) k_filter_tile(Geo g, const __grid_constant__ FilterSet f, FilterTiles t, const T *ring) {
    constexpr int W = FT + 2 * P;  // shared row
    __shared__ T sm[W * W];
    const int x0 = (int)(blockIdx.x % t.ntx) * t.tw, y0 = (int)(blockIdx.x / t.ntx) * t.th;
    const int tw = min(t.tw, g.nx - x0), th = min(t.th, g.ny - y0);
    // columns of the tile over 32 or 64 threads, its rows over groups of them
    const int cols = t.tw <= 32 ? 32 : 64, groups = FNT / cols, col = threadIdx.x % cols, grp = threadIdx.x / cols;
    T *own = (T *)f.out[blockIdx.y] + (int64_t)y0 * g.pitch + x0 + col;
    const T *halo = ring + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * t.h;
#pragma unroll
    for (int i = 0; i < FT / 4; ++i) {
        const int r = i * groups + grp;
        if (r < th && col < tw) sm[(r + P) * W + col + P] = own[r * g.pitch];
    }
    for (int e = threadIdx.x; e < ring_size(P, tw, th); e += FNT) {
        int c, r;
        ring_cell<P>(e, tw, th, c, r);
        sm[(r + P) * W + c + P] = ring ? halo[e] : wrapped(g, (const T *)f.in[blockIdx.y], c, r);
    }
    __syncthreads();
    // x taps, a row per warp, in place
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < th + 2 * P; r += FNT / 32) {
        T *row = sm + r * W + lane;
        const T a = lane < tw ? filter_taps<T, P>(row) : T(0), b = lane + 32 < tw ? filter_taps<T, P>(row + 32) : T(0);
        __syncwarp();
        if (lane < tw) row[P] = a;
        if (lane + 32 < tw) row[32 + P] = b;
    }
    __syncthreads();
    // y taps, up to 16 rows of a column per thread
    const int run = (th + groups - 1) / groups, r0 = grp * run, n = min(run, th - r0) + 2 * P;
    if (col >= tw || r0 >= th) return;
    const T *in = sm + r0 * W + col + P;
    T *o = own + r0 * g.pitch;
    T w[2 * P + 1];
#pragma unroll
    for (int r = 0; r < FT / 4 + 2 * P; ++r) {
        if (r >= n) break;
#pragma unroll
        for (int k = 0; k < 2 * P; ++k) w[k] = w[k + 1];
        w[2 * P] = in[r * W];
        if (r >= 2 * P) o[(r - 2 * P) * g.pitch] = filter_taps<T, P>(w);
    }
}

// As many of the n components at a time as the spare array (g.plane elements) has
// room for; 0 where it has room for none.  Tiles shrink from 64 x 64 to 16 x 16 while
// there are fewer than two per SM and the halos of all n components still fit.
template <typename T, int P>
int filter_tiles(const Geo &g, int n, T *const f[], T *spare, cudaStream_t s) {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 1;
    }();
    FilterTiles t{};
    int64_t tiles = 0, fit = 0;
    FilterSet a{};
    if (g.nx <= FT && g.ny <= FT) {
        for (int q = 0; q < n; ++q) a.in[q] = a.out[q] = f[q];
        t = FilterTiles{g.nx, g.ny, 1, 0};
        k_filter_tile<T, P><<<dim3(1, n), FNT, 0, s>>>(g, a, t, nullptr);
        return 1;
    }
    for (int lx = FT, ly = FT; lx >= 16 && ly >= 16;) {
        const auto even = [](int len, int lim) { return (len + (len + lim - 1) / lim - 1) / ((len + lim - 1) / lim); };
        FilterTiles c;
        c.tw = even(g.nx, lx);
        c.th = even(g.ny, ly);
        c.ntx = (g.nx + c.tw - 1) / c.tw;
        c.h = ring_size(P, c.tw, c.th);
        const int64_t ct = (int64_t)c.ntx * ((g.ny + c.th - 1) / c.th), cf = g.plane / (ct * c.h);
        if (tiles > 0 && cf < n) break;
        t = c;
        tiles = ct;
        fit = cf;
        if (tiles * n >= 2 * sms || fit < n) break;
        if (c.th >= c.tw) ly = (c.th + 1) / 2;
        else lx = (c.tw + 1) / 2;
    }
    if (fit < 1) return 0;
    const int parts = (int)((n + fit - 1) / fit), per = (n + parts - 1) / parts;
    int launches = 0;
    for (int q0 = 0; q0 < n; q0 += per) {
        const int m = n - q0 < per ? n - q0 : per;
        for (int q = 0; q < m; ++q) a.in[q] = a.out[q] = f[q0 + q];
        const dim3 grid((unsigned)tiles, m);
        k_filter_halo<T, P><<<grid, FNT, 0, s>>>(g, a, t, spare);
        k_filter_tile<T, P><<<grid, FNT, 0, s>>>(g, a, t, spare);
        launches += 2;
    }
    return launches;
}

constexpr int FR = 16;  // rows per thread
template <typename T, int P, bool XY>
__global__ void __launch_bounds__(BX *BY) k_filter_in_plane(Geo g, const __grid_constant__ FilterSet f, int nbx, int nby) {
    const T *__restrict__ in = (const T *)f.in[blockIdx.y];
    T *__restrict__ out = (T *)f.out[blockIdx.y];
    const unsigned bxy = blockIdx.x / nbx;
    const int x = (int)(blockIdx.x % nbx) * BX + threadIdx.x;
    const int y0 = ((int)(bxy % nby) * blockDim.y + threadIdx.y) * FR;
    const int64_t z = (int64_t)(bxy / nby) * g.plane;
    if (x >= g.nx || y0 >= g.ny) return;
    constexpr int H = XY ? P : 0;
    int xo[2 * P + 1];
#pragma unroll
    for (int k = 0; k < 2 * P + 1; ++k) {
        int v = x + k - P;
        while (v < 0) v += g.nx;
        while (v >= g.nx) v -= g.nx;
        xo[k] = v;
    }
    // rows y0 - H .. y0 + FR - 1 + H in turn; XY: the x results of the last
    // 2P + 1 rows are kept for the y taps
    int yc = y0 - H;
    while (yc < 0) yc += g.ny;
    const T *row = in + z + (int64_t)yc * g.pitch;
    T *o = out + z + (int64_t)y0 * g.pitch + x;
    const int n = min(FR, g.ny - y0) + 2 * H;
    T w[2 * H + 1];
#pragma unroll
    for (int r = 0; r < FR + 2 * H; ++r) {
        if (r >= n) break;
        T v[2 * P + 1];
#pragma unroll
        for (int k = 0; k < 2 * P + 1; ++k) v[k] = row[xo[k]];
#pragma unroll
        for (int k = 0; k < 2 * H; ++k) w[k] = w[k + 1];
        w[2 * H] = filter_taps<T, P>(v);
        if (r >= 2 * H) {
            *o = XY ? filter_taps<T, XY ? P : 0>(w) : w[0];
            o += g.pitch;
        }
        row += g.pitch;
        if (++yc == g.ny) {
            yc = 0;
            row -= g.plane;
        }
    }
}

// along an axis of n elements `stride` apart; the `others` remaining lines are
// `ostride` apart.  P = 0 copies.
constexpr int FS = 16;  // elements per thread
template <typename T, int P>
__global__ void __launch_bounds__(BX *BY) k_filter_last(Geo g, const __grid_constant__ FilterSet f, int n, int64_t stride,
                                                        int64_t ostride, int nbx, int nseg) {
    const T *__restrict__ in = (const T *)f.in[blockIdx.y];
    T *__restrict__ out = (T *)f.out[blockIdx.y];
    const unsigned rest = blockIdx.x / nbx;
    const int x = (int)(blockIdx.x % nbx) * BX + threadIdx.x;
    const int j0 = ((int)(rest % nseg) * blockDim.y + threadIdx.y) * FS;
    if (x >= g.nx || j0 >= n) return;
    const int64_t o = (int64_t)(rest / nseg) * ostride + x;
    int j = j0 - P;
    while (j < 0) j += n;
    const T *p = in + o + j * stride;
    T *q = out + o + j0 * stride;
    const int len = min(FS, n - j0) + 2 * P;
    T w[2 * P + 1];
#pragma unroll
    for (int r = 0; r < FS + 2 * P; ++r) {
        if (r >= len) break;
#pragma unroll
        for (int k = 0; k < 2 * P; ++k) w[k] = w[k + 1];
        w[2 * P] = *p;
        if (r >= 2 * P) {
            *q = P ? filter_taps<T, P>(w) : w[0];
            q += stride;
        }
        p += stride;
        if (++j == n) {
            j = 0;
            p -= n * stride;
        }
    }
}

template <typename T, int P>
void filter_two(const Geo &g, int dims, int n, T *const f[], T *const scratch[], cudaStream_t s) {
    FilterSet a{}, b{};
    for (int q = 0; q < n; ++q) {
        a.in[q] = b.out[q] = f[q];
        a.out[q] = scratch[q];
        b.in[q] = scratch[q];
    }
    // blocks of 32 columns and as many groups of rows as the axis has (a power of two,
    // at most 8): no warp without work on short axes (1D, 100000 cells FP32, P = 1, E
    // and B: 108 us with blocks of 32 x 8 whatever the axis)
    const auto block = [](int len, int run) {
        int by = 1;
        while (by < BY && by * run < len) by *= 2;
        return dim3(BX, by);
    };
    const dim3 ka = block(g.ny, FR);
    const int nbx = (g.nx + BX - 1) / BX, nby = (g.ny + ka.y * FR - 1) / (ka.y * FR);
    const dim3 ga((unsigned)((int64_t)nbx * nby * g.nz), n);
    if (dims == 3) k_filter_in_plane<T, P, true><<<ga, ka, 0, s>>>(g, a, nbx, nby);
    else k_filter_in_plane<T, P, false><<<ga, ka, 0, s>>>(g, a, nbx, nby);
    const int len = dims == 3 ? g.nz : g.ny, others = dims == 3 ? g.ny : 1;
    const dim3 kb = block(len, FS);
    const int nseg = (len + kb.y * FS - 1) / (kb.y * FS);
    const dim3 gb((unsigned)((int64_t)nbx * nseg * others), n);
    if (dims == 3) k_filter_last<T, P><<<gb, kb, 0, s>>>(g, b, len, g.plane, g.pitch, nbx, nseg);
    else k_filter_last<T, 0><<<gb, kb, 0, s>>>(g, b, len, g.pitch, g.pitch, nbx, nseg);
}

template <typename T, int DIM>
__global__ void k_source(Geo g, Coef<T> c, StagedPtrs<T> P, const T *jx, const T *jy, const T *jz, int norm) {
    Pos p;
    int64_t idx;
    bool in = cell(g, p, idx);
    double s = 0.0;
    if (in) {
        Field<T, T> b[3] = {{P.B[0], g}, {P.B[1], g}, {P.B[2], g}};
        T ex = curl_alpha_b<T, DIM, 0>(b, p, c);
        T ey = curl_alpha_b<T, DIM, 1>(b, p, c);
        T ez = curl_alpha_b<T, DIM, 2>(b, p, c);
        if (jx) ex -= c.q * jx[idx];
        if (jy) ey -= c.q * jy[idx];
        if (jz) ez -= c.q * jz[idx];
        P.dEp[0][idx] = ex;
        P.dEp[1][idx] = ey;
        P.dEp[2][idx] = ez;
        s = (double)ex * ex + (double)ey * ey + (double)ez * ez;
    }
    if (norm) block_sum_to(s, P.partials);
}

template <typename T, int DIM>
__device__ __forceinline__ double sweep_cell(const Geo &g, const Coef<T> &c, const T *const dEp[3],
                                             const T *const in[3], T *const out[3], Pos p, int64_t idx) {
    Field<T, T> f[3] = {{in[0], g}, {in[1], g}, {in[2], g}};
    T nx_ = dEp[0][idx] + apply_a<T, DIM, 0>(f, p, c);
    T ny_ = dEp[1][idx] + apply_a<T, DIM, 1>(f, p, c);
    T nz_ = dEp[2][idx] + apply_a<T, DIM, 2>(f, p, c);
    T ox = in[0][idx], oy = in[1][idx], oz = in[2][idx];
    out[0][idx] = nx_;
    out[1][idx] = ny_;
    out[2][idx] = nz_;
    T dx = nx_ - ox, dy = ny_ - oy, dz = nz_ - oz;
    return (double)dx * dx + (double)dy * dy + (double)dz * dz;
}

template <typename T, int DIM>
__global__ void k_sweep(Geo g, Coef<T> c, const T *p0, const T *p1, const T *p2, const T *i0, const T *i1,
                        const T *i2, T *o0, T *o1, T *o2, double *partials) {
    Pos p;
    int64_t idx;
    bool inb = cell(g, p, idx);
    double s = 0.0;
    const T *dEp[3] = {p0, p1, p2};
    const T *in[3] = {i0, i1, i2};
    T *out[3] = {o0, o1, o2};
    if (inb) s = sweep_cell<T, DIM>(g, c, dEp, in, out, p, idx);
    if (partials) block_sum_to(s, partials);
}

// Residual mode: the sweep index lives on the device (DevStatus.count);
// a stopped solve turns the remaining launches of a chunk into no-ops.
template <typename T, int DIM>
__global__ void k_resid_sweep(Geo g, Coef<T> c, StagedPtrs<T> P) {
    if (P.st->done) return;
    const int s = P.st->count;
    Pos p;
    int64_t idx;
    bool inb = cell(g, p, idx);
    const T *in[3];
    T *out[3];
    for (int q = 0; q < 3; ++q) {
        in[q] = s == 0 ? P.dEp[q] : ((s & 1) ? P.dEa[q] : P.dEb[q]);
        out[q] = ((s + 1) & 1) ? P.dEa[q] : P.dEb[q];
    }
    const T *dEp[3] = {P.dEp[0], P.dEp[1], P.dEp[2]};
    double v = 0.0;
    if (inb) v = sweep_cell<T, DIM>(g, c, dEp, in, out, p, idx);
    block_sum_to(v, P.partials);
}

// Chebyshev semi-iteration (textbook three-term recurrence) for
// (1 - A) x = dE', x_0 = dE': sweep s computes r = dE' - x_s + A x_s,
// d = c1 d + c2 r, x_{s+1} = x_s + d, with c1 = 0, c2 = 1/theta for s = 0 and
// rho_s = 1 / (2 sig - rho_{s-1}), c1 = rho_s rho_{s-1}, c2 = 2 rho_s / delta
// after (rho_0 = 1 / sig, kept in DevStatus.cheb_rho by the update kernel).
template <typename T, int DIM>
__global__ void k_cheb_sweep(Geo g, Coef<T> c, StagedPtrs<T> P, ChebParams cp) {
    if (P.st->done) return;
    const int s = P.st->count;
    double c1 = 0.0, c2 = 1.0 / cp.theta;
    if (s > 0) {
        const double rp = P.st->cheb_rho, rn = 1.0 / (2.0 * cp.sig - rp);
        c1 = rn * rp;
        c2 = 2.0 * rn / cp.delta;
    }
    Pos p;
    int64_t idx;
    bool inb = cell(g, p, idx);
    double v = 0.0;
    if (inb) {
        const T *in[3];
        T *out[3];
        for (int q = 0; q < 3; ++q) {
            in[q] = s == 0 ? P.dEp[q] : ((s & 1) ? P.dEa[q] : P.dEb[q]);
            out[q] = ((s + 1) & 1) ? P.dEa[q] : P.dEb[q];
        }
        Field<T, T> f[3] = {{in[0], g}, {in[1], g}, {in[2], g}};
        const T ax[3] = {apply_a<T, DIM, 0>(f, p, c), apply_a<T, DIM, 1>(f, p, c), apply_a<T, DIM, 2>(f, p, c)};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const T x = in[q][idx];
            const T r = P.dEp[q][idx] - x + ax[q];
            const T d = (s == 0 ? T(0) : T(c1) * P.jf[q][idx]) + T(c2) * r;
            P.jf[q][idx] = d;
            out[q][idx] = x + d;
            v += (double)d * (double)d;
        }
    }
    block_sum_to(v, P.partials);
}

__device__ __forceinline__ double reduce_partials(const double *partials, int64_t n) {
    __shared__ double red[32];
    double s = 0.0;
    for (int64_t q = threadIdx.x; q < n; q += blockDim.x) s += partials[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

__global__ void k_resid_init(const double *partials, int64_t n, DevStatus *st) {
    double t = reduce_partials(partials, n);
    if (threadIdx.x == 0) {
        st->nrm2 = t;
        st->r2 = 0.0;
        st->count = 0;
        st->done = t == 0.0 ? 1 : 0;
        st->noconv = 0;
    }
}

__global__ void k_resid_update(const double *partials, int64_t n, DevStatus *st, double tol2, int m_max) {
    if (st->done) return;
    double t = reduce_partials(partials, n);
    if (threadIdx.x == 0) {
        st->r2 = t;
        st->count += 1;
        if (t <= tol2 * st->nrm2) {
            st->done = 1;
        } else if (st->count >= m_max) {
            st->done = 1;
            st->noconv = 1;
        }
    }
}

__global__ void k_cheb_update(const double *partials, int64_t n, DevStatus *st, ChebParams cp, int resid, double tol2,
                              int m_max) {
    if (st->done) return;
    double t = reduce_partials(partials, n);
    if (threadIdx.x == 0) {
        const int s = st->count;
        st->cheb_rho = s == 0 ? 1.0 / cp.sig : 1.0 / (2.0 * cp.sig - st->cheb_rho);
        st->r2 = t;
        st->count = s + 1;
        if (resid) {
            if (t <= tol2 * st->nrm2) {
                st->done = 1;
            } else if (st->count >= m_max) {
                st->done = 1;
                st->noconv = 1;
            }
        }
    }
}

template <typename T>
__global__ void k_update_e(Geo g, T *e0, T *e1, T *e2, const T *d0, const T *d1, const T *d2_) {
    Pos p;
    int64_t idx;
    if (!cell(g, p, idx)) return;
    e0[idx] += d0[idx];
    e1[idx] += d1[idx];
    e2[idx] += d2_[idx];
}

template <typename T>
__global__ void k_update_e_resid(Geo g, StagedPtrs<T> P) {
    Pos p;
    int64_t idx;
    if (!cell(g, p, idx)) return;
    const int s = P.st->count;
    for (int q = 0; q < 3; ++q) {
        const T *d = s == 0 ? P.dEp[q] : ((s & 1) ? P.dEa[q] : P.dEb[q]);
        P.E[q][idx] += d[idx];
    }
}

template <typename T, int DIM>
__global__ void k_faraday(Geo g, Coef<T> c, const T *e0, const T *e1, const T *e2, T *b0, T *b1, T *b2) {
    Pos p;
    int64_t idx;
    if (!cell(g, p, idx)) return;
    Field<T, T> e[3] = {{e0, g}, {e1, g}, {e2, g}};
    b0[idx] -= curl_e<T, DIM, 0>(e, p, c);
    b1[idx] -= curl_e<T, DIM, 1>(e, p, c);
    b2[idx] -= curl_e<T, DIM, 2>(e, p, c);
}

inline dim3 grid_of(const Geo &g) { return dim3((g.nx + BX - 1) / BX, (g.ny + BY - 1) / BY, g.nz); }

}  // namespace

int64_t staged_partial_slots(const Geo &g) {
    dim3 gr = grid_of(g);
    return (int64_t)gr.x * gr.y * gr.z;
}

template <typename T>
int launch_filter_pass(const Geo &g, int dims, const T *in, T *out, int axis, cudaStream_t s) {
    (void)dims;
    k_filter_pass<T><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, in, out, axis);
    return 1;
}

template <typename T>
int launch_filter_fields(const Geo &g, int dims, int passes, int n, T *const f[], T *const scratch[], T *spare,
                         cudaStream_t s) {
    // flattened launch grids of at most 2^31 - 1 blocks
    const double blocks = (double)((g.nx + BX - 1) / BX) * (double)g.ny * (double)g.nz;
    if (n < 1 || n > 6 || blocks > 2147483647.0) return 0;
    auto run = [&](auto p) {
        constexpr int P = decltype(p)::value;
        if (dims == 2) return filter_tiles<T, P>(g, n, f, spare, s);
        filter_two<T, P>(g, dims, n, f, scratch, s);
        return 2;
    };
    switch (passes) {
        case 1: return run(std::integral_constant<int, 1>());
        case 2: return run(std::integral_constant<int, 2>());
        case 3: return run(std::integral_constant<int, 3>());
    }
    return 0;
}

template <typename T>
int launch_staged_source(const Geo &g, int dims, const Coef<T> &c, const StagedPtrs<T> &p,
                         const T *const jsrc[3], cudaStream_t s, bool norm) {
    const T *jx = jsrc ? jsrc[0] : nullptr, *jy = jsrc ? jsrc[1] : nullptr, *jz = jsrc ? jsrc[2] : nullptr;
    if (dims == 3)
        k_source<T, 3><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p, jx, jy, jz, norm);
    else if (dims == 2)
        k_source<T, 2><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p, jx, jy, jz, norm);
    else
        k_source<T, 1><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p, jx, jy, jz, norm);
    return 1;
}

template <typename T>
int launch_staged_sweep(const Geo &g, int dims, const Coef<T> &c, const StagedPtrs<T> &p, const T *const in[3],
                        T *const out[3], bool resid, cudaStream_t s) {
    double *part = resid ? p.partials : nullptr;
    if (dims == 3)
        k_sweep<T, 3><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p.dEp[0], p.dEp[1], p.dEp[2], in[0], in[1], in[2],
                                                          out[0], out[1], out[2], part);
    else if (dims == 2)
        k_sweep<T, 2><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p.dEp[0], p.dEp[1], p.dEp[2], in[0], in[1], in[2],
                                                          out[0], out[1], out[2], part);
    else
        k_sweep<T, 1><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p.dEp[0], p.dEp[1], p.dEp[2], in[0], in[1], in[2],
                                                          out[0], out[1], out[2], part);
    return 1;
}

template <typename T>
int launch_resid_sweep(const Geo &g, int dims, const Coef<T> &c, const StagedPtrs<T> &p, cudaStream_t s) {
    if (dims == 3)
        k_resid_sweep<T, 3><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p);
    else if (dims == 2)
        k_resid_sweep<T, 2><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p);
    else
        k_resid_sweep<T, 1><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p);
    return 1;
}

int launch_resid_init(double *partials, int64_t nparts, DevStatus *st, cudaStream_t s) {
    k_resid_init<<<1, 1024, 0, s>>>(partials, nparts, st);
    return 1;
}

template <typename T>
int launch_cheb_sweep(const Geo &g, int dims, const Coef<T> &c, const StagedPtrs<T> &p, const ChebParams &cp,
                      cudaStream_t s) {
    if (dims == 3)
        k_cheb_sweep<T, 3><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p, cp);
    else if (dims == 2)
        k_cheb_sweep<T, 2><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p, cp);
    else
        k_cheb_sweep<T, 1><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, p, cp);
    return 1;
}

int launch_cheb_update(double *partials, int64_t nparts, DevStatus *st, const ChebParams &cp, bool resid,
                       double tol2, int m_max, cudaStream_t s) {
    k_cheb_update<<<1, 1024, 0, s>>>(partials, nparts, st, cp, resid ? 1 : 0, tol2, m_max);
    return 1;
}

int launch_resid_update(double *partials, int64_t nparts, DevStatus *st, double tol2, int m_max, cudaStream_t s) {
    k_resid_update<<<1, 1024, 0, s>>>(partials, nparts, st, tol2, m_max);
    return 1;
}

template <typename T>
int launch_update_e(const Geo &g, T *const E[3], const T *const dE[3], cudaStream_t s) {
    k_update_e<T><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, E[0], E[1], E[2], dE[0], dE[1], dE[2]);
    return 1;
}

template <typename T>
int launch_update_e_resid(const Geo &g, const StagedPtrs<T> &p, cudaStream_t s) {
    k_update_e_resid<T><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, p);
    return 1;
}

template <typename T>
int launch_faraday(const Geo &g, int dims, const Coef<T> &c, T *const E[3], T *const B[3], cudaStream_t s) {
    if (dims == 3)
        k_faraday<T, 3><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, E[0], E[1], E[2], B[0], B[1], B[2]);
    else if (dims == 2)
        k_faraday<T, 2><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, E[0], E[1], E[2], B[0], B[1], B[2]);
    else
        k_faraday<T, 1><<<grid_of(g), dim3(BX, BY), 0, s>>>(g, c, E[0], E[1], E[2], B[0], B[1], B[2]);
    return 1;
}

#define FMX_INST(T)                                                                                           \
    template int launch_filter_pass<T>(const Geo &, int, const T *, T *, int, cudaStream_t);                  \
    template int launch_filter_fields<T>(const Geo &, int, int, int, T *const[], T *const[], T *, cudaStream_t); \
    template int launch_staged_source<T>(const Geo &, int, const Coef<T> &, const StagedPtrs<T> &,            \
                                         const T *const[3], cudaStream_t, bool);                              \
    template int launch_staged_sweep<T>(const Geo &, int, const Coef<T> &, const StagedPtrs<T> &,             \
                                        const T *const[3], T *const[3], bool, cudaStream_t);                  \
    template int launch_resid_sweep<T>(const Geo &, int, const Coef<T> &, const StagedPtrs<T> &, cudaStream_t); \
    template int launch_cheb_sweep<T>(const Geo &, int, const Coef<T> &, const StagedPtrs<T> &, const ChebParams &, \
                                      cudaStream_t);                                                         \
    template int launch_update_e<T>(const Geo &, T *const[3], const T *const[3], cudaStream_t);               \
    template int launch_update_e_resid<T>(const Geo &, const StagedPtrs<T> &, cudaStream_t);                  \
    template int launch_faraday<T>(const Geo &, int, const Coef<T> &, T *const[3], T *const[3], cudaStream_t);
FMX_INST(float)
FMX_INST(double)
#undef FMX_INST

}  // namespace fmx
