// 3D z-marching kernels for the source (with the one-pass current filter), the
// sweeps of Algorithm 1 and the Faraday update.  A CTA owns a column tile and
// walks a segment of z planes; each input plane of the tile, with a one-cell
// halo in x and y, is copied once into a shared-memory ring by cp.async,
// planes ahead of the one being computed, so that no register holds data in
// flight; one __syncthreads per plane.  The A operator (Eqs.
// matrixA_1st..matrixA_last) and the averaged curl (Eqs. ampere_aux_x..z) are
// factored into in-plane stencils and 3-point combinations along z, so that an
// iteration reads one plane and carries the z-combinations in registers.  FP32
// grids with even n_x work on column pairs (one row per thread); FP64 grids and
// odd n_x on single columns, four rows per thread.
#include <cuda_runtime.h>

#include <type_traits>

#include "fmx_internal.h"
#include "pair2.cuh"

namespace fmx {
namespace {

constexpr int TY = 8, NTH = 32 * TY, RH = TY + 2;  // pair kernels: rows of the tile, threads, rows with halo

int sm_count() {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 1;
    }();
    return sms;
}

// planes a segment marches over.  The CTAs on one SM share its arithmetic, so a
// launch takes about the CTAs of the fullest SM times the planes each marches
// (two more than it writes), and c of them resident at a time leave their
// latencies open, which a factor 1 + lat/c stands for (0.5; 0.6 for the CTAs of
// two warps, or 64^3 FP64 would leave one of them on an SM: 450 us a step, 300 so); the segment height
// with the least product, 1 to 64 planes, is taken (128 x 128 x 96 FP64 sweep, CTAs
// of four warps: 24 planes, one CTA on each of 128 SMs, 270 us; 7 planes, 448
// CTAs, 250 us).  tiles: CTAs per segment; res: CTAs an SM holds.
int zseg_for(int nz, long long tiles, int res, double lat) {
    const int sms = sm_count();
    int best = 1;
    double least = 1e300;
    for (int z = nz < 64 ? nz : 64; z >= 1; --z) {
        const long long n = (tiles * ((nz + z - 1) / z) + sms - 1) / sms;  // CTAs of the fullest SM
        // rounds of res resident CTAs, then the rest
        const double load = (double)(n / res) * (res + lat) + (n % res ? (double)(n % res) + lat : 0.0);
        if (load * (z + 2) < least) {
            least = load * (z + 2);
            best = z;
        }
    }
    return best;
}

__device__ __forceinline__ int wrapm(int v, int n) { return ((v % n) + n) % n; }

// one element, global -> shared, asynchronous (cp.async, 4 or 8 bytes)
template <typename T>
__device__ __forceinline__ void cp_async_el(T *dst, const T *src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_pair(float *dst, const float *src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------------------
// One column per thread (FP64, odd n_x): a tile of 32 columns x 8 rows, 64
// threads, four rows of a column each (small CTAs, so that the segments share
// the FP64 arithmetic of all SMs evenly: 128 x 128 x 96 FP64 takes 1142 us a step
// against 1254 with 16 rows).  FP64 arithmetic runs at 1/64 of the
// FP32 rate on this part and bounds these kernels, so they are written for the
// fewest operations: the factored form (see plane_terms below), differences
// formed once and shared along the four rows of a thread, partial outputs
// carried as FMA accumulators.  A sweep takes 54 FP64 operations per cell
// against 135 for the 27-point stencils evaluated cell by cell, the filtered
// source 52 against about 150.  128 x 128 x 96 FP64, 16 rows: sweep 685 -> 242 us,
// source 627 -> 231 us (their operations take 213 and 189 us at the FMA rate that
// fmx_fma_peak measures); 201 x 150 x 99 FP32: sweep 53 -> 33 us, source 68 -> 38 us.
//
// The FP64 units sit one to a quarter of an SM, and a warp's rows follow one another
// on its own: with fewer warps than a quarter of them (grids of few cells, or of one
// or two planes) the rows are given to more warps, CR = 1 row per thread (one_row).
constexpr int CX = 32, CW = 2, CNT = 32 * CW;
constexpr int CPW = CX + 2;                                               // row of the tile with its halo
__host__ __device__ constexpr int cpl(int CR) { return CPW * (CR * CW + 2); }  // plane with its halo

// the copies of the tile's planes: plane z0 - 1 + i into ring slot i mod RS
template <typename T, int N, int RS, int CR>
struct ColPlanes {
    static constexpr int CPL = cpl(CR), CCP = (CPL + CNT - 1) / CNT;  // copies of a component plane per thread
    int off[CCP];  // in-plane offsets of the thread's elements
    int64_t base;  // element offset of the plane copied next, wrapped into [0, n_z)
    int slot;
    __device__ __forceinline__ void init(const Geo &g, int x0, int y0, int k0) {
#pragma unroll
        for (int q = 0; q < CCP; ++q) {
            const int e = threadIdx.x + q * CNT;
            off[q] = e < CPL ? wrapm(y0 - 1 + e / CPW, g.ny) * (int)g.pitch + wrapm(x0 - 1 + e % CPW, g.nx) : -1;
        }
        base = (int64_t)wrapm(k0, g.nz) * g.plane;
        slot = 0;
    }
    __device__ __forceinline__ void issue_next(T *ring, const T *const src[N], const Geo &g) {
        T *dst = ring + slot * N * CPL + threadIdx.x;
#pragma unroll
        for (int q = 0; q < CCP; ++q) {
            if (off[q] < 0) continue;
#pragma unroll
            for (int n = 0; n < N; ++n) cp_async_el(dst + n * CPL + q * CNT, src[n] + base + off[q]);
        }
        base += g.plane;
        if (base == (int64_t)g.nz * g.plane) base = 0;
        slot = slot + 1 == RS ? 0 : slot + 1;
    }
};

// the rows of a thread in turn; left: rows of the grid from its first on (the
// warp's, so the branch is uniform).  Rows past the grid are skipped, but not with
// a test per row where there are none: the rows' operations interleave.  FP64 only:
// FP32 arithmetic does not bind, and the second body costs 1% (201 x 150 x 99).
template <int CR, typename F>
__device__ __forceinline__ void each_row(int left, const F &row) {
    if (left >= CR) {
#pragma unroll
        for (int r = 0; r < CR; ++r) row(r);
    } else {
#pragma unroll
        for (int r = 0; r < CR - 1; ++r)
            if (r < left) row(r);
    }
}

template <typename T>
__device__ __forceinline__ T d2s(T a, T v, T b) { return (a + b) - T(2) * v; }  // a - 2 v + b

// out = dEp + A in, or with UPD E = E + dEp + A in (E in place)
constexpr int SWEEP1_RS = 4;
template <typename T, bool UPD, int CR>
__global__ void __launch_bounds__(CNT, 6) k3_sweep1(Geo g, Coef<T> c, const T *p0, const T *p1, const T *p2, const T *i0,
                                                 const T *i1, const T *i2, T *o0, T *o1, T *o2, int zseg) {
    constexpr int RS = SWEEP1_RS, CROWS = CR * CW, CPL = cpl(CR);
    extern __shared__ __align__(16) unsigned char m3raw[];
    T *ring = reinterpret_cast<T *>(m3raw);  // [RS][3][CPL]
    const T *in[3] = {i0, i1, i2};
    const T *dp[3] = {p0, p1, p2};
    T *out[3] = {o0, o1, o2};
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int x0 = blockIdx.x * CX, y0 = blockIdx.y * CROWS;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    const int np = z1 - z0 + 2;  // input planes z0-1 .. z1
    ColPlanes<T, 3, RS, CR> cp;
    cp.init(g, x0, y0, z0 - 1);
    auto issue = [&](int i) {
        if (i < np) cp.issue_next(ring, in, g);
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < RS - 1; ++i) issue(i);
    const int x = x0 + lane, y = y0 + wy * CR;
    const int rows = x < g.nx ? min(CR, g.ny - y) : 0;  // rows of the thread inside the grid
    int64_t cell = (int64_t)z0 * g.plane + (int64_t)y * g.pitch + x;
    const T bxy6 = c.bxy * c.c6, ax2 = c.ax - T(2) * c.axy;
    T xa[CR], xb[CR], ya[CR], yb[CR], za[CR];  // partial outputs o, o+1
#pragma unroll
    for (int r = 0; r < CR; ++r) xa[r] = xb[r] = ya[r] = yb[r] = za[r] = T(0);
    int slot = 0;
    for (int i = 0; i < np; ++i) {
        cp_async_wait<RS - 2>();
        __syncthreads();
        issue(i + RS - 1);
        const T *pl = ring + slot * 3 * CPL + (wy * CR + 1) * CPW + lane + 1;
        slot = slot + 1 == RS ? 0 : slot + 1;
        if (rows <= 0) continue;
        // dE' (and E^n) of the output plane this iteration completes
        T pd[3][CR], pe[UPD ? 3 : 1][CR];
#pragma unroll
        for (int r = 0; r < CR; ++r)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const bool ok = i >= 2 && r < rows;
                pd[q][r] = ok ? __ldg(dp[q] + cell + (int64_t)r * g.pitch) : T(0);
                if (UPD) pe[UPD ? q : 0][r] = ok ? out[q][cell + (int64_t)r * g.pitch] : T(0);
            }
        auto V = [&](int q, int dx, int r) -> T { return pl[q * CPL + r * CPW + dx]; };
        // what row r takes over from row r - 1
        T ex_m = V(0, 0, -1), ex_0 = V(0, 0, 0), b_m = ex_m - V(0, -1, -1), b_0 = ex_0 - V(0, -1, 0);
        T a_m, yp_m;
        {
            const T ey = V(1, 0, -1), eyr = V(1, 1, -1);
            a_m = eyr - ey;
            yp_m = ey + c.c6 * d2s(V(1, -1, -1), ey, eyr);
        }
        T ez_m = V(2, 0, -1), ez_0 = V(2, 0, 0), c_m, c_0, d_m, d_0, zx_0;
        {
            const T er = V(2, 1, -1), er0 = V(2, 1, 0);
            c_m = er - ez_m;
            c_0 = er0 - ez_0;
            d_m = d2s(V(2, -1, -1), ez_m, er);
            d_0 = d2s(V(2, -1, 0), ez_0, er0);
            zx_0 = ez_0 + c.c6 * d_0;
        }
        auto row = [&](int r) {
            // Ex: P = Dbar_yy Ex, X = Dbar_x (Ex + P/6), Gp = Dbar_x Dbar_y Ex
            const T ex_p = V(0, 0, r + 1), b_p = ex_p - V(0, -1, r + 1);
            const T P = d2s(ex_p, ex_0, ex_m), X = b_0 + c.c6 * d2s(b_p, b_0, b_m), Gp = b_p - b_0;
            // Ey: Q = Dbar_xx Ey, Y = Dbar_y (Ey + Q/6), G = Dbar_x Dbar_y Ey
            const T ey = V(1, 0, r), eyr = V(1, 1, r);
            const T Q = d2s(V(1, -1, r), ey, eyr), a_0 = eyr - ey, yp_0 = ey + c.c6 * Q;
            const T Y = yp_0 - yp_m, G = a_0 - a_m;
            // Ez: N = Dbar_x (Ez + Dbar_yy Ez / 6), Np = Dbar_y (Ez + Dbar_xx Ez / 6), T
            const T ez_p = V(2, 0, r + 1), er_p = V(2, 1, r + 1);
            const T c_p = er_p - ez_p, d_p = d2s(V(2, -1, r + 1), ez_p, er_p), zx_p = ez_p + c.c6 * d_p;
            const T N = c_0 + c.c6 * d2s(c_p, c_0, c_m), Np = zx_p - zx_0;
            const T t = c.axy * (d_p + d_m) + (c.ay * d2s(ez_p, ez_0, ez_m) + ax2 * d_0);
            const T zh = c.byz * Y + c.bzx * X;
            const T x1 = bxy6 * G + (c.ayz * P + c.az * ex_0), y1 = bxy6 * Gp + (c.azx * Q + c.az * ey);
            if (i >= 2 && r < rows) {
                // output plane z0 + i - 2 is complete
                const int64_t o = cell + (int64_t)r * g.pitch;
                T v[3] = {xa[r] + x1, ya[r] + y1, za[r] + zh};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    v[q] = pd[q][r] + v[q];
                    if (UPD) v[q] = pe[UPD ? q : 0][r] + v[q];
                    out[q][o] = v[q];
                }
            }
            xa[r] = T(-2) * x1 + (c.bzx * N + (c.bxy * G + (c.ay * P + xb[r])));
            xb[r] = x1 - c.bzx * N;
            ya[r] = T(-2) * y1 + (c.byz * Np + (c.bxy * Gp + (c.ax * Q + yb[r])));
            yb[r] = y1 - c.byz * Np;
            za[r] = t - zh;
            ex_m = ex_0, ex_0 = ex_p, b_m = b_0, b_0 = b_p;
            a_m = a_0, yp_m = yp_0;
            ez_m = ez_0, ez_0 = ez_p, c_m = c_0, c_0 = c_p, d_m = d_0, d_0 = d_p, zx_0 = zx_p;
        };
        each_row<CR>(sizeof(T) == 8 ? g.ny - y : CR, row);
        if (i >= 2) cell += g.plane;
    }
    cp_async_wait<0>();
}

// dE' = C_b (alpha B) - q F j, F = one (1/4, 1/2, 1/4) pass along each axis
// (PASSES = 1) or none (PASSES = 0); HJ: a current is bound.  The terms of
// curl_plane_terms below, per row.
constexpr int SOURCE1_RS = 3;
template <typename T, int PASSES, bool HJ, int CR>
__global__ void __launch_bounds__(CNT) k3_source1(Geo g, Coef<T> c, const T *b0, const T *b1, const T *b2, const T *j0,
                                                  const T *j1, const T *j2, T *o0, T *o1, T *o2, int zseg) {
    constexpr int RS = SOURCE1_RS, N = HJ ? 6 : 3, CROWS = CR * CW, CPL = cpl(CR);
    extern __shared__ __align__(16) unsigned char m3raw[];
    T *ring = reinterpret_cast<T *>(m3raw);  // [RS][N][CPL]
    const T *src[6] = {b0, b1, b2, j0, j1, j2};
    T *out[3] = {o0, o1, o2};
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int x0 = blockIdx.x * CX, y0 = blockIdx.y * CROWS;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    const int np = z1 - z0 + 2;  // input planes z0-1 .. z1
    ColPlanes<T, N, RS, CR> cp;
    cp.init(g, x0, y0, z0 - 1);
    auto issue = [&](int i) {
        if (i < np) cp.issue_next(ring, src, g);
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < RS - 1; ++i) issue(i);
    const int x = x0 + lane, y = y0 + wy * CR;
    const int rows = x < g.nx ? min(CR, g.ny - y) : 0;
    int64_t cell = (int64_t)z0 * g.plane + (int64_t)y * g.pitch + x;
    const T kyc6 = c.ky * c.c6, nkxc6 = -(c.kx * c.c6);
    // the current's factor, with PASSES = 1 over the integer weights' 64 (exact)
    const T qj = PASSES == 1 ? c.q * T(1.0 / 64.0) : c.q;
    T xa[CR], xb[CR], ya[CR], yb[CR], za[CR];
    T up[CR], wp[CR];  // U and W of the plane before
    T jz[HJ ? 3 : 1][2][CR];  // x-y binomial of planes j-2, j-1 (PASSES = 0: the current itself)
#pragma unroll
    for (int r = 0; r < CR; ++r) {
        xa[r] = xb[r] = ya[r] = yb[r] = za[r] = up[r] = wp[r] = T(0);
        if (HJ)
#pragma unroll
            for (int q = 0; q < 3; ++q) jz[HJ ? q : 0][0][r] = jz[HJ ? q : 0][1][r] = T(0);
    }
    int slot = 0;
    for (int i = 0; i < np; ++i) {
        cp_async_wait<RS - 2>();
        __syncthreads();
        issue(i + RS - 1);
        const T *pl = ring + slot * N * CPL + (wy * CR + 1) * CPW + lane + 1;
        slot = slot + 1 == RS ? 0 : slot + 1;
        if (rows <= 0) continue;
        auto V = [&](int q, int dx, int r) -> T { return pl[q * CPL + r * CPW + dx]; };
        auto wx = [&](int r) { return V(0, 0, r) + c.c6 * d2s(V(0, -1, r), V(0, 0, r), V(0, 1, r)); };  // alpha_x Bx
        auto jr = [&](int q, int r) { return (V(3 + q, -1, r) + V(3 + q, 1, r)) + T(2) * V(3 + q, 0, r); };
        T w_m = wx(-1), bz_m = V(2, 0, -1);
        T by_m = V(1, 0, -1), by_0 = V(1, 0, 0), u_m = by_m - V(1, -1, -1), u_0 = by_0 - V(1, -1, 0);
        T s_m[3], s_0[3];
        if constexpr (HJ && PASSES == 1) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                s_m[q] = jr(q, -1);
                s_0[q] = jr(q, 0);
            }
        }
        auto row = [&](int r) {
            const T by_p = V(1, 0, r + 1), u_p = by_p - V(1, -1, r + 1);
            const T U = by_0 + c.c6 * d2s(by_p, by_0, by_m), Ux = u_0 + c.c6 * d2s(u_p, u_0, u_m);
            const T W = wx(r), Wy = W - w_m;
            const T bz = V(2, 0, r), Vy = bz - bz_m, Vx = bz - V(2, -1, r);
            const T x1 = kyc6 * Vy, y1 = nkxc6 * Vx;
            T jn[3];
            if constexpr (HJ) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if constexpr (PASSES == 1) {
                        const T s_p = jr(q, r + 1);
                        jn[q] = (s_p + s_m[q]) + T(2) * s_0[q];
                        s_m[q] = s_0[q];
                        s_0[q] = s_p;
                    } else {
                        jn[q] = V(3 + q, 0, r);
                    }
                }
            }
            if (i >= 2 && r < rows) {
                const int64_t o = cell + (int64_t)r * g.pitch;
                T d[3] = {xa[r] + x1, ya[r] + y1, za[r]};
                if constexpr (HJ) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if constexpr (PASSES == 1) d[q] -= qj * ((jz[q][0][r] + jn[q]) + T(2) * jz[q][1][r]);
                        else d[q] -= qj * jz[q][1][r];
                    }
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) out[q][o] = d[q];
            }
            // the z-differences of U and W before their factor: on smooth fields
            // a difference is exact where the products' sum would round at |B|
            xa[r] = T(-2) * x1 + (c.ky * Vy + (xb[r] - c.kz * (U - up[r])));
            xb[r] = x1;
            ya[r] = T(-2) * y1 + (c.kz * (W - wp[r]) + (yb[r] - c.kx * Vx));
            yb[r] = y1;
            up[r] = U;
            wp[r] = W;
            za[r] = c.kx * Ux - c.ky * Wy;
            if constexpr (HJ) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    jz[q][0][r] = jz[q][1][r];
                    jz[q][1][r] = jn[q];
                }
            }
            w_m = W, bz_m = bz;
            by_m = by_0, by_0 = by_p, u_m = u_0, u_0 = u_p;
        };
        each_row<CR>(sizeof(T) == 8 ? g.ny - y : CR, row);
        if (i >= 2) cell += g.plane;
    }
    cp_async_wait<0>();
}

// B -= c dt curl E^{n+1} (Eqs. faraday_x..z), forward differences: a thread
// walks the planes of its column, E of the plane above carried over; the
// neighbours x+1 and y+1 come through L1.  Bound by memory; the
// one-thread-per-cell kernel spent its time on periodic 64-bit indices (201 x
// 150 x 99 FP32 26.5 -> 20.5 us, 128 x 128 x 96 FP64 49 -> 42).
template <typename T>
__global__ void __launch_bounds__(256) k3_faraday1(Geo g, Coef<T> c, const T *__restrict__ e0, const T *__restrict__ e1,
                                                   const T *__restrict__ e2, T *__restrict__ b0, T *__restrict__ b1,
                                                   T *__restrict__ b2, int zseg) {
    const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (x >= g.nx || y >= g.ny) return;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    const int o = y * (int)g.pitch + x;
    const int ox = o + (x + 1 < g.nx ? 1 : 1 - g.nx), oy = o + (y + 1 < g.ny ? (int)g.pitch : -(g.ny - 1) * (int)g.pitch);
    int64_t z = (int64_t)z0 * g.plane;
    T ex = e0[z + o], ey = e1[z + o];
    for (int k = z0; k < z1; ++k) {
        const int64_t zn = k + 1 < g.nz ? z + g.plane : 0;
        const T ez = e2[z + o], exn = e0[zn + o], eyn = e1[zn + o];
        const T bx = b0[z + o], by = b1[z + o], bz = b2[z + o];
        const T ezx = e2[z + ox], ezy = e2[z + oy], eyx = e1[z + ox], exy = e0[z + oy];
        b0[z + o] = (bx - c.ky * (ezy - ez)) + c.kz * (eyn - ey);
        b1[z + o] = (by - c.kz * (exn - ex)) + c.kx * (ezx - ez);
        b2[z + o] = (bz - c.kx * (eyx - ey)) + c.ky * (exy - ex);
        ex = exn;
        ey = eyn;
        z = zn;
    }
}

// ---------------------------------------------------------------------------
// FP32 sweep, two adjacent columns per thread (even n_x).  The tile is 64
// columns x 8 rows; a smem row holds column x0 + j at index j + 2 (j = -1..64),
// so a thread's own pair sits at an even index and is one 8-byte load, and its
// x-neighbours (columns 2t-1 and 2t+2) are single loads.  The A operator is
// evaluated on column pairs with packed FP32x2 arithmetic.  The planes arrive
// by cp.async like the scalar kernel's (8-byte copies of column pairs, 4-byte
// copies of the two halo columns); dE' of the thread's own pair is prefetched
// into registers two planes ahead (E^n, when the sweep also applies the update
// E^{n+1} = E^n + dE, one plane ahead).
using pair2::f2;
constexpr int TXP = 32, TX2 = 2 * TXP;              // threads along x, columns of the tile
constexpr int RW2 = TX2 + 4, PL2 = RW2 * RH;         // smem row and plane (one component)
constexpr int NPC = TXP * RH, NCP2 = NPC + 2 * RH;  // pair copies and halo copies per plane
constexpr int FAR_RS = 8;    // ring slots of the pair Faraday update
constexpr int SWEEP_RS = 8;  // ring slots of the pair sweep: one plane read, seven in flight

struct Coef3P {
    f2 ax, ay, az, ayz, azx, axy, byz, bzx, bxy, c6, kx, ky, kz, q;
    f2 q64;  // q / 64: the one-pass 3D binomial with integer weights (exact power-of-two scaling)
};
template <int AX>
__device__ __forceinline__ f2 ck(const Coef3P &c) {
    return AX == 0 ? c.kx : (AX == 1 ? c.ky : c.kz);
}

// a thread's (at most two) copy items of a component plane, and the plane the
// z-march copies next: its index unwrapped (which picks the ring slot) and
// the element offset of the plane wrapped periodically, advanced one plane
// per copy so that no plane index is divided by n_z on the way
struct PairCopies {
    int s[2], o[2];  // smem index within a component plane (-1: none), global in-plane offset
    bool w[2];       // column pair (8 bytes) or halo column (4 bytes)
    int ku;          // planes copied so far
    int64_t off;     // element offset of that plane wrapped into [0, n_z)
    __device__ __forceinline__ void init(const Geo &g, int x0, int y0, int k0) {
        const int tid = threadIdx.y * TXP + threadIdx.x;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int q = tid + r * NTH;
            s[r] = -1;
            o[r] = 0;
            w[r] = false;
            if (q < NCP2) {
                int row, j;
                if (q < NPC) {
                    row = q / TXP;
                    j = 2 * (q % TXP);
                    w[r] = true;
                } else {
                    const int h = q - NPC;
                    row = h / 2;
                    j = (h & 1) ? TX2 : -1;
                }
                const int x = wrapm(x0 + j, g.nx), y = wrapm(y0 - 1 + row, g.ny);
                s[r] = row * RW2 + 2 + j;
                o[r] = y * (int)g.pitch + x;
            }
        }
        ku = 0;
        off = (int64_t)wrapm(k0, g.nz) * g.plane;
    }
    // copies the next plane of the N components into ring slot ku mod RS, then
    // moves on to the next plane
    template <int RS, int N = 3>
    __device__ __forceinline__ void issue_next(float *ring, const float *const src[N], const Geo &g) {
        float *slot = ring + (ku & (RS - 1)) * N * PL2;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (s[r] < 0) continue;
            const int64_t go = off + o[r];
#pragma unroll
            for (int c = 0; c < N; ++c) {
                float *dst = slot + c * PL2 + s[r];
                const float *sp = src[c] + go;
                if (w[r]) cp_async_pair(dst, sp);
                else cp_async_el(dst, sp);
            }
        }
        ++ku;
        off += g.plane;
        if (off == (int64_t)g.nz * g.plane) off = 0;
    }
};

// The A operator factored for a z-march.  Operators along different axes
// commute, so every element of A (Eqs. matrixA_1st..matrixA_last, 3D) is an
// in-plane (x, y) stencil of one z-plane followed by a 3-point combination
// along z:
//   (A dE)_x(k) = a_y P_k + a_z Dzz Ex + a_yz Dzz P + b_xy (G_k + c6 Dzz G) + b_zx (N_k - N_(k-1)),
//   (A dE)_y(k) = a_x Q_k + a_z Dzz Ey + a_zx Dzz Q + b_xy (G'_k + c6 Dzz G') + b_yz (N'_k - N'_(k-1)),
//   (A dE)_z(k) = T_k + H_(k+1) - H_k,
// with Dzz f = f_(k+1) - 2 f_k + f_(k-1) and the in-plane fields
//   P = Dbar_yy Ex,  G = Dbar_x(fwd) Dbar_y(bwd) Ey,  N = Dbar_x(fwd) (Ez + c6 Dbar_yy Ez),
//   Q = Dbar_xx Ey,  G' = Dbar_y(fwd) Dbar_x(bwd) Ex,  N' = Dbar_y(fwd) (Ez + c6 Dbar_xx Ez),
//   T = (a_x Dbar_xx + a_y Dbar_yy + a_xy Dbar_xx Dbar_yy) Ez,
//   H = b_zx Dbar_x(bwd) (Ex + c6 Dbar_yy Ex) + b_yz Dbar_y(bwd) (Ey + c6 Dbar_xx Ey).
// Plane j of the sweep's input therefore reaches outputs j-1, j and j+1
// through the combinations below, computed once from plane j alone (21
// shared-memory loads per column pair against 51 for the 27-point form).
struct PlaneTerms {
    f2 x1, x0, xl;  // x: to outputs j-1 and j+1 (x1), to j (x0), to j+1 (xl = x1 - b_zx N)
    f2 y1, y0, yl;  // y: the same with G', N', Q
    f2 zh, zt;      // z: H to output j-1, T - H to output j
};

template <typename F>
__device__ __forceinline__ PlaneTerms plane_terms(const F &V, const Coef3P &c, f2 bxy6) {
    using namespace pair2;
    auto d2 = [](f2 p, f2 o, f2 m) { return fma(o, m2(), add(p, m)); };  // p - 2 o + m
    auto sub = [](f2 a, f2 b) { return fma(b, m1(), a); };
    // Ex at columns x-1, x and rows y-1, y, y+1
    const f2 ex_m = V(0, 0, -1), ex_0 = V(0, 0, 0), ex_p = V(0, 0, 1);
    const f2 exl_m = V(0, -1, -1), exl_0 = V(0, -1, 0), exl_p = V(0, -1, 1);
    // Ey at columns x-1, x, x+1 and rows y-1, y
    const f2 ey_m = V(1, 0, -1), ey_0 = V(1, 0, 0);
    const f2 eyl_m = V(1, -1, -1), eyl_0 = V(1, -1, 0), eyr_m = V(1, 1, -1), eyr_0 = V(1, 1, 0);
    // Ez at columns x-1..x+1 and rows y-1..y+1: ez[dy + 1][dx + 1]
    f2 ez[3][3];
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) ez[dy + 1][dx + 1] = V(2, dx, dy);
    const f2 P = d2(ex_p, ex_0, ex_m), Pl = d2(exl_p, exl_0, exl_m);  // Dbar_yy Ex at x, x-1
    const f2 Q = d2(eyr_0, ey_0, eyl_0), Qm = d2(eyr_m, ey_m, eyl_m);  // Dbar_xx Ey at y, y-1
    const f2 G = sub(sub(eyr_0, ey_0), sub(eyr_m, ey_m));
    const f2 Gp = sub(sub(ex_p, exl_p), sub(ex_0, exl_0));
    const f2 dxz_m = d2(ez[0][2], ez[0][1], ez[0][0]), dxz_0 = d2(ez[1][2], ez[1][1], ez[1][0]),
             dxz_p = d2(ez[2][2], ez[2][1], ez[2][0]);  // Dbar_xx Ez at y-1, y, y+1
    const f2 dyz_0 = d2(ez[2][1], ez[1][1], ez[0][1]), dyz_r = d2(ez[2][2], ez[1][2], ez[0][2]);  // Dbar_yy Ez at x, x+1
    const f2 N = sub(fma(c.c6, dyz_r, ez[1][2]), fma(c.c6, dyz_0, ez[1][1]));
    const f2 Np = sub(fma(c.c6, dxz_p, ez[2][1]), fma(c.c6, dxz_0, ez[1][1]));
    const f2 T = fma(c.axy, d2(dxz_p, dxz_0, dxz_m), fma(c.ay, dyz_0, mul(c.ax, dxz_0)));
    const f2 X = sub(fma(c.c6, P, ex_0), fma(c.c6, Pl, exl_0));
    const f2 Y = sub(fma(c.c6, Q, ey_0), fma(c.c6, Qm, ey_m));
    PlaneTerms t;
    t.zh = fma(c.byz, Y, mul(c.bzx, X));
    t.zt = sub(T, t.zh);
    const f2 bN = mul(c.bzx, N), bNp = mul(c.byz, Np);
    t.x1 = fma(bxy6, G, fma(c.ayz, P, mul(c.az, ex_0)));
    t.x0 = fma(t.x1, m2(), add(bN, fma(c.bxy, G, mul(c.ay, P))));
    t.xl = sub(t.x1, bN);
    t.y1 = fma(bxy6, Gp, fma(c.azx, Q, mul(c.az, ey_0)));
    t.y0 = fma(t.y1, m2(), add(bNp, fma(c.bxy, Gp, mul(c.ax, Q))));
    t.yl = sub(t.y1, bNp);
    return t;
}

// out = dEp + A in, or with UPD: E = E + dEp + A in (the last sweep and the
// update of the step in one pass; E in place).  The CTA marches its input
// planes z0-1..z1 once each: iteration i reads plane z0-1+i from the ring
// (nothing else of the plane is read again), adds its terms to the partial
// outputs held in registers, and completes output plane z0+i-2.  One plane
// is read while the next RS-1 are on their way; one barrier per plane.
// FIRST: the first sweep, whose input is dE' itself: the own pair of an output
// plane was read from the ring one iteration before, so dE' is not fetched a
// second time (512^3: 822 -> 689 us).
template <bool UPD, bool FIRST>
__global__ void __launch_bounds__(NTH, UPD ? 2 : 3) k3_sweep2(Geo g, Coef3P c, const float *p0, const float *p1,
                                                             const float *p2, const float *i0, const float *i1,
                                                             const float *i2, float *o0, float *o1, float *o2, int zseg) {
    using namespace pair2;
    constexpr int RS = SWEEP_RS;
    extern __shared__ __align__(16) unsigned char m3raw[];
    float *ring = reinterpret_cast<float *>(m3raw);  // [RS][3][PL2]
    const float *in[3] = {i0, i1, i2};
    const float *dp[3] = {p0, p1, p2};
    float *out[3] = {o0, o1, o2};
    const int x0 = blockIdx.x * TX2, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    const int np = z1 - z0 + 2;  // input planes z0-1 .. z1
    PairCopies cp;
    cp.init(g, x0, y0, z0 - 1);
    const int px = x0 + 2 * threadIdx.x, py = y0 + threadIdx.y;
    const bool inside = px < g.nx && py < g.ny;
    const int c0 = (threadIdx.y + 1) * RW2 + 2 + 2 * threadIdx.x;
    // copy group i: input plane z0-1+i (empty past the last)
    auto issue = [&](int i) {
        if (i < np) cp.issue_next<RS>(ring, in, g);
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < RS - 1; ++i) issue(i);
    // own-pair offsets: of the output completed next, and of the one two
    // planes later (the register prefetch); outputs lie in [z0, z1), no wrap
    int64_t ocell = (int64_t)z0 * g.plane + (int64_t)py * g.pitch + px;
    int64_t pcell = ocell;
    // dE' (and E^n) of the own pair of outputs o and o+1: two register buffers
    f2 pd[2][3], pe[2][3];
    auto prefetch = [&](int b, bool ok) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            pd[b][q] = mk(0.f, 0.f);
            pe[b][q] = mk(0.f, 0.f);
            if (ok) {
                if (!FIRST) pd[b][q] = __ldg(reinterpret_cast<const float2 *>(dp[q] + pcell));
                if (UPD) pe[b][q] = *reinterpret_cast<const float2 *>(out[q] + pcell);
            }
        }
        pcell += g.plane;
    };
    if (!FIRST || UPD) {
        prefetch(0, inside);
        prefetch(1, inside && z0 + 1 < z1);
    }
    f2 pv[3];  // FIRST: the own pair of the plane before
#pragma unroll
    for (int q = 0; q < 3; ++q) pv[q] = mk(0.f, 0.f);
    const f2 bxy6 = mul(c.bxy, c.c6);
    f2 xa = mk(0.f, 0.f), xb = xa, ya = xa, yb = xa, za = xa;  // partial outputs o, o+1
    auto step = [&](int i, auto bsel) {
        constexpr int b = decltype(bsel)::value;
        cp_async_wait<RS - 2>();
        __syncthreads();
        issue(i + RS - 1);
        if (inside) {
            const float *pl = ring + (i & (RS - 1)) * 3 * PL2 + c0;  // the copy's slot of plane z0-1+i
            auto V = [&](int q, int dx, int dy) -> f2 {
                const float *row = pl + q * PL2 + dy * RW2;
                const f2 pr = *reinterpret_cast<const float2 *>(row);
                return dx == 0 ? pr : (dx > 0 ? mk(pr.y, row[2]) : mk(row[-1], pr.x));
            };
            const PlaneTerms t = plane_terms(V, c, bxy6);
            if (i >= 2) {
                // output plane z0 + i - 2 is complete
                f2 r[3] = {add(xa, t.x1), add(ya, t.y1), add(za, t.zh)};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    r[q] = add(FIRST ? pv[q] : pd[b][q], r[q]);
                    if (UPD) r[q] = add(pe[b][q], r[q]);
                    *reinterpret_cast<float2 *>(out[q] + ocell) = r[q];
                }
                ocell += g.plane;
                if (!FIRST || UPD) prefetch(b, z0 + i < z1);  // output z0 + i, two iterations on
            }
            if (FIRST) {
#pragma unroll
                for (int q = 0; q < 3; ++q) pv[q] = V(q, 0, 0);
            }
            xa = add(xb, t.x0);
            xb = t.xl;
            ya = add(yb, t.y0);
            yb = t.yl;
            za = t.zt;
        }
    };
    for (int i = 0; i < np; i += 2) {
        step(i, std::integral_constant<int, 0>());
        if (i + 1 < np) step(i + 1, std::integral_constant<int, 1>());
    }
    cp_async_wait<0>();
}

// dE' = C_b (alpha B) - q F j on a column pair, 3D (the source of k3_source,
// curl_alpha_b in stencil.cuh); F = one (1/4, 1/2, 1/4) pass along each axis
// (PASSES = 1) or none.  The averaged curl (Eqs. ampere_aux_x..z) factored
// like the sweep's A, the z-differences moved outside:
//   x: k_y (V_k + c6 Dzz V) - k_z (U_k - U_(k-1)),    V = Dbar_y(bwd) Bz,  U = By + c6 Dbar_yy By,
//   y: k_z (W_k - W_(k-1)) - k_x (V'_k + c6 Dzz V'),  V' = Dbar_x(bwd) Bz, W = Bx + c6 Dbar_xx Bx,
//   z: k_x Dbar_x(bwd) U - k_y Dbar_y(bwd) W          (in-plane),
// so plane j of B reaches outputs j-1, j, j+1 through terms of plane j, and U and
// W of plane j-1 (their z-differences are taken before the factor: on smooth
// fields a difference is exact where the products' sum would round at |B|; with
// it the source spills nothing and 512^3 takes 5.39 ms a step against 5.50).
struct CurlTerms {
    f2 x1, x0;  // x: to outputs j-1 and j+1 (x1), to j (x0, without k_z (U - U_(j-1)))
    f2 y1, y0;  // y: the same with V', and W
    f2 U, W;
    f2 z;       // z: to output j
};

template <typename F>
__device__ __forceinline__ CurlTerms curl_plane_terms(const F &V, const Coef3P &c, f2 nkxc6, f2 kyc6) {
    using namespace pair2;
    auto d2 = [](f2 p, f2 o, f2 m) { return fma(o, m2(), add(p, m)); };  // p - 2 o + m
    auto sub = [](f2 a, f2 b) { return fma(b, m1(), a); };
    // Bx at columns x-1..x+1 and rows y-1, y
    const f2 bx_m = V(0, 0, -1), bx_0 = V(0, 0, 0);
    const f2 bxl_m = V(0, -1, -1), bxl_0 = V(0, -1, 0), bxr_m = V(0, 1, -1), bxr_0 = V(0, 1, 0);
    // By at columns x-1, x and rows y-1..y+1
    const f2 by_m = V(1, 0, -1), by_0 = V(1, 0, 0), by_p = V(1, 0, 1);
    const f2 byl_m = V(1, -1, -1), byl_0 = V(1, -1, 0), byl_p = V(1, -1, 1);
    // Bz at (x, y-1), (x, y), (x-1, y)
    const f2 bz_m = V(2, 0, -1), bz_0 = V(2, 0, 0), bzl_0 = V(2, -1, 0);
    const f2 U = fma(c.c6, d2(by_p, by_0, by_m), by_0), Ul = fma(c.c6, d2(byl_p, byl_0, byl_m), byl_0);
    const f2 W = fma(c.c6, d2(bxr_0, bx_0, bxl_0), bx_0), Wm = fma(c.c6, d2(bxr_m, bx_m, bxl_m), bx_m);
    const f2 Vy = sub(bz_0, bz_m), Vx = sub(bz_0, bzl_0);
    CurlTerms t;
    t.x1 = mul(kyc6, Vy);
    t.x0 = fma(t.x1, m2(), mul(c.ky, Vy));
    t.y1 = mul(nkxc6, Vx);
    t.y0 = fma(t.y1, m2(), mul(mul(c.kx, Vx), m1()));
    t.U = U;
    t.W = W;
    t.z = sub(mul(c.kx, sub(U, Ul)), mul(c.ky, sub(W, Wm)));
    return t;
}

// Ring: B (and j) planes of the 64 x 8 tile, RS slots.  The CTA marches its
// input planes z0-1..z1 once each, like the sweep: iteration i reads plane
// z0-1+i (B for the curl terms, j for its x-y binomial), and completes output
// plane z0+i-2; the z part of the binomial combines the x-y results of the
// last three planes, kept in registers.  One plane is read while the next
// RS-1 are on their way; one barrier per plane.
template <int RS, int PASSES, bool HJ>
__global__ void __launch_bounds__(NTH, 3) k3_source2(Geo g, Coef3P c, const float *b0, const float *b1,
                                                    const float *b2, const float *j0, const float *j1,
                                                    const float *j2, float *o0, float *o1, float *o2, int zseg) {
    using namespace pair2;
    constexpr int N = HJ ? 6 : 3;
    extern __shared__ __align__(16) unsigned char m3raw[];
    float *ring = reinterpret_cast<float *>(m3raw);  // [RS][N][PL2]
    const float *src[6] = {b0, b1, b2, j0, j1, j2};
    float *out[3] = {o0, o1, o2};
    const int x0 = blockIdx.x * TX2, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    const int np = z1 - z0 + 2;  // input planes z0-1 .. z1
    PairCopies cp;
    cp.init(g, x0, y0, z0 - 1);
    const int px = x0 + 2 * threadIdx.x, py = y0 + threadIdx.y;
    const bool inside = px < g.nx && py < g.ny;
    const int c0 = (threadIdx.y + 1) * RW2 + 2 + 2 * threadIdx.x;
    // copy group i: input plane z0-1+i (empty past the last)
    auto issue = [&](int i) {
        if (i < np) cp.issue_next<RS, N>(ring, src, g);
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < RS - 1; ++i) issue(i);
    int64_t ocell = (int64_t)z0 * g.plane + (int64_t)py * g.pitch + px;
    const f2 nkxc6 = mul(mul(c.kx, c.c6), m1()), kyc6 = mul(c.ky, c.c6);
    f2 xa = mk(0.f, 0.f), xb = xa, ya = xa, yb = xa, za = xa;  // partial outputs o, o+1
    f2 up = xa, wp = xa;  // U and W of the plane before
    // PASSES = 1: x-y binomial of the current of planes j-2, j-1 (own pair);
    // PASSES = 0: the raw current of plane j-1 in jz[a][1]
    f2 jz[3][2];
#pragma unroll
    for (int a = 0; a < 3; ++a) jz[a][0] = jz[a][1] = xa;
    for (int i = 0; i < np; ++i) {
        cp_async_wait<RS - 2>();
        __syncthreads();
        issue(i + RS - 1);
        if (inside) {
            const float *pl = ring + (i & (RS - 1)) * N * PL2 + c0;  // the copy's slot of plane z0-1+i
            auto V = [&](int q, int dx, int dy) -> f2 {
                const float *row = pl + q * PL2 + dy * RW2;
                const f2 pr = *reinterpret_cast<const float2 *>(row);
                return dx == 0 ? pr : (dx > 0 ? mk(pr.y, row[2]) : mk(row[-1], pr.x));
            };
            const CurlTerms t = curl_plane_terms(V, c, nkxc6, kyc6);
            f2 jn[3];
            if constexpr (HJ) {
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if constexpr (PASSES == 1) {
                        // separable binomial with integer weights (1, 2, 1) per axis,
                        // the 1/64 folded into q: the x-y part here
                        f2 acc = mk(0.f, 0.f);
#pragma unroll
                        for (int dy = -1; dy <= 1; ++dy) {
                            const f2 rowf = fma(V(3 + a, 0, dy), cst(2), add(V(3 + a, -1, dy), V(3 + a, 1, dy)));
                            acc = fma(cst(2 - dy * dy), rowf, acc);
                        }
                        jn[a] = acc;
                    } else {
                        jn[a] = V(3 + a, 0, 0);
                    }
                }
            }
            if (i >= 2) {
                // output plane z0 + i - 2 is complete
                f2 d[3] = {add(xa, t.x1), add(ya, t.y1), za};
                if constexpr (HJ) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        if constexpr (PASSES == 1) {
                            const f2 jsum = fma(jz[a][1], cst(2), add(jz[a][0], jn[a]));
                            d[a] = fma(mul(c.q64, jsum), m1(), d[a]);
                        } else {
                            d[a] = fma(mul(c.q, jz[a][1]), m1(), d[a]);
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) *reinterpret_cast<float2 *>(out[q] + ocell) = d[q];
                ocell += g.plane;
            }
            xa = fma(mul(c.kz, fma(up, m1(), t.U)), m1(), add(xb, t.x0));
            xb = t.x1;
            ya = fma(c.kz, fma(wp, m1(), t.W), add(yb, t.y0));
            yb = t.y1;
            up = t.U;
            wp = t.W;
            za = t.z;
            if constexpr (HJ) {
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    jz[a][0] = jz[a][1];
                    jz[a][1] = jn[a];
                }
            }
        }
    }
    cp_async_wait<0>();
}

// B -= c dt curl E^{n+1} (Eqs. faraday_x..z) on a column pair, 3D: forward
// differences (curl_e in stencil.cuh) of E from the plane ring
template <int A, typename F>
__device__ __forceinline__ f2 curl_e2(const F &V, const Coef3P &c) {
    using namespace pair2;
    constexpr int B = (A + 1) % 3, C = (A + 2) % 3;
    constexpr int bx = B == 0, by = B == 1, bz = B == 2, cx = C == 0, cy = C == 1, cz = C == 2;
    const f2 r = mul(ck<B>(c), fma(V(C, 0, 0, 0), m1(), V(C, bx, by, bz)));
    return fma(mul(ck<C>(c), fma(V(B, 0, 0, 0), m1(), V(B, cx, cy, cz))), m1(), r);
}

__global__ void __launch_bounds__(NTH, 3) k3_faraday2(Geo g, Coef3P c, const float *e0, const float *e1,
                                                     const float *e2, float *b0, float *b1, float *b2, int zseg) {
    using namespace pair2;
    constexpr int RS = FAR_RS, LA = RS - 3;  // LA: copy groups in flight ahead of the plane computed
    extern __shared__ __align__(16) unsigned char m3raw[];
    float *ring = reinterpret_cast<float *>(m3raw);  // [RS][3][PL2] E^{n+1} planes
    const float *in[3] = {e0, e1, e2};
    float *bo[3] = {b0, b1, b2};
    const int x0 = blockIdx.x * TX2, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    PairCopies cp;
    cp.init(g, x0, y0, z0);
    const int px = x0 + 2 * threadIdx.x, py = y0 + threadIdx.y;
    const bool inside = px < g.nx && py < g.ny;
    const int64_t cell = (int64_t)py * g.pitch + px;
    const int c0 = (threadIdx.y + 1) * RW2 + 2 + 2 * threadIdx.x;
    // copy group m: planes z0, z0+1 (m = 0), plane z0+1+m (m >= 1, up to z1)
    auto issue = [&](int m) {
        if (m == 0) cp.issue_next<RS>(ring, in, g);
        if (z0 + 1 + m <= z1) cp.issue_next<RS>(ring, in, g);
        cp_async_commit();
    };
    // B of the own pair, planes k and k+1: two register buffers
    f2 pb[2][3];
    auto ldown = [&](int k, int b) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            pb[b][q] = mk(0.f, 0.f);
            if (inside && k < z1) pb[b][q] = *reinterpret_cast<const float2 *>(bo[q] + (int64_t)k * g.plane + cell);
        }
    };
#pragma unroll
    for (int m = 0; m < LA; ++m) issue(m);
    ldown(z0, 0);
    ldown(z0 + 1, 1);
    auto step = [&](int k, auto bsel) {
        constexpr int b = decltype(bsel)::value;
        cp_async_wait<LA - 1>();
        __syncthreads();
        issue(k - z0 + LA);
        f2 bv[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) bv[q] = pb[b][q];
        ldown(k + 2, b);
        if (inside) {
            const int s0 = ((k - z0) & (RS - 1)) * 3 * PL2, sp1 = ((k - z0 + 1) & (RS - 1)) * 3 * PL2;
            auto V = [&](int q, int dx, int dy, int dz) -> f2 {
                const float *row = ring + (dz > 0 ? sp1 : s0) + q * PL2 + c0 + dy * RW2;
                const f2 pr = *reinterpret_cast<const float2 *>(row);
                return dx == 0 ? pr : (dx > 0 ? mk(pr.y, row[2]) : mk(row[-1], pr.x));
            };
            const f2 r[3] = {curl_e2<0>(V, c), curl_e2<1>(V, c), curl_e2<2>(V, c)};
            const int64_t idx = (int64_t)k * g.plane + cell;
#pragma unroll
            for (int q = 0; q < 3; ++q) *reinterpret_cast<float2 *>(bo[q] + idx) = fma(r[q], m1(), bv[q]);
        }
    };
    for (int k = z0; k < z1; k += 2) {
        step(k, std::integral_constant<int, 0>());
        if (k + 1 < z1) step(k + 1, std::integral_constant<int, 1>());
    }
    cp_async_wait<0>();
}

// ---------------------------------------------------------------------------
// Two sweeps of Algorithm 1 in one z-march (temporal blocking, FP32 column
// pairs, even n_x): dE_(s+2) = dE' + A (dE' + A dE_(s)), both sweeps in the
// factored form of plane_terms.  The first sweep (A stage) is evaluated on the
// output tile grown by one cell on every side in x and y (34 pairs x 10 rows
// around the 32 x 8 pairs of the tile), from an input ring whose planes carry
// a halo of two; each plane of dE_(s+1) it completes goes into one of two
// shared-memory plane buffers, which the second sweep (B stage) reads one
// iteration later, so dE_(s+1) never leaves the SM.  352 threads: every
// thread but the last 12 owns a first-sweep pair, the first 256 also the
// second-sweep pair of the tile.  Iteration i: the A stage reads input plane
// z0-2+i and completes first-sweep plane z0+i-3; the B stage reads
// first-sweep plane z0+i-4 and completes output plane z0+i-5.  One barrier
// per iteration.  With UPD the second sweep also applies E^{n+1} = E^n + dE
// (E in place).
constexpr int FRW = 72;                // floats per row: column x0 + j at index j + 4, j in [-4, 67]
constexpr int FIR = 12, FAR = 10;      // rows of an input plane (y0-2..y0+9) and of a first-sweep plane (y0-1..y0+8)
constexpr int FIPL = FRW * FIR, FAPL = FRW * FAR;
constexpr int FNT = 352, FNA = 340, FNB = 256;
constexpr int FRS = 4;                 // input ring slots: one plane read, three in flight
constexpr int FNI = (FRW / 2) * FIR;   // pair copies per input plane and component (432)

template <bool UPD>
__global__ void __launch_bounds__(FNT, 2) k3_sweeps2f(Geo g, Coef3P c, const float *p0, const float *p1,
                                                     const float *p2, const float *i0, const float *i1,
                                                     const float *i2, float *o0, float *o1, float *o2, int zseg) {
    using namespace pair2;
    extern __shared__ __align__(16) unsigned char m3raw[];
    float *ring = reinterpret_cast<float *>(m3raw);  // [FRS][3][FIPL] input planes, halo 2
    float *abuf = ring + FRS * 3 * FIPL;              // [2][3][FAPL] first-sweep planes, halo 1
    const float *in[3] = {i0, i1, i2};
    const float *dp[3] = {p0, p1, p2};
    float *out[3] = {o0, o1, o2};
    const int x0 = blockIdx.x * TX2, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zseg, z1 = min(z0 + zseg, g.nz);
    const int nin = z1 - z0 + 4;  // input planes z0-2 .. z1+1
    const int tid = threadIdx.x;
    const int64_t vol = (int64_t)g.nz * g.plane;
    // input copy items of this thread (pairs of columns, periodic wrap), and
    // the wrapped offset of the plane copied next
    int cs[2], co[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int q = tid + r * FNT;
        cs[r] = -1;
        co[r] = 0;
        if (q < FNI) {
            const int row = q / (FRW / 2), j = 2 * (q % (FRW / 2)) - 4;
            cs[r] = row * FRW + j + 4;
            co[r] = wrapm(y0 - 2 + row, g.ny) * (int)g.pitch + wrapm(x0 + j, g.nx);
        }
    }
    int64_t koff = (int64_t)wrapm(z0 - 2, g.nz) * g.plane;
    // copy group i: input plane z0-2+i (empty past the last)
    auto issue = [&](int i) {
        if (i < nin) {
            float *slot = ring + (i & (FRS - 1)) * 3 * FIPL;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (cs[r] < 0) continue;
                const int64_t go = koff + co[r];
#pragma unroll
                for (int q = 0; q < 3; ++q) cp_async_pair(slot + q * FIPL + cs[r], in[q] + go);
            }
            koff += g.plane;
            if (koff == vol) koff = 0;
        }
        cp_async_commit();
    };
    // first-sweep pair (A stage) and second-sweep pair (B stage) of this thread
    const bool hasA = tid < FNA, hasB = tid < FNB;
    const int pa = tid % 34 - 1, ra = tid / 34 - 1;  // pair -1..32, row -1..8
    const int pb = tid % 32, rb = tid / 32;          // pair 0..31, row 0..7
    const int cA = (ra + 2) * FRW + 2 * pa + 4;      // input-plane index of the A pair
    const int wA = (ra + 1) * FRW + 2 * pa + 4;      // first-sweep-plane index of the A pair
    const int cB = (rb + 1) * FRW + 2 * pb + 4;      // first-sweep-plane index of the B pair
    const bool outB = hasB && x0 + 2 * pb < g.nx && y0 + rb < g.ny;
    // own-pair offsets: A's dE' of its next plane (wrapped periodically: the
    // grown tile reaches planes z0-1 and z1), B's next output plane
    const int cellA = wrapm(y0 + ra, g.ny) * (int)g.pitch + wrapm(x0 + 2 * pa, g.nx);
    int64_t aoff = (int64_t)wrapm(z0 - 1, g.nz) * g.plane;
    int64_t bcell = (int64_t)z0 * g.plane + (int64_t)(y0 + rb) * g.pitch + (x0 + 2 * pb);
    f2 pa_d[3], pb_d[3], pb_e[3];  // dE' of A's next plane; dE' (and E^n) of B's next output
    auto load_a = [&]() {
#pragma unroll
        for (int q = 0; q < 3; ++q) pa_d[q] = __ldg(reinterpret_cast<const float2 *>(dp[q] + aoff + cellA));
        aoff += g.plane;
        if (aoff == vol) aoff = 0;
    };
    // B's output plane at offset `at` (bcell, or the plane after it)
    auto load_b = [&](bool ok, int64_t at) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            pb_d[q] = ok ? __ldg(reinterpret_cast<const float2 *>(dp[q] + at)) : mk(0.f, 0.f);
            if (UPD) pb_e[q] = ok ? *reinterpret_cast<const float2 *>(out[q] + at) : mk(0.f, 0.f);
        }
    };
#pragma unroll
    for (int i = 0; i < FRS - 1; ++i) issue(i);
    const f2 bxy6 = mul(c.bxy, c.c6);
    f2 ax_a = mk(0.f, 0.f), ax_b = ax_a, ay_a = ax_a, ay_b = ax_a, az_a = ax_a;  // A: partial planes o, o+1
    f2 bx_a = ax_a, bx_b = ax_a, by_a = ax_a, by_b = ax_a, bz_a = ax_a;          // B: the same
    for (int i = 0; i < nin + 1; ++i) {
        cp_async_wait<FRS - 2>();
        __syncthreads();
        issue(i + FRS - 1);
        // A stage: input plane z0-2+i; completes first-sweep plane z0+i-3 (i >= 2)
        if (hasA && i < nin) {
            if (i == 1) load_a();  // dE' of plane z0-1
            const float *pl = ring + (i & (FRS - 1)) * 3 * FIPL + cA;
            auto V = [&](int q, int dx, int dy) -> f2 {
                const float *row = pl + q * FIPL + dy * FRW;
                const f2 pr = *reinterpret_cast<const float2 *>(row);
                return dx == 0 ? pr : (dx > 0 ? mk(pr.y, row[2]) : mk(row[-1], pr.x));
            };
            const PlaneTerms t = plane_terms(V, c, bxy6);
            if (i >= 2) {
                float *dst = abuf + ((i + 1) & 1) * 3 * FAPL + wA;
                *reinterpret_cast<float2 *>(dst) = add(pa_d[0], add(ax_a, t.x1));
                *reinterpret_cast<float2 *>(dst + FAPL) = add(pa_d[1], add(ay_a, t.y1));
                *reinterpret_cast<float2 *>(dst + 2 * FAPL) = add(pa_d[2], add(az_a, t.zh));
                if (i + 1 < nin) load_a();  // dE' of plane z0+i-2, next iteration
            }
            ax_a = add(ax_b, t.x0);
            ax_b = t.xl;
            ay_a = add(ay_b, t.y0);
            ay_b = t.yl;
            az_a = t.zt;
        }
        // B stage: first-sweep plane z0+i-4 (i >= 3); completes output plane z0+i-5 (i >= 5)
        if (hasB && i >= 3) {
            if (i == 4) load_b(outB, bcell);  // output z0
            const float *pl = abuf + (i & 1) * 3 * FAPL + cB;
            auto V = [&](int q, int dx, int dy) -> f2 {
                const float *row = pl + q * FAPL + dy * FRW;
                const f2 pr = *reinterpret_cast<const float2 *>(row);
                return dx == 0 ? pr : (dx > 0 ? mk(pr.y, row[2]) : mk(row[-1], pr.x));
            };
            const PlaneTerms t = plane_terms(V, c, bxy6);
            if (i >= 5) {
                f2 r[3] = {add(bx_a, t.x1), add(by_a, t.y1), add(bz_a, t.zh)};
                if (outB) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        r[q] = add(pb_d[q], r[q]);
                        if (UPD) r[q] = add(pb_e[q], r[q]);
                        *reinterpret_cast<float2 *>(out[q] + bcell) = r[q];
                    }
                }
                bcell += g.plane;
                load_b(outB && z0 + i - 4 < z1, bcell);  // output z0+i-4, next iteration
            }
            bx_a = add(bx_b, t.x0);
            bx_b = t.xl;
            by_a = add(by_b, t.y0);
            by_b = t.yl;
            bz_a = t.zt;
        }
    }
    cp_async_wait<0>();
}

// launch grid of a kernel with CTAs of tx columns x ty rows, zseg planes each
dim3 grid_of(const Geo &g, int tx, int ty, int res, int *zseg, double lat = 0.5) {
    const dim3 t((g.nx + tx - 1) / tx, (g.ny + ty - 1) / ty);
    *zseg = zseg_for(g.nz, (long long)t.x * t.y, res, lat);
    return dim3(t.x, t.y, (g.nz + *zseg - 1) / *zseg);
}
// allows the dynamic shared memory and returns the CTAs an SM holds
template <typename K>
int resident(K k, int threads, size_t bytes) {
    int n = 0;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, bytes) == cudaSuccess && n > 0 ? n : 1;
}

}  // namespace

bool march3d_supported(int dims, int passes) { return dims == 3 && passes >= 0 && passes <= 1; }

// four rows per thread, in the shortest segments, are at most a quarter of the
// chip's warp schedulers' worth of warps: one row per thread then (128 x 127 x 1 FP64,
// m = 4: 147 us a step with four)
bool one_row(const Geo &g) {
    const double tiles = (double)((g.nx + CX - 1) / CX) * (double)((g.ny + 4 * CW - 1) / (4 * CW));
    return tiles * CW * g.nz <= sm_count();
}

template <typename T, int PASSES, bool HJ, int CR>
void run_source(const Geo &g, const Coef<T> &c, const T *const B[3], const T *const J[3], T *const out[3],
                cudaStream_t s) {
    constexpr size_t bytes = (size_t)SOURCE1_RS * (HJ ? 6 : 3) * cpl(CR) * sizeof(T);
    static const int res = resident(k3_source1<T, PASSES, HJ, CR>, CNT, bytes);
    int zseg;
    const dim3 grid = grid_of(g, CX, CR * CW, res, &zseg, 0.6);
    k3_source1<T, PASSES, HJ, CR><<<grid, CNT, bytes, s>>>(g, c, B[0], B[1], B[2], HJ ? J[0] : nullptr,
                                                           HJ ? J[1] : nullptr, HJ ? J[2] : nullptr, out[0], out[1],
                                                           out[2], zseg);
}
template <typename T, int PASSES, bool HJ>
void run_source1(const Geo &g, const Coef<T> &c, const T *const B[3], const T *const J[3], T *const out[3],
                 cudaStream_t s) {
    if (one_row(g)) run_source<T, PASSES, HJ, 1>(g, c, B, J, out, s);
    else run_source<T, PASSES, HJ, 4>(g, c, B, J, out, s);
}

template <typename T, bool UPD, int CR>
void run_sweep(const Geo &g, const Coef<T> &c, const T *const dEp[3], const T *const in[3], T *const out[3],
               cudaStream_t s) {
    constexpr size_t bytes = (size_t)SWEEP1_RS * 3 * cpl(CR) * sizeof(T);
    static const int res = resident(k3_sweep1<T, UPD, CR>, CNT, bytes);
    int zseg;
    const dim3 grid = grid_of(g, CX, CR * CW, res, &zseg, 0.6);
    k3_sweep1<T, UPD, CR><<<grid, CNT, bytes, s>>>(g, c, dEp[0], dEp[1], dEp[2], in[0], in[1], in[2], out[0], out[1],
                                                   out[2], zseg);
}
template <typename T, bool UPD>
void run_sweep1(const Geo &g, const Coef<T> &c, const T *const dEp[3], const T *const in[3], T *const out[3],
                cudaStream_t s) {
    if (one_row(g)) run_sweep<T, UPD, 1>(g, c, dEp, in, out, s);
    else run_sweep<T, UPD, 4>(g, c, dEp, in, out, s);
}

bool pair_path(const Geo &g, float *) { return g.nx % 2 == 0 && g.pitch % 2 == 0; }

Coef3P coef3p(const Coef<float> &c) {
    auto pr = [](float v) { return make_float2(v, v); };
    return Coef3P{pr(c.ax), pr(c.ay), pr(c.az), pr(c.ayz), pr(c.azx), pr(c.axy), pr(c.byz), pr(c.bzx), pr(c.bxy),
                  pr(c.c6), pr(c.kx), pr(c.ky), pr(c.kz), pr(c.q), pr(c.q * (1.f / 64.f))};
}

constexpr int SRC_RS = 4;  // source ring slots (six components: 65 KB)

template <int PASSES, bool HJ>
void run_source2(const Geo &g, const Coef<float> &c, const float *const B[3], const float *const J[3],
                 float *const out[3], cudaStream_t s) {
    constexpr int N = HJ ? 6 : 3;
    constexpr size_t bytes = (size_t)SRC_RS * N * PL2 * sizeof(float);
    static const int res = resident(k3_source2<SRC_RS, PASSES, HJ>, NTH, bytes);
    int zseg;
    const dim3 grid = grid_of(g, TX2, TY, res, &zseg);
    k3_source2<SRC_RS, PASSES, HJ><<<grid, dim3(TXP, TY), bytes, s>>>(
        g, coef3p(c), B[0], B[1], B[2], HJ ? J[0] : nullptr, HJ ? J[1] : nullptr, HJ ? J[2] : nullptr, out[0], out[1],
        out[2], zseg);
}
bool pair_path(const Geo &, double *) { return false; }

template <bool UPD, bool FIRST>
void run_sweep2(const Geo &g, const Coef<float> &c, const float *const dEp[3], const float *const in[3],
                float *const out[3], cudaStream_t s) {
    constexpr size_t bytes = (size_t)SWEEP_RS * 3 * PL2 * sizeof(float);
    static const int res = resident(k3_sweep2<UPD, FIRST>, NTH, bytes);
    const Coef3P cp = coef3p(c);
    int zseg;
    const dim3 grid = grid_of(g, TX2, TY, res, &zseg);
    k3_sweep2<UPD, FIRST><<<grid, dim3(TXP, TY), bytes, s>>>(g, cp, dEp[0], dEp[1], dEp[2], in[0], in[1], in[2], out[0],
                                                     out[1], out[2], zseg);
}

template <bool UPD>
void run_sweeps2f(const Geo &g, const Coef<float> &c, const float *const dEp[3], const float *const in[3],
                  float *const out[3], cudaStream_t s) {
    constexpr size_t bytes = ((size_t)FRS * 3 * FIPL + (size_t)2 * 3 * FAPL) * sizeof(float);
    static const int res = resident(k3_sweeps2f<UPD>, FNT, bytes);
    int zseg;
    const dim3 grid = grid_of(g, TX2, TY, res, &zseg);
    k3_sweeps2f<UPD><<<grid, FNT, bytes, s>>>(g, coef3p(c), dEp[0], dEp[1], dEp[2], in[0], in[1], in[2], out[0],
                                             out[1], out[2], zseg);
}

template <typename T>
int launch_march3d_sweeps2(const Geo &g, const Coef<T> &c, const T *const dEp[3], const T *const in[3],
                           T *const out[3], cudaStream_t s, bool update) {
    if constexpr (std::is_same<T, float>::value) {
        if (pair_path(g, (float *)nullptr)) {
            if (update) run_sweeps2f<true>(g, c, dEp, in, out, s);
            else run_sweeps2f<false>(g, c, dEp, in, out, s);
            return 1;
        }
    }
    return 0;  // FP64 or odd n_x: the caller runs the sweeps one per pass
}

template <typename T>
int launch_march3d_source(const Geo &g, const Coef<T> &c, const T *const B[3], const T *const J[3], int passes,
                          T *const out[3], cudaStream_t s) {
    if constexpr (std::is_same<T, float>::value) {
        if (pair_path(g, (float *)nullptr)) {
            if (!J || !J[0]) run_source2<0, false>(g, c, B, J, out, s);
            else if (passes == 1) run_source2<1, true>(g, c, B, J, out, s);
            else run_source2<0, true>(g, c, B, J, out, s);
            return 1;
        }
    }
    if (!J || !J[0]) run_source1<T, 0, false>(g, c, B, J, out, s);
    else if (passes == 1) run_source1<T, 1, true>(g, c, B, J, out, s);
    else run_source1<T, 0, true>(g, c, B, J, out, s);
    return 1;
}

template <typename T>
int launch_march3d_faraday(const Geo &g, const Coef<T> &c, const T *const E[3], T *const B[3], cudaStream_t s) {
    if constexpr (std::is_same<T, float>::value) {
        if (pair_path(g, (float *)nullptr)) {
            constexpr size_t bytes = (size_t)FAR_RS * 3 * PL2 * sizeof(float);
            static const int res = resident(k3_faraday2, NTH, bytes);
            int zseg;
            const dim3 grid = grid_of(g, TX2, TY, res, &zseg);
            k3_faraday2<<<grid, dim3(TXP, TY), bytes, s>>>(g, coef3p(c), E[0], E[1], E[2], B[0], B[1], B[2], zseg);
            return 1;
        }
    }
    int zseg;
    const dim3 grid = grid_of(g, 32, 8, 8, &zseg);
    k3_faraday1<T><<<grid, 256, 0, s>>>(g, c, E[0], E[1], E[2], B[0], B[1], B[2], zseg);
    return 1;
}

template <typename T>
int launch_march3d_sweep(const Geo &g, const Coef<T> &c, const T *const dEp[3], const T *const in[3], T *const out[3],
                         cudaStream_t s, bool update) {
    if constexpr (std::is_same<T, float>::value) {
        if (pair_path(g, (float *)nullptr)) {
            const bool first = in[0] == dEp[0] && in[1] == dEp[1] && in[2] == dEp[2];
            if (update) first ? run_sweep2<true, true>(g, c, dEp, in, out, s) : run_sweep2<true, false>(g, c, dEp, in, out, s);
            else first ? run_sweep2<false, true>(g, c, dEp, in, out, s) : run_sweep2<false, false>(g, c, dEp, in, out, s);
            return 1;
        }
    }
    if (update) run_sweep1<T, true>(g, c, dEp, in, out, s);
    else run_sweep1<T, false>(g, c, dEp, in, out, s);
    return 1;
}

#define FMX_M3_INST(T)                                                                                           \
    template int launch_march3d_source<T>(const Geo &, const Coef<T> &, const T *const[3], const T *const[3], int, \
                                          T *const[3], cudaStream_t);                                           \
    template int launch_march3d_sweep<T>(const Geo &, const Coef<T> &, const T *const[3], const T *const[3],       \
                                         T *const[3], cudaStream_t, bool);                                        \
    template int launch_march3d_faraday<T>(const Geo &, const Coef<T> &, const T *const[3], T *const[3], cudaStream_t); \
    template int launch_march3d_sweeps2<T>(const Geo &, const Coef<T> &, const T *const[3], const T *const[3],    \
                                           T *const[3], cudaStream_t, bool);
FMX_M3_INST(float)
FMX_M3_INST(double)
#undef FMX_M3_INST

}  // namespace fmx
