// FP64 diagnostics of a state (E^n, B^{n+1/2}):
//   energy of the converged scheme  sum[E.(1-A)E + B^{n-1/2}.S B^{n+1/2}]
//     with B^{n-1/2} = B^{n+1/2} + c dt curl E^n and S = diag(alpha_x,
//     alpha_y, alpha_z) (derived from the symmetry of A and S; the paper
//     does not define a discrete energy);
//   plain sum (E^2 + B^2);
//   D.B at cell centres (Eq. gauss_B);
//   D_x(alpha_yz Ex) + D_y(alpha_zx Ey) + D_z(alpha_xy Ez) at nodes
//     (left-hand side of Eq. gauss_E).
// Every cell's terms are evaluated in FP64 from the stored precision; block
// partials are combined by a single-block kernel in a fixed order.
#include <cuda_runtime.h>

#include "fmx_internal.h"
#include "stencil.cuh"

namespace fmx {
namespace {

constexpr int BX = 32, BY = 8, NT = BX * BY, NQ = 6;

// Sum of each quantity over the block (maximum for 2 and 4), all threads
// call; the first NQ threads write it to the block's partials.
__device__ __forceinline__ void block_partials(const double v[NQ], int t, double *out) {
    __shared__ double red[NQ][NT / 32];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        double x = v[q];
        const bool mx = q == 2 || q == 4;
        for (int o = 16; o > 0; o >>= 1) {
            double y = __shfl_down_sync(0xffffffffu, x, o);
            x = mx ? fmax(x, y) : x + y;
        }
        if ((t & 31) == 0) red[q][t >> 5] = x;
    }
    __syncthreads();
    if (t < NQ) {
        const bool mx = t == 2 || t == 4;
        double x = 0.0;
        for (int w = 0; w < NT / 32; ++w) x = mx ? fmax(x, red[t][w]) : x + red[t][w];
        out[t] = x;
    }
}

// 2D.  FP64 arithmetic bounds the diagnostics of FP32 and FP64 grids alike (it
// runs at 1/64 of the FP32 rate on this part), so the kernel is written for
// the fewest FP64 operations, conversions included.  The energy is summed by
// parts on the periodic lattice,
//   sum E.A E = -a_x S[(Dx Ey)^2 + (Dx Ez)^2] - a_y S[(Dy Ex)^2 + (Dy Ez)^2]
//               + a_xy S[(Dx Dy Ez)^2] - 2 b_xy S[ux uy],
// ux = Dx(bwd) Ex, uy = Dy(bwd) Ey, which also give the node divergence
// alpha_y ux + alpha_x uy; the coefficients multiply once per thread.  A warp
// takes 30 columns (its edge lanes are the neighbours) and walks up a strip of
// rows, each value loaded and converted once, x-neighbours by shuffle: 57
// operations per cell against 154 for the stencils evaluated cell by cell.
// 1536 x 1200 FP32: 234 us against 557, the final sum 6 us against 28.
constexpr int DW = 30;  // columns a warp accounts for

// m = max(m, |v|) on the bit patterns, which order non-negative doubles as
// integers do (no FP64 operation); as fmax, a NaN leaves m
__device__ __forceinline__ void max_abs(long long &m, double v) {
    const long long b = __double_as_longlong(v) & 0x7fffffffffffffffLL;
    if (b > m && b <= 0x7ff0000000000000LL) m = b;
}

template <typename T>
__global__ void __launch_bounds__(NT) k_diag2(Geo g, Coef<double> c, double idx_, double idy_,
                                              const T *__restrict__ e0, const T *__restrict__ e1,
                                              const T *__restrict__ e2, const T *__restrict__ b0,
                                              const T *__restrict__ b1, const T *__restrict__ b2, int nstrip, int L,
                                              double *partials) {
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
    const int strip = (int)(w % nstrip), seg = (int)(w / nstrip);
    const int y0 = seg * L, y1 = min(y0 + L, g.ny);
    double v[NQ] = {0, 0, 0, 0, 0, 0};
    if (y0 < g.ny) {
        const int x = strip * DW - 1 + lane;
        const bool own = lane >= 1 && lane <= DW && x < g.nx;
        const int xc = ((x % g.nx) + g.nx) % g.nx;
        auto at = [&](const T *p, int y) {
            const int yc = y < 0 ? y + g.ny : (y >= g.ny ? y - g.ny : y);
            return (double)p[(int64_t)yc * g.pitch + xc];
        };
        auto lft = [](double a) { return __shfl_up_sync(0xffffffffu, a, 1); };
        auto rgt = [](double a) { return __shfl_down_sync(0xffffffffu, a, 1); };
        double ex = at(e0, y0), ey = at(e1, y0), ez = at(e2, y0), by = at(b1, y0);
        double eym = at(e1, y0 - 1), bym = at(b1, y0 - 1);
        const double exm = at(e0, y0 - 1);
        double uxm = exm - lft(exm), ux = ex - lft(ex), dxez = rgt(ez) - ez;
        double sE = 0, sB = 0, sx = 0, sy = 0, sxy = 0, sb = 0, sw = 0, sd = 0, sg = 0;
        long long md = 0, mg = 0;
        for (int y = y0; y < y1; ++y) {
            const double exp_ = at(e0, y + 1), eyp = at(e1, y + 1), ezp = at(e2, y + 1), byp = at(b1, y + 1);
            const double bx = at(b0, y), bz = at(b2, y);
            const double uxp = exp_ - lft(exp_), uy = ey - eym, dxezp = rgt(ezp) - ezp;
            const double dyex = exp_ - ex, dxey = rgt(ey) - ey, dyez = ezp - ez, dxyez = dxezp - dxez;
            const double bxl = lft(bx), bxr = rgt(bx), uyl = lft(uy), uyr = rgt(uy);
            if (own) {
                sE += ex * ex;
                sE += ey * ey;
                sE += ez * ez;
                sx += dxey * dxey;
                sx += dxez * dxez;
                sy += dyex * dyex;
                sy += dyez * dyez;
                sxy += dxyez * dxyez;
                sb += ux * uy;
                // (B + c dt curl E) . S B
                const double ax = bx + c.c6 * ((bxl + bxr) - 2.0 * bx), ay = by + c.c6 * ((bym + byp) - 2.0 * by);
                sw += (bx + c.ky * dyez) * ax;
                sw += (by - c.kx * dxez) * ay;
                sw += ((bz + c.kx * dxey) - c.ky * dyex) * bz;
                sB += bx * bx;
                sB += by * by;
                sB += bz * bz;
                const double div = (bxr - bx) * idx_ + (byp - by) * idy_;
                const double ga = (ux + c.c6 * ((uxm + uxp) - 2.0 * ux)) * idx_ + (uy + c.c6 * ((uyl + uyr) - 2.0 * uy)) * idy_;
                sd += div * div;
                sg += ga * ga;
                max_abs(md, div);
                max_abs(mg, ga);
            }
            ex = exp_, eym = ey, ey = eyp, ez = ezp, dxez = dxezp, uxm = ux, ux = uxp, bym = by, by = byp;
        }
        v[0] = sE + (c.ax * sx + c.ay * sy - c.axy * sxy + 2.0 * c.bxy * sb) + sw;
        v[1] = sE + sB;
        v[2] = __longlong_as_double(md);
        v[3] = sd;
        v[4] = __longlong_as_double(mg);
        v[5] = sg;
    }
    block_partials(v, threadIdx.x, partials + (int64_t)blockIdx.x * NQ);
}

// 3D, by the same sums by parts: for the diagonal blocks
//   sum E_a A_aa E_a = -a_b S[(D_b E_a)^2] - a_c S[(D_c E_a)^2] + a_bc S[(D_b D_c E_a)^2]
// and for each pair (a, b), c the third axis,
//   2 sum E_a A_ab E_b = -2 b_ab (S[u_a u_b] - 1/6 S[(D_c u_a)(D_c u_b)]),
// u_a = D_a(bwd) E_a at the nodes, whose averages also give the node divergence.
// A warp takes 30 columns of one row and walks up the planes: 88 operations and
// 13 conversions per cell.  160 x 150 x 128 FP32: the whole call 0.84 ms against 2.28.
template <typename T>
__global__ void __launch_bounds__(NT, 2) k_diag3(Geo g, Coef<double> c, double idx_, double idy_, double idz_,
                                              const T *__restrict__ e0, const T *__restrict__ e1,
                                              const T *__restrict__ e2, const T *__restrict__ b0,
                                              const T *__restrict__ b1, const T *__restrict__ b2, int nstrip, int L,
                                              double *partials) {
    const int lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
    const int strip = (int)(w % nstrip);
    const int y = (int)((w / nstrip) % g.ny), z0 = (int)(w / nstrip / g.ny) * L, z1 = min(z0 + L, g.nz);
    double v[NQ] = {0, 0, 0, 0, 0, 0};
    if (z0 < g.nz) {
        const int x = strip * DW - 1 + lane;
        const bool own = lane >= 1 && lane <= DW && x < g.nx;
        const int xc = ((x % g.nx) + g.nx) % g.nx;
        const int64_t oc = (int64_t)y * g.pitch + xc;
        const int64_t om = (int64_t)(y > 0 ? y - 1 : g.ny - 1) * g.pitch + xc;
        const int64_t op = (int64_t)(y + 1 < g.ny ? y + 1 : 0) * g.pitch + xc;
        auto lft = [](double a) { return __shfl_up_sync(0xffffffffu, a, 1); };
        auto rgt = [](double a) { return __shfl_down_sync(0xffffffffu, a, 1); };
        auto alpha = [&](double m, double o, double p) { return o + c.c6 * ((m + p) - 2.0 * o); };
        int64_t zp = (int64_t)(z0 > 0 ? z0 - 1 : g.nz - 1) * g.plane, zc = (int64_t)z0 * g.plane;
        // plane below: E_z for u_z, B_z, and q (the x and y parts of the node divergence)
        double ezm = e2[zp + om], ez = e2[zp + oc], ezp = e2[zp + op], bzb = b2[zp + oc];
        auto node_xy = [&](double uxm, double ux, double uxp, double uy) {
            return alpha(uxm, ux, uxp) * idx_ + alpha(lft(uy), uy, rgt(uy)) * idy_;
        };
        double q0, q1, uxm, ux, uxp, uy, ex, exp_, ey, uzm, uz, uzp, bz;
        {
            const double a = e0[zp + om], b = e0[zp + oc], d = e0[zp + op];
            q0 = node_xy(a - lft(a), b - lft(b), d - lft(d), (double)e1[zp + oc] - (double)e1[zp + om]);
        }
        {
            const double a = e0[zc + om];
            ex = e0[zc + oc];
            exp_ = e0[zc + op];
            ey = e1[zc + oc];
            uxm = a - lft(a);
            ux = ex - lft(ex);
            uxp = exp_ - lft(exp_);
            uy = ey - (double)e1[zc + om];
            q1 = node_xy(uxm, ux, uxp, uy);
            const double fm = e2[zc + om], f = e2[zc + oc], fp = e2[zc + op];
            uzm = fm - ezm;
            uz = f - ez;
            uzp = fp - ezp;
            ezm = fm, ez = f, ezp = fp;
            bz = b2[zc + oc];
        }
        double dyex = exp_ - ex, dxey = rgt(ey) - ey;
        double sE = 0, sB = 0, sx = 0, sy = 0, sz = 0, syz = 0, szx = 0, sxy = 0, sbx = 0, sby = 0, sbz = 0, sw = 0, sd = 0,
               sg = 0;
        long long md = 0, mg = 0;
        for (int k = z0; k < z1; ++k) {
            const int64_t zn = k + 1 < g.nz ? zc + g.plane : 0;
            const double exmn = e0[zn + om], exn = e0[zn + oc], expn = e0[zn + op];
            const double eymn = e1[zn + om], eyn = e1[zn + oc];
            const double ezmn = e2[zn + om], ezn = e2[zn + oc], ezpn = e2[zn + op];
            const double bx = b0[zc + oc], bym = b1[zc + om], by = b1[zc + oc], byp = b1[zc + op], bzn = b2[zn + oc];
            const double uxmn = exmn - lft(exmn), uxn = exn - lft(exn), uxpn = expn - lft(expn), uyn = eyn - eymn;
            const double q2 = node_xy(uxmn, uxn, uxpn, uyn);
            const double dyexn = expn - exn, dzex = exn - ex, dxeyn = rgt(eyn) - eyn, dzey = eyn - ey;
            const double dxez = rgt(ez) - ez, dyez = ezp - ez, dxezp = rgt(ezp) - ezp;
            const double uyr = rgt(uy), uzr = rgt(uz), ay_uz = alpha(uzm, uz, uzp);
            const double uzl_a = lft(ay_uz), uzr_a = rgt(ay_uz), bxl = lft(bx), bxr = rgt(bx);
            if (own) {
                sE += ex * ex;
                sE += ey * ey;
                sE += ez * ez;
                sy += dyex * dyex;
                sz += dzex * dzex;
                sx += dxey * dxey;
                sz += dzey * dzey;
                sx += dxez * dxez;
                sy += dyez * dyez;
                const double dyzex = dyexn - dyex, dxzey = dxeyn - dxey, dxyez = dxezp - dxez;
                syz += dyzex * dyzex;
                szx += dxzey * dxzey;
                sxy += dxyez * dxyez;
                // pairs (x, y), (y, z), (z, x): u_a u_b - (1/6) D_c u_a D_c u_b
                sbz += ux * uy;
                sbz -= (c.c6 * (uxn - ux)) * (uyn - uy);
                sbx += uy * uz;
                sbx -= (c.c6 * (uyr - uy)) * (uzr - uz);
                sby += uz * ux;
                sby -= (c.c6 * (uzp - uz)) * (uxp - ux);
                sw += ((bx + c.ky * dyez) - c.kz * dzey) * alpha(bxl, bx, bxr);
                sw += ((by + c.kz * dzex) - c.kx * dxez) * alpha(bym, by, byp);
                sw += ((bz + c.kx * dxey) - c.ky * dyex) * alpha(bzb, bz, bzn);
                sB += bx * bx;
                sB += by * by;
                sB += bz * bz;
                const double div = ((bxr - bx) * idx_ + (byp - by) * idy_) + (bzn - bz) * idz_;
                const double ga = alpha(q0, q1, q2) + alpha(uzl_a, ay_uz, uzr_a) * idz_;
                sd += div * div;
                sg += ga * ga;
                max_abs(md, div);
                max_abs(mg, ga);
            }
            uxm = uxmn, ux = uxn, uxp = uxpn, uy = uyn, ex = exn, ey = eyn, dyex = dyexn, dxey = dxeyn;
            uzm = ezmn - ezm, uz = ezn - ez, uzp = ezpn - ezp;
            ezm = ezmn, ez = ezn, ezp = ezpn;
            bzb = bz, bz = bzn, q0 = q1, q1 = q2;
            zc = zn;
        }
        v[0] = sE + (c.ax * sx + c.ay * sy + c.az * sz - (c.ayz * syz + c.azx * szx + c.axy * sxy) +
                     2.0 * (c.byz * sbx + c.bzx * sby + c.bxy * sbz)) + sw;
        v[1] = sE + sB;
        v[2] = __longlong_as_double(md);
        v[3] = sd;
        v[4] = __longlong_as_double(mg);
        v[5] = sg;
    }
    block_partials(v, threadIdx.x, partials + (int64_t)blockIdx.x * NQ);
}

// One thread per cell: 1D, and 3D grids of one plane that the strips do not fit
template <typename T, int DIM>
__global__ void k_diag(Geo g, Coef<double> c, double idx_, double idy_, double idz_, const T *e0, const T *e1,
                       const T *e2, const T *b0, const T *b1, const T *b2, double *partials) {
    Pos p;
    p.i = blockIdx.x * BX + threadIdx.x;
    p.j = blockIdx.y * BY + threadIdx.y;
    p.k = blockIdx.z;
    const bool in = p.i < g.nx && p.j < g.ny;
    double v[NQ] = {0, 0, 0, 0, 0, 0};
    if (in) {
        Field<T, double> E[3] = {{e0, g}, {e1, g}, {e2, g}};
        Field<T, double> B[3] = {{b0, g}, {b1, g}, {b2, g}};
        const double inv_d[3] = {idx_, idy_, idz_};
        const int o0[3] = {0, 0, 0};
        double ae[3] = {apply_a<double, DIM, 0>(E, p, c), apply_a<double, DIM, 1>(E, p, c),
                        apply_a<double, DIM, 2>(E, p, c)};
        double ce[3] = {curl_e<double, DIM, 0>(E, p, c), curl_e<double, DIM, 1>(E, p, c),
                        curl_e<double, DIM, 2>(E, p, c)};
        double ws = 0.0, wp = 0.0, div = 0.0, gs = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double ea = E[a](p, 0, 0, 0), ba = B[a](p, 0, 0, 0);
            double sb = ba;
            if (a < DIM) sb += c.c6 * d2<double>(B[a], p, o0, a);
            ws += ea * (ea - ae[a]) + (ba + ce[a]) * sb;
            wp += ea * ea + ba * ba;
            if (a < DIM) div += (at_sh(B[a], p, o0, a, 1) - ba) * inv_d[a];
        }
        // node divergence of alpha_bc E_a, backward along a
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const int b = (a + 1) % 3, cc = (a + 2) % 3;
            double val[2];
            for (int s = 0; s < 2; ++s) {
                int o[3] = {0, 0, 0};
                o[a] = -s;
                // alpha_c (alpha_b E_a) at o
                double w[3];
                for (int t = -1; t <= 1; ++t) {
                    int q[3] = {o[0], o[1], o[2]};
                    if (cc < DIM) q[cc] += t;
                    else if (t != 0) { w[t + 1] = 0.0; continue; }
                    double u = E[a](p, q[0], q[1], q[2]);
                    if (b < DIM) u += c.c6 * d2<double>(E[a], p, q, b);
                    w[t + 1] = u;
                }
                val[s] = cc < DIM ? w[1] + c.c6 * (w[2] - 2.0 * w[1] + w[0]) : w[1];
            }
            gs += (val[0] - val[1]) * inv_d[a];
        }
        v[0] = ws;
        v[1] = wp;
        v[2] = fabs(div);
        v[3] = div * div;
        v[4] = fabs(gs);
        v[5] = gs * gs;
    }
    const int64_t slot = (int64_t)blockIdx.x + (int64_t)gridDim.x * ((int64_t)blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
    block_partials(v, threadIdx.y * BX + threadIdx.x, partials + slot * NQ);
}

__global__ void k_diag_final(const double *partials, int64_t nslots, double *out) {
    __shared__ double red[NQ][32];
    double v[NQ] = {0, 0, 0, 0, 0, 0};
    for (int64_t s = threadIdx.x; s < nslots; s += blockDim.x)
        for (int q = 0; q < NQ; ++q) {
            double x = partials[s * NQ + q];
            v[q] = (q == 2 || q == 4) ? fmax(v[q], x) : v[q] + x;
        }
    for (int q = 0; q < NQ; ++q) {
        double x = v[q];
        const bool mx = q == 2 || q == 4;
        for (int o = 16; o > 0; o >>= 1) {
            double y = __shfl_down_sync(0xffffffffu, x, o);
            x = mx ? fmax(x, y) : x + y;
        }
        if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = x;
    }
    __syncthreads();
    if (threadIdx.x < NQ) {
        const int q = threadIdx.x;
        const bool mx = q == 2 || q == 4;
        double x = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) x = mx ? fmax(x, red[q][w]) : x + red[q][w];
        out[q] = x;
    }
}

}  // namespace

template <typename T>
int launch_diagnostics(const Geo &g, int dims, const Coef<double> &c, const double d[3], T *const E[3],
                       T *const B[3], double *partials, int64_t nparts, double *out_dev, cudaStream_t s) {
    dim3 grid((g.nx + BX - 1) / BX, (g.ny + BY - 1) / BY, g.nz);
    int64_t nslots = (int64_t)grid.x * grid.y * grid.z;
    if (nslots * NQ > nparts) return -1;
    const double ix = 1.0 / d[0], iy = 1.0 / d[1], iz = 1.0 / d[2];
    if (dims > 1) {
        // strips of 30 columns, segments of 1 to 64 rows (2D) or planes (3D), the
        // height at which the fullest SM has the least to do (the first row of a
        // segment costs about one row more).  On grids that leave SMs free the lowest
        // that the partial sums' array holds: a warp's rows follow one another
        const int nstrip = (g.nx + DW - 1) / DW, len = dims == 3 ? g.nz : g.ny;
        const int64_t lines = (int64_t)nstrip * (dims == 3 ? g.ny : 1);
        static const int sms = [] {
            int dev = 0, v = 0;
            cudaGetDevice(&dev);
            return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 1;
        }();
        int64_t L = 6, blocks = 0;
        double least = 1e300;
        for (int64_t h = 1; h <= 64; ++h) {
            const int64_t nb = (lines * ((len + h - 1) / h) + NT / 32 - 1) / (NT / 32);
            if (nb * NQ > nparts) continue;
            const double cost = (double)((nb + sms - 1) / sms) * (double)(h + 1);
            if (cost < least) {
                least = cost;
                L = h;
                blocks = nb;
            }
        }
        if (blocks > 2147483647LL) return -1;
        if (blocks == 0) {
            // no height's partial sums fit the array, which holds one slot per block
            // of 32 x 8 cells: 3D grids of one plane (one thread per cell there)
            if (dims != 3) return -1;
            k_diag<T, 3><<<grid, dim3(BX, BY), 0, s>>>(g, c, ix, iy, iz, E[0], E[1], E[2], B[0], B[1], B[2], partials);
            blocks = nslots;
        } else if (dims == 3)
            k_diag3<T><<<(unsigned)blocks, NT, 0, s>>>(g, c, ix, iy, iz, E[0], E[1], E[2], B[0], B[1], B[2], nstrip,
                                                       (int)L, partials);
        else
            k_diag2<T><<<(unsigned)blocks, NT, 0, s>>>(g, c, ix, iy, E[0], E[1], E[2], B[0], B[1], B[2], nstrip, (int)L,
                                                       partials);
        nslots = blocks;
    } else {
        k_diag<T, 1><<<grid, dim3(BX, BY), 0, s>>>(g, c, ix, iy, iz, E[0], E[1], E[2], B[0], B[1], B[2], partials);
    }
    // the final sum costs FP64 shuffles per warp: few warps for few slots
    const int fin = nslots <= 2048 ? 128 : 1024;
    k_diag_final<<<1, fin, 0, s>>>(partials, nslots, out_dev);
    return 2;
}

template int launch_diagnostics<float>(const Geo &, int, const Coef<double> &, const double[3], float *const[3],
                                       float *const[3], double *, int64_t, double *, cudaStream_t);
template int launch_diagnostics<double>(const Geo &, int, const Coef<double> &, const double[3], double *const[3],
                                        double *const[3], double *, int64_t, double *, cudaStream_t);

}  // namespace fmx
