// Resident engine: every step of an fmx_step call -- current filter, source,
// the whole solve of Algorithm 1 (fixed m or to the residual stop), E update
// and Faraday -- in ONE launch, for grids small enough to live in L2 (the
// latency-bound case: a 64 x 64 FP64 grid has 4096 cells, far too few to fill
// the GPU, and one host read-back per step cost more than the step).
//
// The launch is one thread-block cluster (16 CTAs where the device schedules
// clusters of 16, else 8, one CTA per SM) or, where the arithmetic needs more
// SMs (FP64 runs at 1/64 of the FP32 rate on this class of part), up to 8 clusters
// in one cooperative launch (every CTA co-resident; clusters_for has the sizes).
// Each CTA owns a contiguous
// range of cells (linear index, x fastest).  Phases are separated by
//   - one cluster: the cluster's hardware barrier (barrier.cluster
//     arrive.release / wait.acquire);
//   - several clusters: a cluster barrier, then the cluster's leader thread
//     arrives at a grid barrier in global memory (an atomic arrival count and
//     a generation the last arrival advances with release semantics) and
//     waits for the generation to move with a bounded spin (a limit in SM
//     clock cycles, FMX_ETIMEOUT latched in the status word when it runs out,
//     a wait that gives up as soon as another cluster has), then a second
//     cluster barrier releases the cluster with the leader's verdict.
// Field data other CTAs wrote is read through L2 (ld.global.cg).  The
// residual of a sweep is reduced in FP64 by one warp of each CTA in a fixed order
// (launch_sum): its CTA's values, which it writes into every CTA of the cluster
// (distributed shared memory), then the cluster's; with several clusters each
// leader publishes its cluster's sum, and the warp adds those after the grid
// barrier.  All threads therefore hold bit-identical norms and take the same
// stop decision: control flow stays uniform and every barrier is reached by
// every thread (or every wait gives up within its limit).
//
// Arithmetic per cell is the staged engine's (stencil.cuh): source Eqs.
// ampere_aux_x..z, A of Eqs. matrixA_1st..matrixA_last, Algorithm 1, Eqs.
// faraday_x..z; residual ||dE_(s+1) - dE_(s)||_2 <= tol ||dE'||_2 with at
// least one sweep, none when dE' = 0, FMX_ENOCONV past m_max.
//
// Phase order of one step n (the E update of step n-1 is folded into step
// n's source phase: the source reads only B):
//   S  : E += dE_(n-1) (own cells; n > 0), dE' = c dt curl(alpha B) - q j_f,
//        ||dE'||^2                                                    | barrier
//   W_s: dE_(s+1) = dE' + A dE_(s), ||dE_(s+1) - dE_(s)||^2          | barrier
//   F  : B -= c dt curl(E + dE) (E^{n+1} formed on the fly)          | barrier
// and after the last step one more E += dE.  The current is filtered once per
// launch into the jf workspace (it is constant over the launch).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "fmx_internal.h"
#include "stencil.cuh"

namespace cg = cooperative_groups;

namespace fmx {
namespace {

constexpr int kNT = 256;         // threads per CTA
constexpr int kMaxCluster = 16;  // CTAs per cluster
constexpr int kMaxClusters = 8;  // clusters per launch (DevStatus::xpart)

// value at a periodic shift, read through L2
template <typename T>
struct FieldL2 {
    const T *__restrict__ p;
    Geo g;
    __device__ __forceinline__ T operator()(Pos b, int dx, int dy, int dz) const {
        int x = wrapc(b.i + dx, g.nx), y = wrapc(b.j + dy, g.ny), z = wrapc(b.k + dz, g.nz);
        return __ldcg(p + (int64_t)z * g.plane + (int64_t)y * g.pitch + x);
    }
};

// E^{n+1} = E^n + dE at a periodic shift, rounded to T as the staged update stores it
template <typename T>
struct SumL2 {
    const T *__restrict__ e;
    const T *__restrict__ d;
    Geo g;
    __device__ __forceinline__ T operator()(Pos b, int dx, int dy, int dz) const {
        int x = wrapc(b.i + dx, g.nx), y = wrapc(b.j + dy, g.ny), z = wrapc(b.k + dz, g.nz);
        const int64_t o = (int64_t)z * g.plane + (int64_t)y * g.pitch + x;
        return __ldcg(e + o) + __ldcg(d + o);
    }
};

struct Cells {
    int lo, hi;  // linear cell range of this CTA
    Geo g;
    __device__ __forceinline__ void at(int q, Pos &p, int64_t &idx) const {
        p.i = q % g.nx;
        const int r = q / g.nx;
        p.j = r % g.ny;
        p.k = r / g.ny;
        idx = (int64_t)p.k * g.plane + (int64_t)p.j * g.pitch + p.i;
    }
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_relaxed_gpu(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The phase barrier of a launch (see the file comment).  Every thread calls
// barrier(); it returns false once the launch has given up (a grid wait ran
// out), after which every thread leaves its loops.
struct Sync {
    cg::cluster_group cl;
    DevStatus *st;
    int ncl, cid, crank;
    long long limit;  // SM clock cycles a leader waits at the grid barrier
    int lost;         // self-test: the grid barrier expects one arrival more than come
    int *abort_s;     // this CTA's copy of the leader's verdict (shared memory)

    __device__ bool grid() const { return ncl > 1 || lost; }

    // the leader's arrival and bounded wait at the grid barrier: 1 when every
    // cluster arrived, 0 when the wait ran out or another cluster gave up
    __device__ int grid_wait() const {
        const unsigned target = (unsigned)(ncl + lost);
        const unsigned g0 = ld_acquire_gpu(&st->bar_gen);
        __threadfence();
        const unsigned arrived = atomicAdd(&st->bar_count, 1u) + 1u;
        if (arrived == target) {
            atomicExch(&st->bar_count, 0u);
            __threadfence();
            st_release_gpu(&st->bar_gen, g0 + 1u);
            return 1;
        }
        const long long t0 = clock64();
        while (ld_acquire_gpu(&st->bar_gen) == g0) {
            if (ld_relaxed_gpu(&st->err) != 0) return 0;
            if (clock64() - t0 > limit) {
                atomicCAS(&st->err, 0, (int)FMX_ETIMEOUT);
                return 0;
            }
            __nanosleep(64);
        }
        return 1;
    }

    __device__ bool barrier() const {
        if (!grid()) {
            cl.sync();
            return true;
        }
        __threadfence();
        cl.sync();  // the cluster's phase is done
        if (crank == 0 && threadIdx.x == 0) {
            const int verdict = grid_wait() ? 0 : 1;
            for (int r = 0; r < (int)cl.num_blocks(); ++r) *cl.map_shared_rank(abort_s, r) = verdict;
        }
        cl.sync();  // every cluster's phase is done (or the launch gave up)
        return *abort_s == 0;
    }
};

// Launch-wide FP64 sum of v (every thread calls it and gets the same value,
// or ok = false when the launch gave up).  FP64 adds are the scarce resource
// (1/64 of the FP32 rate, tens of cycles each), so one warp does them: the
// threads' values go to shared memory, the first warp adds eight per lane and
// then across its lanes, its lanes write the CTA's partial into every CTA of
// the cluster, and after the barrier it adds the cluster's partials and hands
// the sum to the CTA.  (All warps reducing by shuffles and every thread adding
// the 16 partials took 1.3 us of a phase of 7.6 us at 64^2 FP64.)  xs: this
// CTA's [2][kMaxCluster] partial slots, alternated by `par` so that the next
// reduction never overwrites slots (or DevStatus::xpart entries) a slower CTA
// still reads.
struct SumSmem {
    double v[kNT];
    double xs[2 * kMaxCluster];
    double tot;
};
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double launch_sum(const Sync &S, double v, SumSmem &sm, int par, bool &ok) {
    const int t = threadIdx.x, lane = t & 31;
    const int C = (int)S.cl.num_blocks();
    sm.v[t] = v;
    __syncthreads();
    if (t < 32) {
        double s = (sm.v[t] + sm.v[t + 32]) + (sm.v[t + 64] + sm.v[t + 96]);
        s += (sm.v[t + 128] + sm.v[t + 160]) + (sm.v[t + 192] + sm.v[t + 224]);
        static_assert(kNT == 256, "eight values per lane");
        s = warp_sum(s);
        if (lane < C) S.cl.map_shared_rank(sm.xs + par * kMaxCluster, lane)[S.crank] = s;
    }
    S.cl.sync();
    if (t < 32) {
        const double tot = warp_sum(lane < C ? sm.xs[par * kMaxCluster + lane] : 0.0);
        if (t == 0) {
            sm.tot = tot;
            if (S.grid() && S.crank == 0) __stcg(&S.st->xpart[par][S.cid], tot);
        }
    }
    if (S.grid()) {
        ok = S.barrier();
        if (!ok) return 0.0;
        if (t < 32) {
            const double all = warp_sum(lane < S.ncl ? __ldcg(&S.st->xpart[par][lane]) : 0.0);
            if (t == 0) sm.tot = all;
        }
    }
    __syncthreads();
    ok = true;
    return sm.tot;
}

// (A dE) of a cell in 2D: apply_a (stencil.cuh) with each difference formed
// once, 23 operations instead of about 33.  at(k, dx, dy): component k at a
// neighbour; own receives the cell's own values.
template <typename T, typename F>
__device__ __forceinline__ void apply_a_2d(const F &at, const Coef<T> &c, T own[3], T out[3]) {
    const T x = at(0, 0, 0), xu = at(0, 0, 1), xd = at(0, 0, -1), xl = at(0, -1, 0), xlu = at(0, -1, 1);
    const T y = at(1, 0, 0), yl = at(1, -1, 0), yr = at(1, 1, 0), yd = at(1, 0, -1), yrd = at(1, 1, -1);
    const T z = at(2, 0, 0), zl = at(2, -1, 0), zr = at(2, 1, 0), zu = at(2, 0, 1), zd = at(2, 0, -1);
    const T zlu = at(2, -1, 1), zru = at(2, 1, 1), zld = at(2, -1, -1), zrd = at(2, 1, -1);
    own[0] = x;
    own[1] = y;
    own[2] = z;
    out[0] = c.ay * ((xu + xd) - T(2) * x) + c.bxy * ((yr - y) - (yrd - yd));
    out[1] = c.ax * ((yl + yr) - T(2) * y) + c.bxy * ((xu - xlu) - (x - xl));
    const T d0 = (zl + zr) - T(2) * z, du = (zlu + zru) - T(2) * zu, dd = (zld + zrd) - T(2) * zd;
    out[2] = (c.ax - T(2) * c.axy) * d0 + c.ay * ((zu + zd) - T(2) * z) + c.axy * (du + dd);
}

template <typename T>
struct ResidentArgs {
    StagedPtrs<T> P;   // E, B in place; J raw; jf, tmp, dEp, dEa, dEb workspace
    Coef<T> c;
    int nsteps;
    int resid;         // 1: Algorithm 1 to the residual stop; 0: m sweeps
    int m, m_max;
    double tol2;
    int jpasses;       // current filter passes per active axis (0: j used as is)
    int have_j;
    long long limit;   // grid-barrier wait limit, SM clock cycles
    int lost;          // self-test of the wait's time-out
};

template <typename T, int DIM>
__global__ void __launch_bounds__(kNT) k_resident(ResidentArgs<T> a, Geo g) {
    __shared__ SumSmem sums;
    __shared__ int abort_s;
    Sync S{cg::this_cluster(), a.P.st, 0, 0, 0, a.limit, a.lost, &abort_s};
    const int C = (int)S.cl.num_blocks();
    S.crank = (int)S.cl.block_rank();
    S.ncl = (int)(gridDim.x / C);
    S.cid = (int)(blockIdx.x / C);  // the clusters tile the 1D grid in order
    const int b = S.cid * C + S.crank, NB = S.ncl * C;
    const int64_t N = (int64_t)g.nx * g.ny * g.nz;
    Cells cells{(int)(N * b / NB), (int)(N * (b + 1) / NB), g};
    const int t = threadIdx.x;
    StagedPtrs<T> &P = a.P;
    const Coef<T> &c = a.c;
    int par = 0;
    bool ok = true;

    // the current: p binomial passes per active axis (axis order x, y, z, x, ...
    // as the staged filter), ping-ponging between tmp and jf so the last pass
    // lands in jf
    const T *jsrc[3] = {a.have_j ? P.J[0] : nullptr, a.have_j ? P.J[1] : nullptr, a.have_j ? P.J[2] : nullptr};
    if (a.have_j && a.jpasses > 0) {
        const int n = a.jpasses * DIM;
        for (int comp = 0; comp < 3 && ok; ++comp) {
            const T *src = P.J[comp];
            for (int q = 0; q < n && ok; ++q) {
                T *dst = ((n - 1 - q) % 2 == 0) ? P.jf[comp] : P.tmp;
                const int axis = q % DIM;
                FieldL2<T> f{src, g};
                int dx, dy, dz;
                unit(axis, 1, dx, dy, dz);
                for (int qq = cells.lo + t; qq < cells.hi; qq += kNT) {
                    Pos p;
                    int64_t idx;
                    cells.at(qq, p, idx);
                    dst[idx] = T(0.25) * f(p, -dx, -dy, -dz) + T(0.5) * f(p, 0, 0, 0) + T(0.25) * f(p, dx, dy, dz);
                }
                ok = S.barrier();
                src = dst;
            }
            jsrc[comp] = P.jf[comp];
        }
    }

    const T *dfin[3] = {nullptr, nullptr, nullptr};  // dE of the previous step (E update pending)
    int last = 0, steps_done = 0, noconv = 0;
    long long total = 0;
    double n2 = 0.0, r2 = 0.0;
    FieldL2<T> bf[3] = {{P.B[0], g}, {P.B[1], g}, {P.B[2], g}};
    for (int n = 0; n < a.nsteps && ok; ++n) {
        // ---- S: pending E update, source, ||dE'||^2
        double v = 0.0;
        for (int q = cells.lo + t; q < cells.hi; q += kNT) {
            Pos p;
            int64_t idx;
            cells.at(q, p, idx);
            if (dfin[0]) {
#pragma unroll
                for (int k = 0; k < 3; ++k) P.E[k][idx] = __ldcg(P.E[k] + idx) + __ldcg(dfin[k] + idx);
            }
            T ex = curl_alpha_b<T, DIM, 0>(bf, p, c);
            T ey = curl_alpha_b<T, DIM, 1>(bf, p, c);
            T ez = curl_alpha_b<T, DIM, 2>(bf, p, c);
            if (jsrc[0]) ex -= c.q * __ldcg(jsrc[0] + idx);
            if (jsrc[1]) ey -= c.q * __ldcg(jsrc[1] + idx);
            if (jsrc[2]) ez -= c.q * __ldcg(jsrc[2] + idx);
            P.dEp[0][idx] = ex;
            P.dEp[1][idx] = ey;
            P.dEp[2][idx] = ez;
            v += (double)ex * ex + (double)ey * ey + (double)ez * ez;
        }
        if (a.resid) {
            n2 = launch_sum(S, v, sums, par, ok);
            par ^= 1;
        } else {
            ok = S.barrier();
        }
        if (!ok) break;
        // ---- W_s: sweeps of Algorithm 1
        int s = 0;
        bool stop = a.resid ? n2 == 0.0 : a.m == 0;
        while (!stop) {
            const T *in[3];
            T *out[3];
            for (int k = 0; k < 3; ++k) {
                in[k] = s == 0 ? P.dEp[k] : ((s & 1) ? P.dEa[k] : P.dEb[k]);
                out[k] = ((s + 1) & 1) ? P.dEa[k] : P.dEb[k];
            }
            FieldL2<T> f[3] = {{in[0], g}, {in[1], g}, {in[2], g}};
            double w = 0.0;
            for (int q = cells.lo + t; q < cells.hi; q += kNT) {
                Pos p;
                int64_t idx;
                cells.at(q, p, idx);
                T own[3], av[3];
                const T p0 = __ldcg(P.dEp[0] + idx), p1 = __ldcg(P.dEp[1] + idx), p2 = __ldcg(P.dEp[2] + idx);
                av[0] = apply_a<T, DIM, 0>(f, p, c);
                av[1] = apply_a<T, DIM, 1>(f, p, c);
                av[2] = apply_a<T, DIM, 2>(f, p, c);
#pragma unroll
                for (int k = 0; k < 3; ++k) own[k] = __ldcg(in[k] + idx);
                const T nx_ = p0 + av[0], ny_ = p1 + av[1], nz_ = p2 + av[2];
                const T dx = nx_ - own[0], dy = ny_ - own[1], dz = nz_ - own[2];
                out[0][idx] = nx_;
                out[1][idx] = ny_;
                out[2][idx] = nz_;
                w += (double)dx * dx + (double)dy * dy + (double)dz * dz;
            }
            ++s;
            if (a.resid) {
                r2 = launch_sum(S, w, sums, par, ok);
                par ^= 1;
                if (!ok) break;
                if (r2 <= a.tol2 * n2) {
                    stop = true;
                } else if (s >= a.m_max) {
                    stop = true;
                    noconv = 1;
                }
            } else {
                ok = S.barrier();
                if (!ok) break;
                stop = s >= a.m;
            }
        }
        if (!ok) break;
        for (int k = 0; k < 3; ++k) dfin[k] = s == 0 ? P.dEp[k] : ((s & 1) ? P.dEa[k] : P.dEb[k]);
        last = s;
        total += s;
        // ---- F: Faraday with E^{n+1} = E^n + dE formed on the fly
        {
            SumL2<T> e[3] = {{P.E[0], dfin[0], g}, {P.E[1], dfin[1], g}, {P.E[2], dfin[2], g}};
            for (int q = cells.lo + t; q < cells.hi; q += kNT) {
                Pos p;
                int64_t idx;
                cells.at(q, p, idx);
                const T c0 = curl_e<T, DIM, 0>(e, p, c), c1 = curl_e<T, DIM, 1>(e, p, c),
                        c2 = curl_e<T, DIM, 2>(e, p, c);
                P.B[0][idx] = __ldcg(P.B[0] + idx) - c0;
                P.B[1][idx] = __ldcg(P.B[1] + idx) - c1;
                P.B[2][idx] = __ldcg(P.B[2] + idx) - c2;
            }
            ok = S.barrier();
        }
        if (!ok) break;
        ++steps_done;
        if (noconv) break;
    }
    if (!ok) return;  // a grid wait ran out: FMX_ETIMEOUT is latched in the status word
    // the last step's E update (everyone has passed the Faraday barrier)
    if (dfin[0]) {
        for (int q = cells.lo + t; q < cells.hi; q += kNT) {
            Pos p;
            int64_t idx;
            cells.at(q, p, idx);
#pragma unroll
            for (int k = 0; k < 3; ++k) P.E[k][idx] = __ldcg(P.E[k] + idx) + __ldcg(dfin[k] + idx);
        }
    }
    if (b == 0 && t == 0) {
        DevStatus *st = P.st;
        st->nrm2 = n2;
        st->r2 = r2;
        st->count = last;
        st->done = 1;
        st->noconv = noconv;
        st->steps = steps_done;
        st->sweeps_total = total;
    }
}

// The same engine for 2D grids that fit the shared memory of one cluster: CTA r
// owns rows r R .. r R + R - 1 (R = ceil(n_y / C)) of E, B, dE' and both sweep
// buffers there, with one halo row on either side, and every phase reads its
// own shared memory only; a CTA that computes a border row also writes it into
// the halo of the CTA above or below (distributed shared memory), which the
// phase's cluster barrier orders.  Nothing goes through L2 between the first
// load and the last store.  (Through L2 a phase took 6.6 us at 64^2, in FP32 as
// in FP64: about 22 loads of 700 cycles and a barrier that waits for the
// stores to reach L2.)  Only without a filtered current.
// us per step (20 steps a call, either side with the 22 us that a clock query per
// call then took), 64^2: FP64 to 1e-13 (12 sweeps) 119 -> 91.5, FP32 to 1e-5 (5 sweeps)
// 53 -> 40; 128^2 FP32 (3 sweeps) 59 -> 42.5; without the query 60.5, 14.4 and 16.1.
// A fixed sweep takes 3.2 us in FP64 (its 26 operations per cell: 2 us) and 0.8 us in
// FP32.
template <typename T>
__global__ void __launch_bounds__(kNT) k_resident_rows(ResidentArgs<T> a, Geo g, int R) {
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ SumSmem sums;
    __shared__ int abort_s;
    Sync S{cg::this_cluster(), a.P.st, 1, 0, 0, a.limit, 0, &abort_s};
    S.crank = (int)S.cl.block_rank();
    const int used = (g.ny + R - 1) / R;  // CTAs that own rows; the others only keep the barriers
    const int rank = S.crank, y0 = rank * R, rows = rank < used ? min(R, g.ny - y0) : 0;
    const int nx = g.nx, comp = (R + 2) * nx;  // a component: halo row, own rows, halo row (after the own rows)
    T *sm = reinterpret_cast<T *>(rsm);        // E[3], B[3], dE'[3], dEa[3], dEb[3]
    const int t = threadIdx.x;
    const Coef<T> &c = a.c;
    // the neighbours' shared memory, and where this CTA's border rows go there:
    // its first row into the halo above the rows of the CTA below, its last row
    // into the halo row 0 of the CTA above
    const int below = rows ? (rank + used - 1) % used : 0, above = rows ? (rank + 1) % used : 0;
    T *const smb = S.cl.map_shared_rank(sm, below), *const sma = S.cl.map_shared_rank(sm, above);
    const int top_b = (min(R, g.ny - below * R) + 1) * nx;
    auto put = [&](int k, int i, int j, T v) {
        sm[k * comp + (j + 1) * nx + i] = v;
        if (j == 0) smb[k * comp + top_b + i] = v;
        if (j == rows - 1) sma[k * comp + i] = v;
    };
    // the CTA's cells, a stride of kNT apart
    const int di = kNT % nx, dj = kNT / nx, i0 = t % nx, j0 = t / nx;
    auto cells = [&](auto f) {
        for (int i = i0, j = j0; j < rows;) {
            f(i, j);
            i += di;
            j += dj;
            if (i >= nx) {
                i -= nx;
                ++j;
            }
        }
    };
    auto gidx = [&](int i, int j) { return (int64_t)(y0 + j) * g.pitch + i; };

    // E and B of the own rows, pushed to the halos as every later border row is
    S.cl.sync();  // every CTA of the cluster is there before its memory is written
    cells([&](int i, int j) {
        const int64_t q = gidx(i, j);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            put(k, i, j, a.P.E[k][q]);
            put(3 + k, i, j, a.P.B[k][q]);
        }
    });
    S.cl.sync();

    int par = 0, last = 0, steps_done = 0, noconv = 0;
    bool ok = true;
    long long total = 0;
    double n2 = 0.0, r2 = 0.0;
    for (int n = 0; n < a.nsteps; ++n) {
        // ---- source, ||dE'||^2
        double v = 0.0;
        cells([&](int i, int j) {
            const int o = (j + 1) * nx + i, xm = i > 0 ? -1 : nx - 1, xp = i + 1 < nx ? 1 : 1 - nx;
            const T *bx = sm + 3 * comp + o, *by = sm + 4 * comp + o, *bz = sm + 5 * comp + o;
            auto ax = [&](const T *p) { return p[0] + c.c6 * ((p[xp] + p[xm]) - T(2) * p[0]); };
            auto ay = [&](const T *p) { return p[0] + c.c6 * ((p[nx] + p[-nx]) - T(2) * p[0]); };
            T d[3] = {c.ky * (bz[0] - bz[-nx]), -(c.kx * (bz[0] - bz[xm])),
                      c.kx * (ay(by) - ay(by + xm)) - c.ky * (ax(bx) - ax(bx - nx))};
            const int64_t q = gidx(i, j);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (a.have_j) d[k] -= c.q * __ldg(a.P.J[k] + q);
                put(6 + k, i, j, d[k]);
                v += (double)d[k] * d[k];
            }
        });
        if (a.resid) {
            n2 = launch_sum(S, v, sums, par, ok);
            par ^= 1;
        } else {
            S.cl.sync();
        }
        // ---- sweeps
        int s = 0, in = 6;
        bool stop = a.resid ? n2 == 0.0 : a.m == 0;
        while (!stop) {
            const int out = in == 9 ? 12 : 9;
            double w = 0.0;
            cells([&](int i, int j) {
                const int o = (j + 1) * nx + i, xm = i > 0 ? -1 : nx - 1, xp = i + 1 < nx ? 1 : 1 - nx;
                const T *p = sm + in * comp + o;
                auto at = [&](int k, int dx, int dy) { return p[k * comp + (dx < 0 ? xm : (dx > 0 ? xp : 0)) + dy * nx]; };
                T own[3], av[3];
                apply_a_2d<T>(at, c, own, av);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const T x = sm[(6 + k) * comp + o] + av[k], d = x - own[k];
                    put(out + k, i, j, x);
                    w += (double)d * d;
                }
            });
            ++s;
            in = out;
            if (a.resid) {
                r2 = launch_sum(S, w, sums, par, ok);
                par ^= 1;
                if (r2 <= a.tol2 * n2) {
                    stop = true;
                } else if (s >= a.m_max) {
                    stop = true;
                    noconv = 1;
                }
            } else {
                S.cl.sync();
                stop = s >= a.m;
            }
        }
        last = s;
        total += s;
        // ---- E^{n+1} = E^n + dE on the own rows and the halo row above them, Faraday
        for (int q = t; q < (rows ? (rows + 1) * nx : 0); q += kNT) {
#pragma unroll
            for (int k = 0; k < 3; ++k) sm[k * comp + nx + q] += sm[(in + k) * comp + nx + q];
        }
        __syncthreads();
        cells([&](int i, int j) {
            const int o = (j + 1) * nx + i, xp = i + 1 < nx ? 1 : 1 - nx;
            const T *ex = sm + o, *ey = sm + comp + o, *ez = sm + 2 * comp + o;
            const T bx = sm[3 * comp + o], by = sm[4 * comp + o], bz = sm[5 * comp + o];
            put(3, i, j, bx - c.ky * (ez[nx] - ez[0]));
            put(4, i, j, by + c.kx * (ez[xp] - ez[0]));
            put(5, i, j, (bz - c.kx * (ey[xp] - ey[0])) + c.ky * (ex[nx] - ex[0]));
        });
        S.cl.sync();
        ++steps_done;
        if (noconv) break;
    }
    cells([&](int i, int j) {
        const int64_t q = gidx(i, j);
        const int o = (j + 1) * nx + i;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            a.P.E[k][q] = sm[k * comp + o];
            a.P.B[k][q] = sm[(3 + k) * comp + o];
        }
    });
    if (rank == 0 && t == 0) {
        DevStatus *st = a.P.st;
        st->nrm2 = n2;
        st->r2 = r2;
        st->count = last;
        st->done = 1;
        st->noconv = noconv;
        st->steps = steps_done;
        st->sweeps_total = total;
    }
}

template <typename T, int DIM>
struct ResidentLauncher {
    // dynamic shared memory (unused) of more than half an SM's: one CTA per SM,
    // so that a cluster's CTAs spread over as many SMs (and FP64 pipes) as it has
    static size_t spread_bytes() {
        static size_t b = (size_t)-1;
        if (b == (size_t)-1) {
            int dev = 0, per_sm = 0, per_block = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
            cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            size_t want = (size_t)per_sm / 2 + 1024;
            if (want > (size_t)per_block) want = 0;
            if (want > 0 &&
                cudaFuncSetAttribute(k_resident<T, DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want) !=
                    cudaSuccess)
                want = 0;
            cudaGetLastError();
            b = want;
        }
        return b;
    }
    static cudaLaunchAttribute cluster_attr(int cs) {
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = cs;
        at.val.clusterDim.y = 1;
        at.val.clusterDim.z = 1;
        return at;
    }
    // cluster size: 16 CTAs where the device runs clusters of 16, else 8
    static int cluster() {
        static int cs = -1;
        if (cs < 0) {
            auto k = k_resident<T, DIM>;
            cs = 8;
            if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
                cudaLaunchConfig_t cfg = {};
                cudaLaunchAttribute at[1] = {cluster_attr(16)};
                cfg.gridDim = dim3(16);
                cfg.blockDim = dim3(kNT);
                cfg.dynamicSmemBytes = spread_bytes();
                cfg.attrs = at;
                cfg.numAttrs = 1;
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1) cs = 16;
            }
            cudaGetLastError();
        }
        return cs;
    }
    // clusters the device can hold at once (cooperative launches need them all
    // resident), capped by the status word's partial slots
    static int max_clusters() {
        static int mc = -1;
        if (mc < 0) {
            const int cs = cluster();
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1] = {cluster_attr(cs)};
            cfg.gridDim = dim3(cs);
            cfg.blockDim = dim3(kNT);
            cfg.dynamicSmemBytes = spread_bytes();
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, k_resident<T, DIM>, &cfg) != cudaSuccess || n < 1) n = 1;
            cudaGetLastError();
            mc = n < kMaxClusters ? n : kMaxClusters;
        }
        return mc;
    }
    // set once a cooperative launch over clusters has been refused
    static bool &coop_refused() {
        static bool r = false;
        return r;
    }
    // Clusters of a launch.  A grid barrier costs ~3 us per phase (an L2 atomic
    // round trip and a poll) on top of a cluster's; other clusters pay when they
    // take more work off the cluster's SMs than that.  Where that is depends on
    // the path: the shared-memory engine (k_resident_rows, one cluster only) is
    // far ahead of several clusters through L2 until FP64 arithmetic binds it, a
    // 3D cell has about six times the operations of a 2D one, a 1D cell a few.
    // us per step by clusters, random fields, 10 steps a call, residual to 1e-13
    // in FP64 and 1e-5 in FP32 (m = 4 in brackets):
    //   FP64 3D     16^3 767 (1), 731 (2); 17^3 1084 (1), 798 (2), 751 (3), 687 (4);
    //               20^3 1438 (1), 1059 (2), 724 (4) [112 (1), 100 (2), 84 (4)];
    //               22^3 1358 (2), 736 (6)
    //   FP64 2D     shared memory 80 x 64 318 (1), 480 (2); 90^2 470 (1), 475 (2), 432 (3),
    //               466 (5); 100^2 513 (1), 523 (3), 473 (5); 128^2 705 (1), 483 (7);
    //               filtered current 80 x 64 379 (1), 423 (2); 100^2 587 (1), 469 (5)
    //   FP64 1D     8000 143 (1), 203 (2); 12000 201 (1), 227 (6); 16384 232 (1), 239 (7)
    //   FP32 2D     shared memory 160^2 54 (1), 94 (7); 200^2 74 (1), 104 (7);
    //               through L2 256^2 186 (1), 117 (7); filtered 150^2 98 (1), 98 (7)
    //   FP32 3D     25^3 92 (1), 101 (4); 29^3 124 (1), 103 (7); 32^3 148 (1), 121 (4)
    //   FP32 1D     20000 66 (1), 74 (5); 40000 111 (1), 85 (5)
    // FP32 with fixed m stays on one cluster up to 65536 cells whatever the path:
    // several clusters report a barrier's time-out through a synchronising
    // read-back, one cluster only enqueues (and can be captured).
    static int clusters_for(const Geo &g, const ResidentArgs<T> &a) {
        if (coop_refused()) return 1;
        const int64_t cells = (int64_t)g.nx * g.ny * g.nz;
        int64_t one;
        if (sizeof(T) == 8) one = DIM == 3 ? 4096 : 8192;
        else one = rows_bytes(g, a) ? cells : (a.resid ? 24576 : 65536);
        if (cells <= one) return 1;
        const int64_t per_cta = sizeof(T) == 8 ? 128 : 512;
        const int64_t want = (cells + per_cta * cluster() - 1) / (per_cta * cluster());
        const int mc = max_clusters();
        return want < mc ? (int)want : mc;
    }
    static int rows_limit() {  // shared memory of a CTA
        static const int lim = [] {
            int dev = 0, v = 0;
            cudaGetDevice(&dev);
            return cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess ? v : 0;
        }();
        return lim;
    }
    // shared memory per CTA of the shared-memory engine; 0 where it does not apply
    static size_t rows_bytes(const Geo &g, const ResidentArgs<T> &a) {
        if (DIM != 2 || a.lost || (a.have_j && a.jpasses > 0)) return 0;
        const int cs = cluster(), R = (g.ny + cs - 1) / cs;
        const size_t need = (size_t)15 * (R + 2) * g.nx * sizeof(T);
        // half the cluster's CTAs with rows at least; 4 KB for the static part
        if (2 * ((g.ny + R - 1) / R) < cs || need + 4096 > (size_t)rows_limit()) return 0;
        return need;
    }
    // the shared-memory engine, where the grid takes one cluster and fits it;
    // false where it does not apply
    static bool run_rows(const Geo &g, const ResidentArgs<T> &a, int ncl, cudaStream_t s) {
        const size_t need = ncl == 1 ? rows_bytes(g, a) : 0;
        if (need == 0) return false;
        const int cs = cluster(), R = (g.ny + cs - 1) / cs;
        auto k = k_resident_rows<T>;
        static const bool attr =
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, rows_limit() - 4096) == cudaSuccess &&
            (cs <= 8 || cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess);
        if (!attr) {
            cudaGetLastError();
            return false;
        }
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1] = {cluster_attr(cs)};
        cfg.gridDim = dim3(cs);
        cfg.blockDim = dim3(kNT);
        // more than half an SM's shared memory: one CTA per SM
        cfg.dynamicSmemBytes = need > spread_bytes() ? need : spread_bytes();
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelEx(&cfg, k, a, g, R) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    }
    // ncl receives the launch's clusters
    static cudaError_t run(const Geo &g, const ResidentArgs<T> &a, int &ncl, cudaStream_t s) {
        ncl = clusters_for(g, a);
        if (run_rows(g, a, ncl, s)) return cudaSuccess;
        const int cs = cluster();
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2] = {cluster_attr(cs), {}};
        at[1].id = cudaLaunchAttributeCooperative;
        at[1].val.cooperative = 1;
        cfg.gridDim = dim3(cs * ncl);
        cfg.blockDim = dim3(kNT);
        cfg.dynamicSmemBytes = spread_bytes();
        cfg.stream = s;
        cfg.attrs = at;
        cfg.numAttrs = ncl > 1 ? 2 : 1;
        cudaError_t e = cudaLaunchKernelEx(&cfg, k_resident<T, DIM>, a, g);
        if (e != cudaSuccess && ncl > 1) {
            // this device or driver does not co-schedule clusters cooperatively:
            // one cluster from now on
            cudaGetLastError();
            coop_refused() = true;
            ncl = 1;
            cfg.gridDim = dim3(cs);
            cfg.numAttrs = 1;
            e = cudaLaunchKernelEx(&cfg, k_resident<T, DIM>, a, g);
        }
        return e;
    }
};

}  // namespace

template <typename T>
int resident_cluster_size(int dims) {
    return dims == 3 ? ResidentLauncher<T, 3>::cluster()
                     : (dims == 2 ? ResidentLauncher<T, 2>::cluster() : ResidentLauncher<T, 1>::cluster());
}

template <typename T>
int launch_resident(const Geo &g, int dims, const Coef<T> &c, const StagedPtrs<T> &P, int nsteps, bool resid, int m,
                    double tol2, int m_max, int jpasses, const ResidentWait &wait, cudaStream_t s) {
    ResidentArgs<T> a;
    a.P = P;
    a.c = c;
    a.nsteps = nsteps;
    a.resid = resid ? 1 : 0;
    a.m = m;
    a.m_max = m_max;
    a.tol2 = tol2;
    a.jpasses = jpasses;
    a.have_j = P.J[0] != nullptr;
    a.limit = wait.limit_cycles;
    a.lost = wait.lost_arrival ? 1 : 0;
    int ncl = 1;
    cudaError_t e = dims == 3 ? ResidentLauncher<T, 3>::run(g, a, ncl, s)
                              : (dims == 2 ? ResidentLauncher<T, 2>::run(g, a, ncl, s)
                                           : ResidentLauncher<T, 1>::run(g, a, ncl, s));
    return e == cudaSuccess ? ncl : -1;
}

template int resident_cluster_size<float>(int);
template int resident_cluster_size<double>(int);
template int launch_resident<float>(const Geo &, int, const Coef<float> &, const StagedPtrs<float> &, int, bool, int,
                                    double, int, int, const ResidentWait &, cudaStream_t);
template int launch_resident<double>(const Geo &, int, const Coef<double> &, const StagedPtrs<double> &, int, bool,
                                     int, double, int, int, const ResidentWait &, cudaStream_t);

}  // namespace fmx
