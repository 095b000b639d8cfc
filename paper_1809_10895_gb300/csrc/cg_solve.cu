// cg_solve.cu -- a whole Jacobi-PCG solve in one cooperative launch: FP64, or
// FP32 inside FP64 defect correction.
//
// As two kernels per iteration inside a conditional graph node, an iteration
// costs 18 us of node latency beside the kernels' own time.  Here the blocks
// stay resident: stencil products, updates and outer residuals are phases of
// one loop, each ended by a grid reduction (grid_red.cuh), and every block
// derives alpha, beta and the stop tests itself.  The sweeps: sweeps.cuh.
#include <algorithm>

#include "cell_ops.cuh"
#include "grid_red.cuh"
#include "rf_internal.cuh"
#include "sweeps.cuh"

namespace rf {

namespace {

struct CgShared {
    union {
        Sweep64Shared w64;
        Sweep32Shared w32;
    };
    IxSum part[2][CT / 32];
    float partf[3][CT / 32];
    double tot[4];
    double alpha, beta, rho, stop2;
    int done, status, iter, abort;
};

// Sums over the grid's threads.  fin runs on one thread while the rest wait, so
// it has no FP64 division, root or compare (a microsecond together; an FP32
// iteration over 256 x 256 x 64 cells took 46.6 us with them and block sums in
// FP64, 45.7 without).
template <int NV, class Fin>
__device__ __forceinline__ bool cg_reduce(GridRed &R, CgShared &s, const double (&v)[NV], Fin fin)
{
    return grid_red_sum<NV>(R, s.part, s.tot, &s.abort, v, fin);
}

template <bool NARROW>
__global__ void __launch_bounds__(CT, SWEEP_OCC)
k_cg64_solve(Grid g, Tiles tw, const double *__restrict__ Tx, const double *__restrict__ Ty,
             const double *__restrict__ Tz, const double *__restrict__ diag, const double *__restrict__ dinv,
             double *x, double *r, double *z, double *p0, double *p1, double *q, void *red, int *fault, CgScal *sc)
{
    count_launch(g, KK_ONE_LAUNCH);
    if (sc->done) return;                          // converged at the start, or the Picard attempt is over
    count_work(g, KK_ONE_LAUNCH);
    __shared__ CgShared s;
    GridRed R = grid_red_begin(red, fault, g.wait_tries);
    const double stop2 = sc->stop2 * sc->stop2;
    const int max_it = sc->max_it;
    if (threadIdx.x == 0) {
        s.rho = sc->rho;
        s.beta = 0.0;
        s.done = 0;
        s.status = CG_OK;
        s.abort = 0;
    }
    __syncthreads();
    const Op64 A{Tx, Ty, Tz, diag};
    int it = 0;
    for (;;) {
        const double beta = s.beta;
        const bool first = it == 0;
        const double *pin = (it & 1) ? p1 : p0;
        double *pout = (it & 1) ? p0 : p1;
        double acc[1] = {0.0};
        // ---- p = z + beta p_old, q = A p, p.q
        struct Raw {
            double z, o;
        };
        auto none = [](long long) { return NoOwn{}; };
        auto out = [&](long long c, double v, double Av, bool, NoOwn) {
            pout[c] = v;
            q[c] = Av;
            acc[0] = fma(v, Av, acc[0]);
        };
        if (NARROW)
            cells64<NoOwn>(g, A, [&](long long c) { return first ? z[c] : fma(beta, pin[c], z[c]); }, none, out);
        else
            sweep64<Raw, NoOwn>(
                g, tw, A, s.w64, [&](long long c) { return Raw{__ldcs(&z[c]), first ? 0.0 : __ldcs(&pin[c])}; },
                [&](const Raw &a) { return fma(beta, a.o, a.z); }, none, out);
        if (!cg_reduce<1>(R, s, acc, [&]() {
                const double pq = s.tot[0];
                s.alpha = ix_div(s.rho, pq);
                if (!is_positive(pq) || !is_finite(s.alpha)) {
                    s.status = CG_NONFINITE;
                    s.done = 1;
                }
            }))
            break;
        if (s.done) break;
        // ---- x += alpha p, r -= alpha q, z = D^-1 r, r.r, r.z
        const double alpha = s.alpha;
        double v[2] = {0.0, 0.0};
        cg64_update_cells(g, alpha, dinv, pout, q, x, r, z, v);
        it++;
        if (!cg_reduce<2>(R, s, v, [&]() {
                const double rr = s.tot[0], rz = s.tot[1];
                if (!is_finite(rr) || !is_finite(rz)) {
                    s.status = CG_NONFINITE;
                    s.done = 1;
                } else if (not_above(rr, stop2)) {
                    s.done = 1;
                } else if (it >= max_it) {
                    s.status = CG_MAXIT;
                    s.done = 1;
                } else {
                    s.beta = ix_div(rz, s.rho);
                    s.rho = rz;
                }
            }))
            break;
        if (s.done) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->iter = it;
        sc->total = it;
        sc->rho = s.rho;
        sc->rr = s.tot[0];
        sc->status = s.abort ? CG_NONFINITE : s.status;
        sc->done = 1;
    }
}

// FP32 sums within the block, FP64 across blocks.
template <int NV, class Fin>
__device__ __forceinline__ bool cg_reduce_f32(GridRed &R, CgShared &s, float (&v)[NV], Fin fin)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; i++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
        if (lane == 0) s.partf[i][wid] = v[i];
    }
    __syncthreads();
    return grid_red<OpIxSum, NV>(
        R, s.tot, &s.abort,
        [&](int i) {
            const float *p = s.partf[i];
            return (double)(((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7])));
        },
        fin);
}

// Defect correction from the assembly's (or the start kernels') first
// residual: outer and inner hold its scalars.
struct MixedArgs {
    Grid g;
    Tiles t64, t32;
    const uint8_t *flags;
    const double *Tx, *Ty, *Tz, *diag, *b;
    const float *K32, *cb32, *dinv32;
    double *x;
    float *r32, *z32, *d32, *p0, *p1, *q32;
    void *red;
    int *fault;
    CgScal *outer, *inner;
    double tol, tol_inner;
    int inner_max_it, outer_max_it;
};

template <bool NARROW>
__global__ void __launch_bounds__(CT, SWEEP_OCC)
k_mixed_solve(const __grid_constant__ MixedArgs M)
{
    const Grid &g = M.g;
    count_launch(g, KK_ONE_LAUNCH);
    if (M.outer->done) return;
    count_work(g, KK_ONE_LAUNCH);
    __shared__ CgShared s;
    GridRed R = grid_red_begin(M.red, M.fault, g.wait_tries);
    if (threadIdx.x == 0) {
        s.rho = M.inner->rho;
        s.stop2 = M.inner->stop2 * M.inner->stop2;
        s.beta = 0.0;
        s.iter = !M.inner->done;                   // an inner solve is due
        s.done = 0;
        s.status = CG_OK;
        s.abort = 0;
    }
    __syncthreads();
    const long long N = g.N, n4 = N / 4, stride = (long long)gridDim.x * CT;
    const long long t0 = (long long)blockIdx.x * CT + threadIdx.x;
    int outer = M.outer->iter, total = 0;
    for (;;) {
        // ---- inner FP32 PCG, A d = r from d = 0
        int it = 0;
        while (s.iter) {
            const float beta = (float)s.beta;
            const bool first = it == 0;
            const float *pin = (it & 1) ? M.p1 : M.p0;
            float *pout = (it & 1) ? M.p0 : M.p1;
            float w[1] = {NARROW ? cells32(g, M.K32, M.cb32, M.z32, pin, pout, M.q32, beta, first)
                                 : sweep32(g, M.t32, s.w32, M.K32, M.cb32, M.z32, pin, pout, M.q32, beta, first)};
            if (!cg_reduce_f32<1>(R, s, w, [&]() {
                    const double pq = s.tot[0];
                    s.alpha = ix_div(s.rho, pq);
                    if (!is_positive(pq) || !is_finite(s.alpha)) s.status = CG_NONFINITE;
                }))
                break;
            if (s.status != CG_OK) break;
            const float alpha = (float)s.alpha;
            float v[2] = {0.0f, 0.0f};
            cg32_update_cells(g, alpha, first, M.dinv32, pout, M.q32, M.d32, M.r32, M.z32, v);
            it++;
            if (!cg_reduce_f32<2>(R, s, v, [&]() {
                    const double rr = s.tot[0], rz = s.tot[1];
                    if (!is_finite(rr) || !is_finite(rz)) s.status = CG_NONFINITE;
                    else if (not_above(rr, s.stop2) || it >= M.inner_max_it) s.iter = 0;   // applied even at the cap
                    else {
                        s.beta = ix_div(rz, s.rho);
                        s.rho = rz;
                    }
                }))
                break;
            if (s.status != CG_OK) break;
        }
        total += it;
        if (s.abort || s.status != CG_OK) break;
        // ---- x += d
        if (it > 0) {
            for (long long u = t0; u < n4; u += stride) {
                const float4 d = reinterpret_cast<const float4 *>(M.d32)[u];
                double2 a = reinterpret_cast<double2 *>(M.x)[2 * u], c = reinterpret_cast<double2 *>(M.x)[2 * u + 1];
                a.x += ix_f2d(d.x);
                a.y += ix_f2d(d.y);
                c.x += ix_f2d(d.z);
                c.y += ix_f2d(d.w);
                reinterpret_cast<double2 *>(M.x)[2 * u] = a;
                reinterpret_cast<double2 *>(M.x)[2 * u + 1] = c;
            }
            for (long long c = 4 * n4 + t0; c < N; c += stride) M.x[c] += ix_f2d(M.d32[c]);
        }
        __syncthreads();
        if (gridDim.x > 1) {
            if (threadIdx.x == 0 && !grid_red_wait(R)) s.abort = 1;
            __syncthreads();
            if (s.abort) break;
        }
        // ---- r = b - A x in FP64, seeds of the next inner solve
        float f[3] = {0.0f, 0.0f, 0.0f};           // r.r, b.b, r.z
        const Op64 A{M.Tx, M.Ty, M.Tz, M.diag};
        resid64_sweep<NARROW>(g, M.t64, A, s.w64, M.flags, M.x, M.b, M.dinv32, M.r32, M.z32, nullptr, f);
        outer++;
        if (!cg_reduce_f32<3>(R, s, f, [&]() {
                const double rr = s.tot[0], bb = s.tot[1], rz = s.tot[2];
                if (!(is_finite(rr) && is_finite(bb) && is_finite(rz))) {
                    s.status = CG_NONFINITE;
                    s.done = 1;
                } else if (not_above(rr, M.tol * M.tol * bb)) {
                    s.done = 1;
                } else if (outer >= M.outer_max_it) {
                    s.status = CG_MAXIT;
                    s.done = 1;
                }
                s.rho = rz;
                s.stop2 = M.tol_inner * M.tol_inner * rr;
                s.beta = 0.0;
                s.iter = is_positive(rr);
            }))
            break;
        if (s.done) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        M.outer->iter = outer;
        M.outer->status = s.abort ? CG_NONFINITE : s.status;
        M.outer->done = 1;
        M.inner->total += total;
        M.inner->done = 1;
    }
}

}  // namespace

// Instances, and their blocks on this grid (0: it cannot run): what fits the
// GPU at once, but no more than there are tiles and planes, or cells, to share out.
static auto *cg64_fn(const Grid &g) { return narrow_grid(g, CX, CY) ? k_cg64_solve<true> : k_cg64_solve<false>; }
static auto *mixed_fn(const Grid &g) { return narrow_grid(g, CX, CY) ? k_mixed_solve<true> : k_mixed_solve<false>; }

static int solve_blocks(const void *fn, int sms)
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, CT, 0) != cudaSuccess || occ < 1) return 0;
    return std::min(occ * sms, GR_BLOCKS);
}

static int blocks_for(const Grid &g, int blocks, long long items)
{
    const long long shares = narrow_grid(g, CX, CY) ? (g.N + CT - 1) / CT : items;
    return (int)std::min<long long>(blocks, shares);
}

int cg64_solve_blocks(const Grid &g, int sms) { return solve_blocks((const void *)cg64_fn(g), sms); }
int mixed_solve_blocks(const Grid &g, int sms) { return solve_blocks((const void *)mixed_fn(g), sms); }

cudaError_t launch_cg64_solve(cudaStream_t s, int blocks, const Grid &g, const double *Tx, const double *Ty,
                              const double *Tz, const double *diag, const double *dinv, double *x, double *r,
                              double *z, double *p0, double *p1, double *q, void *red, int *fault, CgScal *sc)
{
    Grid gg = g;
    Tiles tw = make_tiles_balanced(g, blocks, CX, CY);
    blocks = blocks_for(g, blocks, tw.items);
    void *args[] = {&gg, &tw, &Tx, &Ty, &Tz, &diag, &dinv, &x, &r, &z, &p0, &p1, &q, &red, &fault, &sc};
    return cudaLaunchCooperativeKernel((void *)cg64_fn(g), dim3((unsigned)blocks), dim3(CT), args, 0, s);
}

cudaError_t launch_mixed_solve(cudaStream_t s, int blocks, const Grid &g, const uint8_t *flags, const double *Tx,
                               const double *Ty, const double *Tz, const double *diag, const double *b,
                               const float *K32, const float *cb32, const float *dinv32, double *x, float *r32,
                               float *z32, float *d32, float *p0, float *p1, float *q32, void *red, int *fault,
                               CgScal *outer, CgScal *inner, double tol, double tol_inner, int inner_max_it,
                               int outer_max_it)
{
    MixedArgs M{};
    M.g = g;
    M.t64 = make_tiles_balanced(g, blocks, CX, CY);
    M.t32 = make_tiles_balanced(g, blocks, CX, FY);
    M.flags = flags;
    M.Tx = Tx;
    M.Ty = Ty;
    M.Tz = Tz;
    M.diag = diag;
    M.b = b;
    M.K32 = K32;
    M.cb32 = cb32;
    M.dinv32 = dinv32;
    M.x = x;
    M.r32 = r32;
    M.z32 = z32;
    M.d32 = d32;
    M.p0 = p0;
    M.p1 = p1;
    M.q32 = q32;
    M.red = red;
    M.fault = fault;
    M.outer = outer;
    M.inner = inner;
    M.tol = tol;
    M.tol_inner = tol_inner;
    M.inner_max_it = inner_max_it;
    M.outer_max_it = outer_max_it;
    blocks = blocks_for(g, blocks, std::max(M.t64.items, M.t32.items));
    void *args[] = {&M};
    return cudaLaunchCooperativeKernel((void *)mixed_fn(g), dim3((unsigned)blocks), dim3(CT), args, 0, s);
}

}  // namespace rf
