// attempt_small.cu -- one Picard attempt of a small grid in one kernel launch.
//
// On a small grid every kernel of an attempt is latency: a working node of the
// attempt's graph costs about 12 us with its conditional loop, whatever the
// grid's size, and an attempt runs some fifty of them (200 cells: 6 Picard
// iterations of 3 CG iterations each; 41 attempts of them 19.4 ms from the
// graph, 4.6 ms here).  Here the whole attempt -- start copy,
// closures, assembly, PCG (FP64, or FP32 inside FP64 defect correction),
// Picard test, water balance, acceptance -- is one cooperative launch whose
// phases are separated by grid barriers of one or two microseconds (block
// barriers when the grid fits one block), with the per-cell arithmetic of the
// other kernels (cell_ops.cuh).
//
// Every reduction is one grid barrier (grid_red.cuh) after which all blocks
// hold bit-identical scalars and take the same decisions.  Sums run on the
// integer pipes (ix_sum.cuh) and their scalars without FP64 divisions and
// compares: of the 7240 cycles of a CG iteration on one block the two sums
// took 4430, staged in shared memory and added by one warp in FP64 (200 cells,
// 30 steps: 4.33 -> 3.94 ms; 30 000 cells on 117 blocks, 6 steps: 0.97 -> 0.94).
//
// Every loop is bounded as in the graph (max_it, outer_max_it, n_max), and a
// barrier wait that runs out sets the fault flag and ends the kernel.
#include <math.h>

#include <algorithm>

#include "cell_ops.cuh"
#include "grid_red.cuh"
#include "rf_internal.cuh"
#include "rf_reduce.cuh"

namespace rf {

namespace {

constexpr int AT_THREADS = 256;
constexpr int AT_WARPS = AT_THREADS / 32;
constexpr int AT_NV = 4;
static_assert(AT_NV <= GR_NV && AT_WARPS == 8, "reduction layout");

struct Shared {
    IxSum part[AT_NV][AT_WARPS];
    double partm[AT_WARPS];
    double tot[AT_NV];
    float partf[AT_NV][AT_WARPS];
    double alpha, beta, rho, stop2, max_dh;
    int done, ok, iter, abort;
    FxTables fx;
};

struct Ctx {
    Shared *s;
    GridRed R;
};

// Barrier over the grid's threads; false when a wait ran out.
__device__ __forceinline__ bool grid_sync(Ctx &C)
{
    __syncthreads();
    if (gridDim.x > 1) {
        if (threadIdx.x == 0 && !grid_red_wait(C.R)) C.s->abort = 1;
        __syncthreads();
    }
    return !C.s->abort;
}

// Sum NV FP64 values over the grid and run fin(totals) on thread 0 of every
// block; its results are visible to the block on return.
template <int NV, class Fin>
__device__ __forceinline__ bool grid_sum(Ctx &C, double (&v)[NV], Fin fin)
{
    Shared &s = *C.s;
    return grid_red_sum<NV>(C.R, s.part, s.tot, &s.abort, v, [&]() { fin(s.tot); });
}

// The same for FP32 thread values: FP32 within a block, FP64 across blocks.
template <int NV, class Fin>
__device__ __forceinline__ bool grid_sum_f32(Ctx &C, float (&v)[NV], Fin fin)
{
    Shared &s = *C.s;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; i++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
        if (lane == 0) s.partf[i][wid] = v[i];
    }
    __syncthreads();
    return grid_red<OpIxSum, NV>(
        C.R, s.tot, &s.abort,
        [&](int i) {
            const float *p = s.partf[i];
            return (double)(((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7])));
        },
        [&]() { fin(s.tot); });
}

// Maximum of non-negative doubles' bits over the grid (all ones: not finite).
__device__ __forceinline__ bool grid_max(Ctx &C, unsigned long long m)
{
    Shared &s = *C.s;
    const double t = OpMaxBits::warp(__longlong_as_double((long long)m));
    if ((threadIdx.x & 31) == 0) s.partm[threadIdx.x >> 5] = t;
    __syncthreads();
    return grid_red<OpMaxBits, 1>(
        C.R, s.tot, &s.abort,
        [&](int) {
            const int lane = threadIdx.x & 31;
            return OpMaxBits::warp(lane < AT_WARPS ? s.partm[lane] : 0.0);
        },
        [&]() { s.max_dh = s.tot[0]; });
}

// FP32 operator of an active cell (K32 is NaN on inactive cells).
template <class Get>
__device__ __forceinline__ float apply32(const Grid &g, int p, const float *K32, const float *cb32, Get get)
{
    int i, j, k;
    cell_ijk(g, p, i, j, k);
    const float KP = K32[p], vP = get(p);
    float acc = cb32[p] * vP;
    auto face = [&](bool in, int q, float w) {
        if (!in) return;
        const float KN = K32[q], vN = get(q);
        if (KN >= 0.0f) acc = fmaf(w * 0.5f * (KP + KN), vP - vN, acc);
    };
    face(i > 0, p - 1, g.w32[0]);
    face(i < g.nx - 1, p + 1, g.w32[0]);
    face(j > 0, p - g.nx, g.w32[1]);
    face(j < g.ny - 1, p + g.nx, g.w32[1]);
    face(k > 0, p - (int)g.sxy, g.w32[2]);
    face(k < g.nz - 1, p + (int)g.sxy, g.w32[2]);
    return acc;
}

template <int PREC>
__global__ void __launch_bounds__(AT_THREADS, 2)
k_attempt_small(const __grid_constant__ AttemptArgs A)
{
    __shared__ Shared s;
    const Grid &g = A.g;
    const StepParams &sp = A.sp;
    const int N = (int)g.N, stride = (int)(gridDim.x * AT_THREADS), p0 = (int)(blockIdx.x * AT_THREADS + threadIdx.x);
    Ctx C{&s, grid_red_begin(A.red, A.fault, g.wait_tries)};
    if (threadIdx.x == 0) s.abort = 0;
    {
        const uint64_t *src = reinterpret_cast<const uint64_t *>(&g.tab->fx);
        uint64_t *dst = reinterpret_cast<uint64_t *>(&s.fx);
        for (int i = threadIdx.x; i < (int)(sizeof(FxTables) / 8); i += AT_THREADS) dst[i] = src[i];
    }
    count_launch(g, KK_ONE_LAUNCH);
    count_work(g, KK_ONE_LAUNCH);
    __syncthreads();
    auto cell_closure = [&](int p, double hp, double *K) {
        double th, k, c;
        closure(A.soils[A.zone[p]], A.Ks[p], hp, g.tab, &s.fx, g.arith, th, k, c);
        A.theta_k[p] = th;
        K[p] = k;
        A.Can[p] = c;
    };
    if (A.copy_h) {
        for (int p = p0; p < N; p += stride) {
            const double hp = A.h[p];
            A.H[0][p] = hp;
            if (A.do_closure) {
                if (A.flags[p] & FLAG_ACTIVE) cell_closure(p, hp, A.K[0]);
                else { A.theta_k[p] = 0.0; A.K[0][p] = -1.0; A.Can[p] = 0.0; }
            }
        }
    }
    if (!grid_sync(C)) return;

    int half = 0, it = 0, cg_total = 0, conv = 0, fail = 0;
    double max_dh = 0.0;
    double *rr64 = A.r, *zz64 = A.z;
    for (;;) {
        const double *hk = A.H[half];
        double *x = A.H[half ^ 1];
        double *Kin = A.K[half], *Kout = A.K[half ^ 1];
        // ---- assembly and first residual
        double v[3] = {0.0, 0.0, 0.0};
        float f3[3] = {0.0f, 0.0f, 0.0f};
        for (int p = p0; p < N; p += stride) {
            const uint8_t fl = A.flags[p];
            const double hkP = hk[p];
            x[p] = hkP;
            if (!(fl & FLAG_ACTIVE)) {
                A.c[p] = 0.0; A.b[p] = 0.0; A.Tx[p] = 0.0; A.Ty[p] = 0.0; A.Tz[p] = 0.0;
                A.diag[p] = 0.0; A.dinv[p] = 0.0;
                A.K32[p] = __int_as_float(0x7fc00000); A.cb32[p] = 0.0f; A.dinv32[p] = 0.0f;
                if (PREC == 0) { rr64[p] = 0.0; zz64[p] = 0.0; }
                else { A.r32[p] = 0.0f; A.z32[p] = 0.0f; A.d32[p] = 0.0f; }
                continue;
            }
            int i, j, k;
            cell_ijk(g, p, i, j, k);
            CellSystem cs;
            assemble_cell<true>(g, A.soils, A.zone, A.Ks, fl, sp, p, i, j, k, hk, A.h, A.theta_k, A.theta_n, Kin,
                                A.Can, A.theta_p, sp.eps_chord, sp.V_dt, cs);
            A.c[p] = cs.c;
            A.b[p] = cs.rhs;
            if (A.s0) A.s0[p] = cs.s0;
            A.Tx[p] = cs.Tup[0];
            A.Ty[p] = cs.Tup[1];
            A.Tz[p] = cs.Tup[2];
            A.diag[p] = cs.diag;
            A.K32[p] = ix_d2f(cs.KP);
            A.cb32[p] = ix_d2f(cs.cb);
            const double rp = cs.rhs - (cs.diag * hkP - cs.sT);
            if (PREC == 0) {
                const double di = ix_rcp64(cs.diag), zp = di * rp;
                A.dinv[p] = di;
                A.dinv32[p] = ix_d2f(di);
                rr64[p] = rp;
                zz64[p] = zp;
                v[0] = fma(rp, zp, v[0]);
                v[1] = fma(rp, rp, v[1]);
                v[2] = fma(cs.rhs, cs.rhs, v[2]);
            } else {
                const float di = __frcp_rn(ix_d2f(cs.diag)), rf = ix_d2f(rp), zf = di * rf, bf = ix_d2f(cs.rhs);
                A.dinv32[p] = di;
                A.r32[p] = rf;
                A.z32[p] = zf;
                A.d32[p] = 0.0f;
                f3[0] = fmaf(rf, rf, f3[0]);
                f3[1] = fmaf(bf, bf, f3[1]);
                f3[2] = fmaf(rf, zf, f3[2]);
            }
        }
        int cg = 0;
        bool lin_ok = true;
        if (PREC == 0) {
            if (!grid_sum<3>(C, v, [&](const double *t) {
                    s.rho = t[0];
                    s.stop2 = A.tol_cg * A.tol_cg * t[2];
                    s.ok = is_finite(t[0]) && is_finite(t[1]) && is_finite(t[2]);
                    s.done = !s.ok || not_above(t[1], s.stop2);
                    s.beta = 0.0;
                }))
                return;
            while (!s.done) {
                const double *pin = A.p[cg & 1];
                double *pout = A.p[(cg & 1) ^ 1];
                const double beta = s.beta;
                const bool first = cg == 0;
                auto get = [&](long long q) { return first ? zz64[q] : fma(beta, pin[q], zz64[q]); };
                double w[1] = {0.0};
                if (gridDim.x == 1) {
                    // one block: p once per cell and a block barrier, instead
                    // of once per neighbour (a multiply-add each, on a pipe
                    // that an instruction of seven warps holds 128 cycles)
                    for (int p = p0; p < N; p += stride)
                        if (A.flags[p] & FLAG_ACTIVE) pout[p] = get(p);
                    __syncthreads();
                    for (int p = p0; p < N; p += stride) {
                        if (!(A.flags[p] & FLAG_ACTIVE)) continue;
                        const double qp = apply64(g, p, A.Tx, A.Ty, A.Tz, A.diag, [&](long long q) { return pout[q]; });
                        A.q[p] = qp;
                        w[0] = fma(pout[p], qp, w[0]);
                    }
                } else {
                    for (int p = p0; p < N; p += stride) {
                        if (!(A.flags[p] & FLAG_ACTIVE)) continue;
                        const double pp = get(p), qp = apply64(g, p, A.Tx, A.Ty, A.Tz, A.diag, get);
                        pout[p] = pp;
                        A.q[p] = qp;
                        w[0] = fma(pp, qp, w[0]);
                    }
                }
                if (!grid_sum<1>(C, w, [&](const double *t) {
                        s.alpha = ix_div(s.rho, t[0]);
                        if (!is_positive(t[0]) || !is_finite(s.alpha)) { s.ok = 0; s.done = 1; }
                    }))
                    return;
                if (s.done) break;
                const double alpha = s.alpha;
                double w2[2] = {0.0, 0.0};
                for (int p = p0; p < N; p += stride) {
                    const double di = A.dinv[p];
                    if (di == 0.0) continue;
                    x[p] = fma(alpha, pout[p], x[p]);
                    const double rp = fma(-alpha, A.q[p], rr64[p]), zp = di * rp;
                    rr64[p] = rp;
                    zz64[p] = zp;
                    w2[0] = fma(rp, rp, w2[0]);
                    w2[1] = fma(rp, zp, w2[1]);
                }
                cg++;
                if (!grid_sum<2>(C, w2, [&](const double *t) {
                        if (!is_finite(t[0]) || !is_finite(t[1])) { s.ok = 0; s.done = 1; }
                        else if (not_above(t[0], s.stop2)) s.done = 1;
                        else if (cg >= A.cg_max_it) { s.ok = 0; s.done = 1; }
                        else {
                            s.beta = ix_div(t[1], s.rho);
                            s.rho = t[1];
                        }
                    }))
                    return;
            }
            lin_ok = s.ok;
        } else {
            // defect correction: outer FP64 residuals, inner FP32 Jacobi-PCG
            auto outer_fin = [&](const double *t) {   // r.r, b.b, r.z of the FP32 seeds
                s.ok = is_finite(t[0]) && is_finite(t[1]) && is_finite(t[2]);
                s.done = !s.ok || not_above(t[0], A.tol_cg * A.tol_cg * t[1]);
                s.stop2 = A.tol_inner * A.tol_inner * t[0];
                s.rho = t[2];
                s.beta = 0.0;
                s.iter = is_positive(t[0]);
            };
            if (!grid_sum_f32<3>(C, f3, outer_fin)) return;
            int outer = 1;
            while (!s.done) {
                if (outer >= A.outer_max_it) { lin_ok = false; break; }
                int inner = 0;
                bool run = s.iter != 0;
                while (run) {
                    const float *pin = A.p32[inner & 1];
                    float *pout = A.p32[(inner & 1) ^ 1];
                    const float beta = (float)s.beta;
                    const bool first = inner == 0;
                    auto get = [&](int q) { return first ? A.z32[q] : fmaf(beta, pin[q], A.z32[q]); };
                    float w[1] = {0.0f};
                    for (int p = p0; p < N; p += stride) {
                        if (!(A.flags[p] & FLAG_ACTIVE)) continue;
                        const float pp = get(p), qp = apply32(g, p, A.K32, A.cb32, get);
                        pout[p] = pp;
                        A.q32[p] = qp;
                        w[0] = fmaf(pp, qp, w[0]);
                    }
                    if (!grid_sum_f32<1>(C, w, [&](const double *t) {
                            s.alpha = ix_div(s.rho, t[0]);
                            if (!is_positive(t[0]) || !is_finite(s.alpha)) s.ok = 0;
                        }))
                        return;
                    if (!s.ok) break;
                    const float alpha = (float)s.alpha;
                    float w2[2] = {0.0f, 0.0f};
                    for (int p = p0; p < N; p += stride) {
                        const float di = A.dinv32[p];
                        if (di == 0.0f) continue;
                        A.d32[p] = fmaf(alpha, pout[p], A.d32[p]);
                        const float rp = fmaf(-alpha, A.q32[p], A.r32[p]), zp = di * rp;
                        A.r32[p] = rp;
                        A.z32[p] = zp;
                        w2[0] = fmaf(rp, rp, w2[0]);
                        w2[1] = fmaf(rp, zp, w2[1]);
                    }
                    inner++;
                    if (!grid_sum_f32<2>(C, w2, [&](const double *t) {
                            s.iter = 1;
                            if (!is_finite(t[0]) || !is_finite(t[1])) s.ok = 0;
                            else if (not_above(t[0], s.stop2) || inner >= A.inner_max_it) s.iter = 0;
                            else {
                                s.beta = ix_div(t[1], s.rho);
                                s.rho = t[1];
                            }
                        }))
                        return;
                    run = s.ok && s.iter;
                }
                cg += inner;
                if (!s.ok) { lin_ok = false; break; }
                for (int p = p0; p < N; p += stride) x[p] += ix_f2d(A.d32[p]);
                if (!grid_sync(C)) return;
                float f[3] = {0.0f, 0.0f, 0.0f};
                for (int p = p0; p < N; p += stride) {
                    if (!(A.flags[p] & FLAG_ACTIVE)) continue;
                    const double bp = A.b[p];
                    // an inactive neighbour's head may be anything; its face's T = 0 needs a number
                    const double rp = bp - apply64(g, p, A.Tx, A.Ty, A.Tz, A.diag, [&](long long q) {
                                          return (A.flags[q] & FLAG_ACTIVE) ? x[q] : 0.0;
                                      });
                    const float rf = ix_d2f(rp), zf = A.dinv32[p] * rf, bf = ix_d2f(bp);
                    A.r32[p] = rf;
                    A.z32[p] = zf;
                    A.d32[p] = 0.0f;
                    f[0] = fmaf(rf, rf, f[0]);
                    f[1] = fmaf(bf, bf, f[1]);
                    f[2] = fmaf(rf, zf, f[2]);
                }
                outer++;
                if (!grid_sum_f32<3>(C, f, outer_fin)) return;
            }
            lin_ok = lin_ok && s.ok;
        }
        // ---- closures at the new iterate, Picard test
        unsigned long long m = 0;
        for (int p = p0; p < N; p += stride) {
            if (!(A.flags[p] & FLAG_ACTIVE)) {
                A.theta_k[p] = 0.0;
                Kout[p] = -1.0;
                A.Can[p] = 0.0;
                continue;
            }
            const double xp = x[p];
            unsigned long long d = (unsigned long long)__double_as_longlong(xp - hk[p]) & 0x7fffffffffffffffULL;
            if (d > 0x7e37e43c8800759cULL) d = ~0ULL;      // above 1e300, NaN or inf
            m = d > m ? d : m;
            cell_closure(p, xp, Kout);
        }
        if (!grid_max(C, m)) return;
        it++;
        half ^= 1;
        const double mx = s.max_dh;
        if (!lin_ok) {
            fail = 1;
        } else {
            cg_total += cg;
            max_dh = mx;
            if (__double_as_longlong(mx) == -1LL) fail = 1;
            else if (mx <= A.tol_picard) conv = 1;
        }
        if (conv || fail || it >= A.n_max) break;
    }
    // ---- water balance of the converged system; on one block, acceptance too
    // (with grid barriers, whose wait may run out, the host accepts once the
    // launch has ended without a fault)
    if (conv) {
        const bool accept = gridDim.x == 1;
        const double *x = A.H[half], *Kold = A.K[half ^ 1];
        const double dt = sp.dt;
        double v[4] = {0.0, 0.0, 0.0, 0.0};   // lin, dS, in, out
        for (int p = p0; p < N; p += stride) {
            const uint8_t fl = A.flags[p];
            const double xp = x[p], hnP = A.h[p], thx = A.theta_k[p], thn = A.theta_n[p];
            if (fl & FLAG_ACTIVE) {
                v[0] += A.s0 ? dt * (A.c[p] * xp - A.s0[p]) : A.c[p] * dt * (xp - hnP);
                v[1] += g.V * (thx - thn);
                if (fl & 0x3f) {
                    double fin, fout;
                    boundary_fluxes(g, A.soils[A.zone[p]], A.Ks[p], fl, sp, xp, hnP, Kold[p], fin, fout);
                    v[2] += dt * fin;
                    v[3] += dt * fout;
                }
            }
            if (accept) {
                if (A.keep_theta_p) A.theta_p[p] = thn;
                A.h[p] = xp;
                A.theta_n[p] = thx;
                if (half) A.K[0][p] = A.K[1][p];
            }
        }
        if (!grid_sum<4>(C, v, [&](const double *t) {
                if (blockIdx.x == 0) {
                    A.res->lin_change = t[0];
                    A.res->dstore = t[1];
                    A.res->bnd_in = t[2];
                    A.res->bnd_out = t[3];
                }
            }))
            return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        A.ctl->it = it;
        A.ctl->conv = conv;
        A.ctl->fail = fail;
        A.ctl->cg_total = cg_total;
        A.ctl->max_dh = max_dh;
        __threadfence_system();
    }
}

}  // namespace

cudaError_t launch_attempt_small(cudaStream_t s, const AttemptArgs &A, int mixed, int blocks)
{
    void *fn = mixed ? (void *)k_attempt_small<1> : (void *)k_attempt_small<0>;
    void *args[] = {const_cast<AttemptArgs *>(&A)};
    if (blocks == 1) return cudaLaunchKernel(fn, dim3(1), dim3(AT_THREADS), args, 0, s);
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)blocks), dim3(AT_THREADS), args, 0, s);
}

int attempt_small_blocks(long long N, int sms, int mixed)
{
    int o = 0;
    void *fn = mixed ? (void *)k_attempt_small<1> : (void *)k_attempt_small<0>;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, AT_THREADS, 0) != cudaSuccess || o < 1) return 0;
    const long long want = (N + AT_THREADS - 1) / AT_THREADS;
    if (want <= 2) return 1;         // one block's barrier is cheaper than a second block is fast
    return (int)std::min<long long>({want, (long long)sms * o, GR_BLOCKS});
}

}  // namespace rf
