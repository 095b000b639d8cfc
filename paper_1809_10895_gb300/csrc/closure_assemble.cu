// closure_assemble.cu -- per-cell closures (Eq. 2-4, Eq. A6), Picard-system
// assembly (Sec. 2.2), water-balance reductions.
//
// Layout: structure-of-arrays over all nx*ny*nz cells, x fastest.  Inactive
// cells carry K = -1 (a sentinel the stencil kernels test instead of reading
// the flag array) and zeros elsewhere.
#include <math.h>

#include "cell_ops.cuh"
#include "ix64.cuh"
#include "rf_internal.cuh"
#include "rf_reduce.cuh"
#include "tiles.cuh"

namespace rf {

// Largest |h - hprev| of a block's cells and whether one was not finite, as
// the bits of a non-negative double (order as integers: no FP64 compares).
struct MaxDh {
    unsigned long long d;
    int bad;
};

// Grid maximum of the blocks' values; true in the last block, whose thread 0
// then holds the result.
__device__ __forceinline__ bool grid_max_dh(MaxDh &m, double *partials, unsigned int *ticket)
{
    __shared__ unsigned long long sd[RED_THREADS / 32];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto block = [&]() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, m.d, o);
            m.d = v > m.d ? v : m.d;
        }
        if (lane == 0) sd[wid] = m.d;
        m.bad = __syncthreads_or(m.bad);
        if (threadIdx.x == 0)
            for (int w = 1; w < RED_THREADS / 32; w++) m.d = sd[w] > m.d ? sd[w] : m.d;
        __syncthreads();
    };
    block();
    unsigned long long *part = reinterpret_cast<unsigned long long *>(partials);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = m.d;
        part[gridDim.x + blockIdx.x] = (unsigned long long)m.bad;
        __threadfence();
        am_last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;   // wraps to 0 for the next use
    }
    __syncthreads();
    if (!am_last) return false;
    __threadfence();
    m.d = 0;
    m.bad = 0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += RED_THREADS) {
        const unsigned long long v = __ldcg(&part[b]);
        m.d = v > m.d ? v : m.d;
        m.bad |= __ldcg(&part[gridDim.x + b]) != 0;
    }
    block();
    return true;
}

// Closures of every cell at h; with hprev, also max|h - hprev| and whether
// an update was not finite.  In FP64 (table-driven exp and log, 106 FP64
// instructions a cell) the kernel was bound by the FP64 pipe; in fixed point
// it is bound by the integer pipes.  512 x 512 x 64 watershed, 12.6 M active
// cells: 3288 -> 446 us (1.5 TB/s of its 651 MB); 1 M cells: 34 us.  Loading
// the next cell's inputs ahead takes 80 registers or spills: 5 to 15 % slower;
// twice the blocks: 2.5 % faster there, 10 % slower on 1 M cells.  The
// tables (10 KB) sit in shared memory, where a gather costs its bank
// conflicts only.
template <bool DF>
__device__ __forceinline__ void closure_cells(const Grid &g, const DevSoil *__restrict__ soils,
                                              const uint8_t *__restrict__ zone, const double *__restrict__ Ks,
                                              const uint8_t *__restrict__ flags, const double *__restrict__ h,
                                              const double *__restrict__ hprev, double *__restrict__ theta,
                                              double *__restrict__ K, double *__restrict__ Can, MaxDh &m)
{
    __shared__ FxTables fx;
    if (!DF) {
        const uint64_t *src = reinterpret_cast<const uint64_t *>(&g.tab->fx);
        uint64_t *dst = reinterpret_cast<uint64_t *>(&fx);
        for (int i = threadIdx.x; i < (int)(sizeof(FxTables) / 8); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    m = MaxDh{0, 0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride) {
        if (!(flags[p] & FLAG_ACTIVE)) {
            theta[p] = 0.0;
            K[p] = -1.0;
            Can[p] = 0.0;
            continue;
        }
        const double hp = h[p];
        if (hprev) {
            const unsigned long long d = (unsigned long long)__double_as_longlong(hp - hprev[p]) & 0x7fffffffffffffffULL;
            if (d <= 0x7e37e43c8800759cULL) m.d = d > m.d ? d : m.d;   // 1e300
            else m.bad = 1;                                            // NaN or inf
        }
        double th, k, c;
        if (DF) closure_df(soils[zone[p]], Ks[p], hp, g.tab, th, k, c);
        else closure(soils[zone[p]], Ks[p], hp, g.tab, &fx, g.arith, th, k, c);
        theta[p] = th;
        K[p] = k;
        Can[p] = c;
    }
}

template <bool DF>
__global__ void __launch_bounds__(RED_THREADS)
k_closure(Grid g, const DevSoil *__restrict__ soils, const uint8_t *__restrict__ zone,
          const double *__restrict__ Ks, const uint8_t *__restrict__ flags, const double *__restrict__ h,
          const double *__restrict__ hprev, double *__restrict__ theta, double *__restrict__ K,
          double *__restrict__ Can, double *partials, unsigned int *ticket, StepResults *res)
{
    count_launch(g, KK_CLOSURE);
    count_work(g, KK_CLOSURE);
    MaxDh m;
    closure_cells<DF>(g, soils, zone, Ks, flags, h, hprev, theta, K, Can, m);
    if (hprev) {
        if (grid_max_dh(m, partials, ticket) && threadIdx.x == 0) {
            res->max_dh = __longlong_as_double((long long)m.d);
            res->nonfinite = m.bad;
        }
    }
}

// End of a Picard iteration on the device: closures at the new iterate x
// (which also serve the next assembly, or the next step once accepted), the
// exit test max|x - h^k| <= tol over all active cells (global, Sec. 2.3),
// and the loop control.  A failed linear solve or a non-finite update fails
// the attempt.  The last block sets the Picard loop condition; every launch
// sets it, so the loop always terminates (at the latest after n_max).
template <bool DF>
__global__ void __launch_bounds__(RED_THREADS)
k_closure_picard(Grid g, const DevSoil *__restrict__ soils, const uint8_t *__restrict__ zone,
                 const double *__restrict__ Ks, const uint8_t *__restrict__ flags, const double *__restrict__ x,
                 const double *__restrict__ hk, double *__restrict__ theta, double *__restrict__ K,
                 double *__restrict__ Can, double *partials, unsigned int *ticket, PicardCtl *ctl,
                 const CgScal *cg_status, const CgScal *cg_count, CondSet cond)
{
    count_launch(g, KK_CLOSURE_PICARD);
    if (ctl->done) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(cond, 0);
        return;
    }
    count_work(g, KK_CLOSURE_PICARD);
    MaxDh m;
    closure_cells<DF>(g, soils, zone, Ks, flags, x, hk, theta, K, Can, m);
    if (grid_max_dh(m, partials, ticket) && threadIdx.x == 0) {
        const double max_dh = __longlong_as_double((long long)m.d);
        const int it = ++ctl->it;
        if (cg_status->status != CG_OK) {
            ctl->fail = 1;
        } else {
            ctl->cg_total += cg_count->total;
            ctl->max_dh = max_dh;
            if (m.bad) ctl->fail = 1;
            else if (max_dh <= ctl->tol) {
                ctl->conv = 1;
                ctl->mb_pending = 1;
            }
        }
        ctl->done = (ctl->conv || ctl->fail || it >= ctl->n_max) ? 1 : 0;
        set_cond(cond, ctl->done ? 0 : 1);
    }
}

// Assembly of V C^k (h - h^n)/dt = sum_f T_f (h_N - h) + G + B (Sec. 2.2):
//   c = V C^k / dt, C^k the chord slope of theta* (or C(h^k) when
//   |h^k - h^n| <= eps); T_f = Kbar_f A_f/d_f, Kbar_f = (K_P + K_N)/2;
//   explicit gravity A_z (Kbar_top - Kbar_bottom) with K at h^k;
//   boundary terms per face class (Dirichlet at the half cell with K(h_D),
//   imposed flux, free drainage -K(h^k) A_z, seepage as Dirichlet 0 while the
//   cell is saturated at the step start).
// Outputs: c, b, upper-face coefficients Tx/Ty/Tz (0 where the face is not an
// interior face), diag(A), 1/diag; FP32 copies of K (NaN on inactive cells,
// so that max(w (K_P + K_N), 0) closes their faces without a test) and of c
// plus the Dirichlet diagonal terms for the mixed-precision operator.
// The Picard attempt is over (skip set): the linear-solve loops that follow
// are empty.
template <int MODE>
__device__ __forceinline__ bool assemble_skipped(const int *skip, const SolveStart &st)
{
    if (!(skip && *skip)) return false;
    if (MODE != ASM_ONLY && blockIdx.x == 0 && threadIdx.x == 0) {
        st.sc->done = 1;
        set_cond(st.cond, 0);
        if (MODE == ASM_MIXED) {
            st.inner->done = 1;
            set_cond(st.cond_inner, 0);
        }
    }
    return true;
}

// Outputs of an inactive cell (hkP: its raw h^k, kept in x).
template <int MODE>
__device__ __forceinline__ void assemble_inactive(long long p, double *__restrict__ c_out, double *__restrict__ b,
                                                  double *__restrict__ Tx, double *__restrict__ Ty,
                                                  double *__restrict__ Tz, double *__restrict__ diag_out,
                                                  double *__restrict__ dinv, float *__restrict__ K32,
                                                  float *__restrict__ cb32, float *__restrict__ dinv32, double hkP,
                                                  const SolveStart &st)
{
    c_out[p] = 0.0; b[p] = 0.0; Tx[p] = 0.0; Ty[p] = 0.0; Tz[p] = 0.0;
    diag_out[p] = 0.0; dinv[p] = 0.0;
    K32[p] = __int_as_float(0x7fc00000); cb32[p] = 0.0f; dinv32[p] = 0.0f;   // NaN: fails every K >= 0 test
    if (MODE != ASM_ONLY) st.x[p] = hkP;
    if (MODE == ASM_CG64) { st.r[p] = 0.0; st.z[p] = 0.0; }
    if (MODE == ASM_MIXED) { st.r32[p] = 0.0f; st.z32[p] = 0.0f; st.d32[p] = 0.0f; }
}

// Start scalars of the linear solve from the reduced norms (v: r.z, r.r, b.b
// in FP64; a_*: the FP32 seeds').
template <int MODE>
__device__ __forceinline__ void assemble_finish(double (&v)[3], float a_rr, float a_bb, float a_rz,
                                                const SolveStart &st, double *partials, unsigned int *ticket)
{
    if (MODE == ASM_CG64) {
        if (grid_reduce<OpSum, 3>(v, partials, ticket) && threadIdx.x == 0)
            cg64_start_scalars(st.sc, v, st.tol, st.max_it, st.cond);
    } else if (MODE == ASM_MIXED) {
        // the residual is formed in FP64; its norms (a stopping test and CG
        // seeds) are summed in FP32 within a block, in FP64 across blocks
        float vf[3] = {a_rr, a_bb, a_rz};
        double w[3];
        if (grid_reduce_f32<3>(vf, w, partials, ticket) && threadIdx.x == 0) {
            const double u[4] = {w[0], w[1], w[0], w[2]};
            st.sc->iter = 1;
            st.sc->done = 0;
            st.sc->status = CG_OK;
            st.inner->total = 0;
            outer_residual_scalars(st.sc, st.inner, u, st.tol, st.tol_inner, st.inner_max_it, st.outer_max_it,
                                   st.cond, st.cond_inner);
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(RED_THREADS)
k_assemble(Grid g, const DevSoil *__restrict__ soils, const uint8_t *__restrict__ zone,
           const double *__restrict__ Ks, const uint8_t *__restrict__ flags, const StepParams *__restrict__ spp,
           const double *__restrict__ hk, const double *__restrict__ hn, const double *__restrict__ thk,
           const double *__restrict__ thn, const double *__restrict__ K, const double *__restrict__ Can,
           double *__restrict__ c_out, double *__restrict__ b, double *__restrict__ Tx, double *__restrict__ Ty,
           double *__restrict__ Tz, double *__restrict__ diag_out, double *__restrict__ dinv,
           float *__restrict__ K32, float *__restrict__ cb32, float *__restrict__ dinv32, const int *skip,
           SolveStart st, double *partials, unsigned int *ticket, double *__restrict__ s0_out,
           const double *__restrict__ thp)
{
    count_launch(g, KK_ASSEMBLE);
    if (assemble_skipped<MODE>(skip, st)) return;
    count_work(g, KK_ASSEMBLE);
    const double eps = spp->eps_chord;
    const double V_dt = spp->V_dt;
    double v[3] = {0.0, 0.0, 0.0};
    float a_rr = 0.0f, a_bb = 0.0f, a_rz = 0.0f;   // mixed start: norms of the FP32 seeds, summed in FP32
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride) {
        const uint8_t fl = flags[p];
        if (!(fl & FLAG_ACTIVE)) {
            assemble_inactive<MODE>(p, c_out, b, Tx, Ty, Tz, diag_out, dinv, K32, cb32, dinv32, hk[p], st);
            continue;
        }
        int i, j, k;
        cell_ijk(g, p, i, j, k);
        const double hkP = hk[p];
        CellSystem cs;
        assemble_cell<MODE != ASM_ONLY>(g, soils, zone, Ks, fl, *spp, p, i, j, k, hk, hn, thk, thn, K, Can, thp, eps,
                                        V_dt, cs);
        const double c = cs.c, rhs = cs.rhs, diag = cs.diag, cb = cs.cb, sT = cs.sT, KP = cs.KP;
        const double *Tup = cs.Tup;
        c_out[p] = c;
        b[p] = rhs;
        if (s0_out) s0_out[p] = cs.s0;   // modified Picard: the water balance needs the storage part
        Tx[p] = Tup[0];
        Ty[p] = Tup[1];
        Tz[p] = Tup[2];
        // 1/diag: in FP64 for the FP64 PCG; the mixed path's Jacobi scaling
        // is FP32 only (its FP64 copy is not read), so it skips the FP64
        // reciprocal, a dozen instructions on the narrow FP64 pipe
        double di = 0.0;
        float di32;
        if (MODE == ASM_MIXED) {
            di32 = __frcp_rn((float)diag);
        } else {
            di = ix_rcp64(diag);
            dinv[p] = di;
            di32 = (float)di;
        }
        diag_out[p] = diag;
        K32[p] = (float)KP;
        cb32[p] = (float)cb;
        dinv32[p] = di32;
        if (MODE != ASM_ONLY) {
            // first residual of the linear solve from x0 = h^k
            const double rp = rhs - (diag * hkP - sT);
            st.x[p] = hkP;
            if (MODE == ASM_CG64) {
                const double zp = di * rp;
                st.r[p] = rp;
                st.z[p] = zp;
                v[0] += rp * zp;
                v[1] += rp * rp;
                v[2] += rhs * rhs;
            } else {
                const float rf = (float)rp;
                const float zf = di32 * rf;
                const float bf = (float)rhs;
                st.r32[p] = rf;
                st.z32[p] = zf;
                st.d32[p] = 0.0f;
                a_rr = fmaf(rf, rf, a_rr);
                a_bb = fmaf(bf, bf, a_bb);
                a_rz = fmaf(rf, zf, a_rz);
            }
        }
    }
    assemble_finish<MODE>(v, a_rr, a_bb, a_rz, st, partials, ticket);
}

// The same assembly for grids that fill the GPU with 32 x 8 column tiles: a
// block walks its tile's planes upwards, K and h^k of a plane (with a one-cell
// halo) in shared memory, those of the planes below and above in registers,
// everything else loaded a plane ahead.  The face coefficients
// T = (K_P + K_N) hw, their sum and the two reciprocals are positive, so they
// run in integer arithmetic (ix64.cuh) beside the narrow FP64 pipe, which
// bounds the kernel; the top face of a plane is the bottom face of the next.
// FP64 keeps the signed work: 10 instructions a cell (18 with the first residual)
// instead of 31.  512 x 512 x 64 watershed (12.6 M active cells): 1105 us
// with one cell per thread and all of it in FP64, 719 us with the diagonal's
// six adds left in FP64, 652 here; 384 x 320 x 64 mixed 540 -> 381 -> 333 us.
template <int MODE>
__global__ void __launch_bounds__(RED_THREADS, 2)
k_assemble_tiled(Grid g, Tiles tw, const DevSoil *__restrict__ soils, const uint8_t *__restrict__ zone,
                 const double *__restrict__ Ks, const uint8_t *__restrict__ flags,
                 const StepParams *__restrict__ spp, const double *__restrict__ hk, const double *__restrict__ hn,
                 const double *__restrict__ thk, const double *__restrict__ thn, const double *__restrict__ K,
                 const double *__restrict__ Can, double *__restrict__ c_out, double *__restrict__ b,
                 double *__restrict__ Tx, double *__restrict__ Ty, double *__restrict__ Tz,
                 double *__restrict__ diag_out, double *__restrict__ dinv, float *__restrict__ K32,
                 float *__restrict__ cb32, float *__restrict__ dinv32, const int *skip, SolveStart st,
                 double *partials, unsigned int *ticket, double *__restrict__ s0_out,
                 const double *__restrict__ thp)
{
    count_launch(g, KK_ASSEMBLE);
    if (assemble_skipped<MODE>(skip, st)) return;
    count_work(g, KK_ASSEMBLE);
    __shared__ long long sK[2][TY + 2][TX + 2];
    __shared__ double sH[2][TY + 2][TX + 2];
    constexpr long long CLOSED = K_CLOSED;
    const double eps = spp->eps_chord, V_dt = spp->V_dt;
    const int form = storage_form(*spp);
    const IxNum hwx = ix_unpack((uint64_t)__double_as_longlong(g.hw[0]));
    const IxNum hwy = ix_unpack((uint64_t)__double_as_longlong(g.hw[2]));
    const IxNum hwz = ix_unpack((uint64_t)__double_as_longlong(g.hw[4]));
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    int hx = 0, hy = 0;
    if (threadIdx.x < HALO) halo_cell(threadIdx.x, hx, hy);
    double v[3] = {0.0, 0.0, 0.0};
    float a_rr = 0.0f, a_bb = 0.0f, a_rz = 0.0f;   // mixed start: norms of the FP32 seeds, summed in FP32
    struct Pl {
        double hn, thk, thn, can;
        uint8_t fl;
    };
    for (long long item = blockIdx.x; item < tw.items; item += gridDim.x) {
        const TileItem it = tile_item(g, tw, item);
        const int i = it.i0 + tx, j = it.j0 + ty;
        const bool inside = i < g.nx && j < g.ny;
        const long long col = i + (long long)g.nx * j;
        const bool halo = threadIdx.x < HALO && it.i0 + hx >= 0 && it.i0 + hx < g.nx && it.j0 + hy >= 0 &&
                          it.j0 + hy < g.ny;
        const long long hcol = (it.i0 + hx) + (long long)g.nx * (it.j0 + hy);
        auto ldK = [&](int k) -> long long {
            return inside && k >= 0 && k < g.nz ? __double_as_longlong(K[col + g.sxy * k]) : CLOSED;
        };
        auto ldh = [&](int k) -> double { return inside && k >= 0 && k < g.nz ? hk[col + g.sxy * k] : 0.0; };
        auto load = [&](int k, bool act) {
            Pl l{0.0, 0.0, 0.0, 0.0, 0};
            if (act) {
                const long long p = col + g.sxy * k;
                l.hn = hn[p];
                l.thk = thk[p];
                l.thn = thn[p];
                l.can = Can[p];
                l.fl = flags[p];
            }
            return l;
        };
        long long Kc = ldK(it.k0), Kn = ldK(it.k0 + 1), Kh = CLOSED;
        double hm = 0.0, hc = ldh(it.k0), hu = ldh(it.k0 + 1), hh = 0.0;
        if (halo) {
            Kh = __double_as_longlong(K[hcol + g.sxy * it.k0]);
            hh = hk[hcol + g.sxy * it.k0];
        }
        Pl nxt = load(it.k0, Kc >= 0);
        double Tbot = 0.0;
        if (it.k0 > 0) {
            const long long Kb = ldK(it.k0 - 1);
            Tbot = face_coef(g, Kb, Kc, g.hw[4], hwz);
            hm = Kb >= 0 ? ldh(it.k0 - 1) : 0.0;
        }
        for (int k = it.k0; k < it.k1; k++) {
            const int buf = k & 1;
            const long long p = col + g.sxy * k;
            const Pl cur = nxt;
            sK[buf][ty + 1][tx + 1] = Kc;
            sH[buf][ty + 1][tx + 1] = Kc >= 0 ? hc : 0.0;    // a closed face's head is multiplied by T = 0
            if (threadIdx.x < HALO) {
                sK[buf][hy + 1][hx + 1] = Kh;
                sH[buf][hy + 1][hx + 1] = Kh >= 0 ? hh : 0.0;
            }
            long long K2 = CLOSED;
            double h2 = 0.0;
            if (k + 1 < it.k1) {
                K2 = ldK(k + 2);
                h2 = ldh(k + 2);
                nxt = load(k + 1, Kn >= 0);
                if (halo) {
                    Kh = __double_as_longlong(K[hcol + g.sxy * (k + 1)]);
                    hh = hk[hcol + g.sxy * (k + 1)];
                }
            }
            __syncthreads();
            double Ttop = 0.0;
            if (Kc >= 0) {
                const double hkP = hc;
                double c, s0;
                storage_terms(form, *spp, V_dt, eps, hkP, cur.hn, cur.thk, cur.thn, cur.can, thp, p, c, s0);
                const long long kxm = sK[buf][ty + 1][tx], kxp = sK[buf][ty + 1][tx + 2];
                const long long kym = sK[buf][ty][tx + 1], kyp = sK[buf][ty + 2][tx + 1];
                const double T0 = face_coef(g, kxm, Kc, g.hw[0], hwx), T1 = face_coef(g, Kc, kxp, g.hw[0], hwx);
                const double T2 = face_coef(g, kym, Kc, g.hw[2], hwy), T3 = face_coef(g, Kc, kyp, g.hw[2], hwy);
                Ttop = face_coef(g, Kc, Kn, g.hw[4], hwz);
                const double hz = Kn >= 0 ? hu : 0.0;
                double diag = diag_sum(c, {T0, T1, T2, T3, Tbot, Ttop});
                double rhs = fma(Ttop, g.gd[F_ZMAX], fma(Tbot, g.gd[F_ZMIN], s0));   // explicit gravity
                if (g.tilted) {
                    rhs = fma(T0, g.gd[F_XMIN], fma(T1, g.gd[F_XMAX], rhs));
                    rhs = fma(T2, g.gd[F_YMIN], fma(T3, g.gd[F_YMAX], rhs));
                }
                double sT = 0.0;
                if (MODE != ASM_ONLY) {
                    sT = T0 * sH[buf][ty + 1][tx];
                    sT = fma(T1, sH[buf][ty + 1][tx + 2], sT);
                    sT = fma(T2, sH[buf][ty][tx + 1], sT);
                    sT = fma(T3, sH[buf][ty + 2][tx + 1], sT);
                    sT = fma(Tbot, hm, sT);
                    sT = fma(Ttop, hz, sT);
                }
                double cb = c;
                if (cur.fl & 0x3f) {
                    const double KP = __longlong_as_double(Kc);
                    for (int f = 0; f < 6; f++)
                        if (cur.fl & (1u << f))
                            boundary_face(g, soils, zone, Ks, *spp, p, f, cur.hn, KP, diag, cb, rhs);
                }
                c_out[p] = c;
                b[p] = rhs;
                if (s0_out) s0_out[p] = s0;
                Tx[p] = T1;
                Ty[p] = T3;
                Tz[p] = Ttop;
                float di32;
                double di = 0.0;
                if (MODE == ASM_MIXED) {
                    di32 = __frcp_rn(ix_d2f(diag));
                } else {
                    di = ix_rcp64(diag);
                    dinv[p] = di;
                    di32 = ix_d2f(di);
                }
                diag_out[p] = diag;
                K32[p] = ix_d2f(__longlong_as_double(Kc));
                cb32[p] = ix_d2f(cb);
                dinv32[p] = di32;
                if (MODE != ASM_ONLY) {
                    const double rp = rhs - fma(diag, hkP, -sT);     // first residual, x0 = h^k
                    st.x[p] = hkP;
                    if (MODE == ASM_CG64) {
                        const double zp = di * rp;
                        st.r[p] = rp;
                        st.z[p] = zp;
                        v[0] = fma(rp, zp, v[0]);
                        v[1] = fma(rp, rp, v[1]);
                        v[2] = fma(rhs, rhs, v[2]);
                    } else {
                        const float rf = ix_d2f(rp);
                        const float zf = di32 * rf;
                        const float bf = ix_d2f(rhs);
                        st.r32[p] = rf;
                        st.z32[p] = zf;
                        st.d32[p] = 0.0f;
                        a_rr = fmaf(rf, rf, a_rr);
                        a_bb = fmaf(bf, bf, a_bb);
                        a_rz = fmaf(rf, zf, a_rz);
                    }
                }
            } else if (inside) {
                assemble_inactive<MODE>(p, c_out, b, Tx, Ty, Tz, diag_out, dinv, K32, cb32, dinv32, hc, st);
            }
            Tbot = Ttop;
            hm = Kc >= 0 ? hc : 0.0;
            Kc = Kn;
            Kn = K2;
            hc = hu;
            hu = h2;
        }
        __syncthreads();
    }
    assemble_finish<MODE>(v, a_rr, a_bb, a_rz, st, partials, ticket);
}

// Water balance of the accepted step's last linear system (x = h^{n+1}):
// sum c dt (x - h^n), sum V (theta*(x) - theta*(h^n)), and dt times the
// boundary inflow / outflow of that system, split per face by sign.
// After a Picard attempt (ctl given): only when it converged; the final
// iterate and the K of its last system sit in the buffers of the last
// iteration's half: x_odd / K_odd after an odd number of iterations, x_even /
// K_even after an even number.
__global__ void __launch_bounds__(RED_THREADS)
k_mass_balance(Grid g, const DevSoil *__restrict__ soils, const uint8_t *__restrict__ zone,
               const double *__restrict__ Ks, const uint8_t *__restrict__ flags,
               const StepParams *__restrict__ spp, const double *__restrict__ x_odd,
               const double *__restrict__ x_even, const double *__restrict__ hn, const double *__restrict__ c,
               const double *__restrict__ K_odd, const double *__restrict__ K_even, const double *__restrict__ thx,
               const double *__restrict__ thn, double *partials, unsigned int *ticket, StepResults *res,
               const PicardCtl *ctl, const double *__restrict__ s0)
{
    count_launch(g, KK_MASS_BALANCE);
    if (ctl && !ctl->conv) return;
    count_work(g, KK_MASS_BALANCE);
    const bool odd = !ctl || (ctl->it & 1);
    const double *__restrict__ x = odd ? x_odd : x_even;
    const double *__restrict__ Kold = odd ? K_odd : K_even;
    const double dt = spp->dt;
    double v[4] = {0.0, 0.0, 0.0, 0.0};   // lin, dS, in, out
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride) {
        const uint8_t fl = flags[p];
        if (!(fl & FLAG_ACTIVE)) continue;
        const double xp = x[p], hnP = hn[p];
        // storage of the solved system: c (x - h^n), or with modified Picard
        // c x - s0 = c (x - h^k) + V (theta*^k - theta*^n) / dt (times dt)
        v[0] += s0 ? dt * (c[p] * xp - s0[p]) : c[p] * dt * (xp - hnP);
        v[1] += g.V * (thx[p] - thn[p]);
        if (!(fl & 0x3f)) continue;
        double fin, fout;
        boundary_fluxes(g, soils[zone[p]], Ks[p], fl, *spp, xp, hnP, Kold[p], fin, fout);
        v[2] += dt * fin;
        v[3] += dt * fout;
    }
    if (grid_reduce<OpSum, 4>(v, partials, ticket) && threadIdx.x == 0) {
        res->lin_change = v[0];
        res->dstore = v[1];
        res->bnd_in = v[2];
        res->bnd_out = v[3];
    }
}

__global__ void __launch_bounds__(RED_THREADS)
k_storage(Grid g, const uint8_t *__restrict__ flags, const double *__restrict__ theta, double *partials,
          unsigned int *ticket, StepResults *res)
{
    count_launch(g, KK_STORAGE);
    count_work(g, KK_STORAGE);
    double v[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride)
        if (flags[p] & FLAG_ACTIVE) v[0] += g.V * theta[p];
    if (grid_reduce<OpSum, 1>(v, partials, ticket) && threadIdx.x == 0) res->storage = v[0];
}

__global__ void __launch_bounds__(RED_THREADS)
k_accept(Grid g, const double *__restrict__ xf, double *__restrict__ h, const double *__restrict__ thk,
         double *__restrict__ thn, const double *__restrict__ K1, double *__restrict__ K0, int copyK)
{
    count_launch(g, KK_ACCEPT);
    count_work(g, KK_ACCEPT);
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride) {
        h[p] = xf[p];
        thn[p] = thk[p];
        if (copyK) K0[p] = K1[p];
    }
}

// Check of a state uploaded into src: the number of active cells whose head
// is not finite (res->nonfinite); then, only when there is none, the commit
// dst = src with non-finite values on inactive cells replaced by 0.
__global__ void __launch_bounds__(RED_THREADS)
k_state_check(Grid g, const uint8_t *__restrict__ flags, const double *__restrict__ src, double *partials,
              unsigned int *ticket, StepResults *res)
{
    double v[1] = {0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride)
        if ((flags[p] & FLAG_ACTIVE) && !isfinite(src[p])) v[0] += 1.0;
    if (grid_reduce<OpSum, 1>(v, partials, ticket) && threadIdx.x == 0) res->nonfinite = v[0] > 0.0;
}

__global__ void __launch_bounds__(RED_THREADS)
k_state_commit(Grid g, const double *__restrict__ src, double *__restrict__ dst, const StepResults *res)
{
    if (res->nonfinite) return;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < g.N; p += stride) {
        const double v = src[p];
        dst[p] = isfinite(v) ? v : 0.0;
    }
}

void launch_state_check_commit(cudaStream_t s, int nblk, const Grid &g, const uint8_t *flags, const double *src,
                               double *dst, double *partials, unsigned int *ticket, StepResults *res)
{
    k_state_check<<<nblk, RED_THREADS, 0, s>>>(g, flags, src, partials, ticket, res);
    k_state_commit<<<nblk, RED_THREADS, 0, s>>>(g, src, dst, res);
}

// Both precisions' tables: the double-float ones from double arithmetic,
// the FP64 ones from long double (extended or quadruple precision on the
// hosts this builds for), each rounded once.
static void fill_ff_tables(FFTables *t)
{
    for (int j = 0; j < F64_TAB; j++) {
        const long double e = exp2l((long double)j / (long double)F64_TAB);
        const double hi = (double)e;
        t->e2[j] = make_double2(hi, (double)(e - (long double)hi));
    }
    for (int j = 0; j <= F64_TAB; j++) {
        const long double F = 1.0L + (long double)j / (long double)F64_TAB;
        const long double lf = logl(F);
        const double hi = (double)(rintl(lf * 4398046511104.0L) / 4398046511104.0L);   // 2^42 grid
        t->lF[j] = make_double2(hi, (double)(lf - (long double)hi));
        t->invF[j] = (double)(1.0L / F);
    }
    for (int j = 0; j < FX_TAB; j++) {
        const long double F = 1.0L + (long double)j / (long double)FX_TAB;
        t->fx.rc[j] = (uint32_t)ceill(2147483648.0L / F);   // rounded up, so that r >= 0
        t->fx.lg[j] = (uint64_t)rintl(-log2l((long double)t->fx.rc[j] / 2147483648.0L) * 9223372036854775808.0L);
        t->fx.e2[j] = (uint64_t)rintl(exp2l((long double)j / (long double)FX_TAB) * 9223372036854775808.0L);
    }
    for (int j = 0; j < 64; j++) {
        const double e = exp2((double)j / 64.0);
        const double c = 1.0 + ((double)j + 0.5) / 64.0;
        const double lc = log(c), ic = 1.0 / c;
        const float eh = (float)e, lh = (float)lc, ih = (float)ic;
        t->exp2j[j] = make_float2(eh, (float)(e - (double)eh));
        t->logc[j] = make_float2(lh, (float)(lc - (double)lh));
        t->invc[j] = make_float2(ih, (float)(ic - (double)ih));
    }
}

// Constants, computed once per process (quadruple-precision logarithms on a
// host whose long double is software cost most of a millisecond).
const FFTables *ff_tables()
{
    static FFTables t;
    static const bool filled = (fill_ff_tables(&t), true);
    (void)filled;
    return &t;
}

void launch_closure(cudaStream_t s, int nblk, const Grid &g, const DevSoil *soils, const uint8_t *zone,
                    const double *Ks, const uint8_t *flags, const double *h, const double *hprev,
                    double *theta, double *K, double *Can, double *partials, unsigned int *ticket,
                    StepResults *res)
{
    auto *fn = g.arith == ARITH_DF ? k_closure<true> : k_closure<false>;
    fn<<<nblk, RED_THREADS, 0, s>>>(g, soils, zone, Ks, flags, h, hprev, theta, K, Can, partials, ticket, res);
}

void launch_closure_picard(cudaStream_t s, int nblk, const Grid &g, const DevSoil *soils, const uint8_t *zone,
                           const double *Ks, const uint8_t *flags, const double *x, const double *hk,
                           double *theta, double *K, double *Can, double *partials, unsigned int *ticket,
                           PicardCtl *ctl, const CgScal *cg_status, const CgScal *cg_count, CondSet cond)
{
    auto *fn = g.arith == ARITH_DF ? k_closure_picard<true> : k_closure_picard<false>;
    fn<<<nblk, RED_THREADS, 0, s>>>(g, soils, zone, Ks, flags, x, hk, theta, K, Can, partials, ticket, ctl, cg_status,
                                    cg_count, cond);
}

// Tiles where the planes fill them and there are enough cells that marching
// through planes beats one cell per thread (below, every launch is latency and
// the general kernel's one cell per thread is the shorter chain).  us, tiled / one
// cell per thread, alone (fused with the first residual the tiled form gains
// some 30 us more on 600 000 cells): 256 x 256 x 64 199 / 267, 128 x 128 x 64 61 /
// 72, 45 x 45 x 60 (0.66 of the tiles filled) 19 / 16, 33 x 33 x 500 (0.43) 66 / 39,
// 16 x 4 x 10000 (0.25) 95 / 44; steps of 600 000 cells: 0.75 filled 23.2 / 23.4 ms,
// 0.62 30.7 / 30.8, 0.5 equal, 0.43 25.6 / 25.5.  The harmonic mean divides in FP64
// for every face, each twice in a tile's walk but for the vertical ones: 0.75
// filled 152 / 120, 0.94 185 / 170, full 107 / 113 (642 000 cells).
static bool assemble_tiled(const Grid &g)
{
    const long long area = (long long)((g.nx + TX - 1) / TX) * TX * ((g.ny + TY - 1) / TY) * TY;
    return g.N >= 32768 && (g.harmonic ? 16 * g.sxy > 15 * area : 8 * g.sxy >= 5 * area);
}

void launch_assemble(cudaStream_t s, int nblk, const Grid &g, const DevSoil *soils, const uint8_t *zone,
                     const double *Ks, const uint8_t *flags, const StepParams *sp, const double *hk,
                     const double *hn, const double *theta_k, const double *theta_n, const double *K,
                     const double *Can, double *c, double *b, double *Tx, double *Ty, double *Tz,
                     double *diag, double *dinv, float *K32, float *cb32, float *dinv32, const int *skip,
                     int mode, const SolveStart *start, double *partials, unsigned int *ticket, double *s0,
                     const double *theta_p)
{
    SolveStart st{};
    if (start) st = *start;
    if (assemble_tiled(g)) {
        const Tiles tw = make_tiles(g, nblk);
        const int nb = tile_blocks(tw, g, nblk);
        auto *fn = mode == ASM_CG64 ? k_assemble_tiled<ASM_CG64>
                                    : mode == ASM_MIXED ? k_assemble_tiled<ASM_MIXED> : k_assemble_tiled<ASM_ONLY>;
        fn<<<nb, RED_THREADS, 0, s>>>(g, tw, soils, zone, Ks, flags, sp, hk, hn, theta_k, theta_n, K, Can, c, b, Tx, Ty,
                                      Tz, diag, dinv, K32, cb32, dinv32, skip, st, partials, ticket, s0, theta_p);
        return;
    }
    auto *fn = mode == ASM_CG64 ? k_assemble<ASM_CG64> : mode == ASM_MIXED ? k_assemble<ASM_MIXED> : k_assemble<ASM_ONLY>;
    fn<<<nblk, RED_THREADS, 0, s>>>(g, soils, zone, Ks, flags, sp, hk, hn, theta_k, theta_n, K, Can, c, b, Tx, Ty, Tz,
                                    diag, dinv, K32, cb32, dinv32, skip, st, partials, ticket, s0, theta_p);
}

void launch_accept(cudaStream_t s, int nblk, const Grid &g, const double *x_final, double *h,
                   const double *theta_k, double *theta_n, const double *K1, double *K0, int copyK)
{
    k_accept<<<nblk, RED_THREADS, 0, s>>>(g, x_final, h, theta_k, theta_n, K1, K0, copyK);
}

void launch_mass_balance(cudaStream_t s, int nblk, const Grid &g, const DevSoil *soils, const uint8_t *zone,
                         const double *Ks, const uint8_t *flags, const StepParams *sp, const double *x_odd,
                         const double *x_even, const double *hn, const double *c, const double *K_odd,
                         const double *K_even, const double *theta_x, const double *theta_n, double *partials,
                         unsigned int *ticket, StepResults *res, const PicardCtl *ctl, const double *s0)
{
    k_mass_balance<<<nblk, RED_THREADS, 0, s>>>(g, soils, zone, Ks, flags, sp, x_odd, x_even, hn, c, K_odd, K_even,
                                                theta_x, theta_n, partials, ticket, res, ctl, s0);
}

void launch_storage(cudaStream_t s, int nblk, const Grid &g, const uint8_t *flags, const double *theta,
                    double *partials, unsigned int *ticket, StepResults *res)
{
    k_storage<<<nblk, RED_THREADS, 0, s>>>(g, flags, theta, partials, ticket, res);
}

}  // namespace rf
