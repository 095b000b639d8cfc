// sweeps.cuh -- stencil sweeps over z planes of column tiles, as device
// functions of the one-launch solves (cg_solve.cu) and of the single-phase
// kernels (pcg.cu).
//
// FP64 (product and outer residual): a block sweeps the z planes
// of 32 x 16 column tiles; a thread owns two y-adjacent cells.  The vector's
// value (p = z + beta p_old) is formed once per cell; x / y neighbours come from
// shared memory (the plane plus a one-cell halo, two buffers, one barrier a
// plane), z neighbours from registers.  Everything is loaded a plane (the
// cell's own vector: two planes) ahead.  Inactive cells need no mask: their
// diagonal and face coefficients, z and p are 0.
//
// FP32: 32 x 32 tiles, four y-adjacent cells a thread, faces
// recomputed from K (NaN on inactive cells and outside the grid, so that
// max(w (K_P + K_N), 0) closes their faces), each face between two of a
// thread's cells and each vertical face formed once.
#pragma once

#include "ix64.cuh"
#include "rf_internal.cuh"
#include "tiles.cuh"

namespace rf {

// Two blocks an SM: three (80 registers) time 5-10 % worse everywhere but on
// the largest FP64 product.
constexpr int SWEEP_OCC = 2;
constexpr int CX = 32, CY = 16, CT = 256;          // tile, threads (32 x 8, two rows each)
constexpr int CHALO = 2 * CY + 2 * CX;             // -x column, +x column, -y row, +y row

struct Sweep64Shared {
    double p[2][CY + 2][CX + 2];
    double ty[2][CY / 2 + 1][CX];                  // Ty of the row below each thread row
    double tx[2][CY];                              // Tx of the -x halo column
};
constexpr int FY = 32, FHALO = 2 * FY + 2 * CX;    // FP32 tile height (four rows a thread), its halo
struct Sweep32Shared {
    float p[2][FY + 2][CX + 2], K[2][FY + 2][CX + 2];
};

#ifdef __CUDACC__
// Halo cell h of a CX x ny tile, as offsets from its corner: -x column, +x
// column, -y row, +y row.
__device__ __forceinline__ void halo_of(int h, int ny, int &hx, int &hy)
{
    if (h < ny) { hx = -1; hy = h; }
    else if (h < 2 * ny) { hx = CX; hy = h - ny; }
    else if (h < 2 * ny + CX) { hx = h - 2 * ny; hy = -1; }
    else { hx = h - 2 * ny - CX; hy = ny; }
}

// The face coefficients of the FP64 operator.
struct Op64 {
    const double *Tx, *Ty, *Tz, *diag;
};

// Sweep of the FP64 operator over this block's items: value(c) is the vector
// at cell c as a pair of loads (a, b) combined by mix; out(c, v, Av, e) takes an
// in-grid cell's value and product, and what own(c) loaded a plane ahead.
struct NoOwn {};
template <class Raw, class Own, class Load, class Mix, class LoadOwn, class Out>
__device__ __forceinline__ void sweep64(const Grid &g, const Tiles &tw, const Op64 &A, Sweep64Shared &s, Load load,
                                        Mix mix, LoadOwn own, Out out)
{
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, h = threadIdx.x;
    int hx, hy;
    halo_of(h, CY, hx, hy);
    const long long sxy = g.sxy;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    for (long long item = blockIdx.x; item < tw.items; item += gridDim.x) {
        const TileItem t = tile_item(g, tw, item);
        const int i = t.i0 + tx, j = t.j0 + 2 * ty;
        const bool in0 = i < nx && j < ny, in1 = i < nx && j + 1 < ny;
        const long long col = i + (long long)nx * j;
        const bool halo = h < CHALO && t.i0 + hx >= 0 && t.i0 + hx < nx && t.j0 + hy >= 0 && t.j0 + hy < ny;
        const long long hcol = (t.i0 + hx) + (long long)nx * (t.j0 + hy);
        auto raw = [&](bool in, long long c, int k) {
            Raw a{};
            if (in && k >= 0 && k < nz) a = load(c + sxy * k);
            return a;
        };
        struct Coef {
            double d0, d1, x0, x1, y0, y1, z0, z1, hT;
            Raw h;
            Own e0, e1;
        };
        auto coef = [&](int k) {
            Coef a{};
            const long long c = col + sxy * k;
            if (in0) {
                a.d0 = __ldcs(&A.diag[c]);
                a.x0 = __ldcs(&A.Tx[c]);
                a.y0 = __ldcs(&A.Ty[c]);
                a.z0 = __ldcs(&A.Tz[c]);
                a.e0 = own(c);
            }
            if (in1) {
                a.d1 = __ldcs(&A.diag[c + nx]);
                a.x1 = __ldcs(&A.Tx[c + nx]);
                a.y1 = __ldcs(&A.Ty[c + nx]);
                a.z1 = __ldcs(&A.Tz[c + nx]);
                a.e1 = own(c + nx);
            }
            if (halo) {
                const long long hc = hcol + sxy * k;
                a.h = load(hc);
                if (hx == -1) a.hT = A.Tx[hc];
                if (hy == -1) a.hT = A.Ty[hc];
            }
            return a;
        };
        Raw rn0 = raw(in0, col, t.k0 + 1), rn1 = raw(in1, col + nx, t.k0 + 1);
        Coef nxt = coef(t.k0);
        double tzm0 = 0.0, tzm1 = 0.0;
        if (t.k0 > 0) {
            if (in0) tzm0 = A.Tz[col + sxy * (t.k0 - 1)];
            if (in1) tzm1 = A.Tz[col + nx + sxy * (t.k0 - 1)];
        }
        double pm0 = mix(raw(in0, col, t.k0 - 1)), pm1 = mix(raw(in1, col + nx, t.k0 - 1));
        double pc0 = mix(raw(in0, col, t.k0)), pc1 = mix(raw(in1, col + nx, t.k0));
        for (int k = t.k0; k < t.k1; k++) {
            const int b = k & 1;
            const Coef cur = nxt;
            const double pn0 = mix(rn0), pn1 = mix(rn1);
            s.p[b][2 * ty + 1][tx + 1] = pc0;
            s.p[b][2 * ty + 2][tx + 1] = pc1;
            s.ty[b][ty + 1][tx] = cur.y1;
            if (h < CHALO) {
                s.p[b][hy + 1][hx + 1] = mix(cur.h);
                if (hx == -1) s.tx[b][hy] = cur.hT;
                if (hy == -1) s.ty[b][0][hx] = cur.hT;
            }
            if (k + 1 < t.k1) {
                nxt = coef(k + 1);
                rn0 = raw(in0, col, k + 2);
                rn1 = raw(in1, col + nx, k + 2);
            }
            const double txm0l = __shfl_up_sync(0xffffffffu, cur.x0, 1);
            const double txm1l = __shfl_up_sync(0xffffffffu, cur.x1, 1);
            __syncthreads();
            const long long c = col + sxy * k;
            double a0 = 0.0, a1 = 0.0;
            // a warp without an active cell has only zeros
            // (tested on the bits: a compare would go to the FP64 pipe)
            const bool act0 = __double_as_longlong(cur.d0) != 0, act1 = __double_as_longlong(cur.d1) != 0;
            if (__any_sync(0xffffffffu, act0 || act1)) {
                const double txm0 = tx > 0 ? txm0l : s.tx[b][2 * ty], txm1 = tx > 0 ? txm1l : s.tx[b][2 * ty + 1];
                a0 = cur.d0 * pc0;
                a1 = cur.d1 * pc1;
                a0 = fma(-txm0, s.p[b][2 * ty + 1][tx], a0);
                a1 = fma(-txm1, s.p[b][2 * ty + 2][tx], a1);
                a0 = fma(-cur.x0, s.p[b][2 * ty + 1][tx + 2], a0);
                a1 = fma(-cur.x1, s.p[b][2 * ty + 2][tx + 2], a1);
                a0 = fma(-s.ty[b][ty][tx], s.p[b][2 * ty][tx + 1], a0);
                a1 = fma(-cur.y0, pc0, a1);
                a0 = fma(-cur.y0, pc1, a0);
                a1 = fma(-cur.y1, s.p[b][2 * ty + 3][tx + 1], a1);
                a0 = fma(-tzm0, pm0, a0);
                a1 = fma(-tzm1, pm1, a1);
                a0 = fma(-cur.z0, pn0, a0);
                a1 = fma(-cur.z1, pn1, a1);
            }
            if (in0) out(c, pc0, a0, act0, cur.e0);
            if (in1) out(c + nx, pc1, a1, act1, cur.e1);
            tzm0 = cur.z0;
            tzm1 = cur.z1;
            pm0 = pc0;
            pm1 = pc1;
            pc0 = pn0;
            pc1 = pn1;
        }
        __syncthreads();
    }
}

// The same cell by cell, for grids that do not fill a tile (narrow_grid): values
// of the neighbours are formed again, terms added in the same order.
template <class Own, class Value, class LoadOwn, class Out>
__device__ __forceinline__ void cells64(const Grid &g, const Op64 &A, Value value, LoadOwn own, Out out)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < g.N; c += stride) {
        int i, j, k;
        cell_ijk(g, c, i, j, k);
        const Own e = own(c);
        const double d = A.diag[c], v = value(c);
        const bool act = __double_as_longlong(d) != 0;
        double a = 0.0;
        if (act) {
            a = d * v;
            if (i > 0) a = fma(-A.Tx[c - 1], value(c - 1), a);
            if (i < g.nx - 1) a = fma(-A.Tx[c], value(c + 1), a);
            if (j > 0) a = fma(-A.Ty[c - g.nx], value(c - g.nx), a);
            if (j < g.ny - 1) a = fma(-A.Ty[c], value(c + g.nx), a);
            if (k > 0) a = fma(-A.Tz[c - g.sxy], value(c - g.sxy), a);
            if (k < g.nz - 1) a = fma(-A.Tz[c], value(c + g.sxy), a);
        }
        out(c, v, a, act, e);
    }
}

// FP32 stencil product cell by cell (as sweep32).
__device__ __forceinline__ float cells32(const Grid &g, const float *__restrict__ K32, const float *__restrict__ cb32,
                                         const float *z, const float *pin, float *pout, float *q, float beta,
                                         bool first)
{
    const float wx = g.w32[0] * 0.5f, wy = g.w32[1] * 0.5f, wz = g.w32[2] * 0.5f;
    float acc = 0.0f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < g.N; c += stride) {
        int i, j, k;
        cell_ijk(g, c, i, j, k);
        const float K = K32[c];
        auto value = [&](long long n) { return first ? z[n] : fmaf(beta, pin[n], z[n]); };
        float v = 0.0f, a = 0.0f;
        if (K >= 0.0f) {
            v = value(c);
            a = cb32[c] * v;
            auto face = [&](bool in, long long n, float w) {
                if (in) a = fmaf(fmaxf(w * (K + K32[n]), 0.0f), v - value(n), a);
            };
            face(i > 0, c - 1, wx);
            face(i < g.nx - 1, c + 1, wx);
            face(j > 0, c - g.nx, wy);
            face(j < g.ny - 1, c + g.nx, wy);
            face(k > 0, c - g.sxy, wz);
            face(k < g.nz - 1, c + g.sxy, wz);
        }
        pout[c] = v;
        q[c] = a;
        acc = fmaf(v, a, acc);
    }
    return acc;
}

// FP32 stencil product over this block's items: p = z + beta p_old, q = A p;
// returns this thread's p.q.
__device__ __forceinline__ float sweep32(const Grid &g, const Tiles &tw, Sweep32Shared &s, const float *__restrict__ K32,
                                         const float *__restrict__ cb32, const float *z, const float *pin, float *pout,
                                         float *q, float beta, bool first)
{
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, h = threadIdx.x;
    int hx, hy;
    halo_of(h, FY, hx, hy);
    const long long sxy = g.sxy;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const float wx = g.w32[0] * 0.5f, wy = g.w32[1] * 0.5f, wz = g.w32[2] * 0.5f;
    const float closed = __int_as_float(0x7fc00000);
    float acc = 0.0f;
    auto face = [](float kP, float pP, float kN, float pN, float w) {
        return fmaxf(w * (kP + kN), 0.0f) * (pP - pN);
    };
    for (long long item = blockIdx.x; item < tw.items; item += gridDim.x) {
        const TileItem t = tile_item(g, tw, item);
        const int i = t.i0 + tx, j = t.j0 + 4 * ty;
        const long long col = i + (long long)nx * j;
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; u++) in[u] = i < nx && j + u < ny;
        const bool halo = h < FHALO && t.i0 + hx >= 0 && t.i0 + hx < nx && t.j0 + hy >= 0 && t.j0 + hy < ny;
        const long long hcol = (t.i0 + hx) + (long long)nx * (t.j0 + hy);
        struct Raw {
            float z[4], o[4], K[4];
        };
        auto raw = [&](int k) {
            Raw a;
#pragma unroll
            for (int u = 0; u < 4; u++) {
                a.z[u] = a.o[u] = 0.0f;
                a.K[u] = closed;
                if (in[u] && k >= 0 && k < nz) {
                    const long long c = col + (long long)nx * u + sxy * k;
                    a.K[u] = K32[c];
                    a.z[u] = __ldcs(&z[c]);
                    if (!first) a.o[u] = __ldcs(&pin[c]);
                }
            }
            return a;
        };
        float pc[4], Kc[4], carry[4];
        {
            const Raw a = raw(t.k0 - 1), b = raw(t.k0);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                pc[u] = fmaf(beta, b.o[u], b.z[u]);
                Kc[u] = b.K[u];
                carry[u] = face(Kc[u], pc[u], a.K[u], fmaf(beta, a.o[u], a.z[u]), wz);
            }
        }
        Raw rn = raw(t.k0 + 1);
        float cbn[4], hz = 0.0f, ho = 0.0f, hK = closed;
        auto next = [&](int k) {
#pragma unroll
            for (int u = 0; u < 4; u++) cbn[u] = in[u] ? __ldcs(&cb32[col + (long long)nx * u + sxy * k]) : 0.0f;
            if (halo) {
                const long long hc = hcol + sxy * k;
                hK = K32[hc];
                hz = z[hc];
                if (!first) ho = pin[hc];
            }
        };
        next(t.k0);
        for (int k = t.k0; k < t.k1; k++) {
            const int b = k & 1;
            float cb[4], pn[4], Kn[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                cb[u] = cbn[u];
                pn[u] = fmaf(beta, rn.o[u], rn.z[u]);
                Kn[u] = rn.K[u];
                s.p[b][4 * ty + u + 1][tx + 1] = pc[u];
                s.K[b][4 * ty + u + 1][tx + 1] = Kc[u];
            }
            if (h < FHALO) {
                s.p[b][hy + 1][hx + 1] = fmaf(beta, ho, hz);
                s.K[b][hy + 1][hx + 1] = hK;
            }
            if (k + 1 < t.k1) {
                next(k + 1);
                rn = raw(k + 2);
            }
            __syncthreads();
            float qv[4], ym = face(Kc[0], pc[0], s.K[b][4 * ty][tx + 1], s.p[b][4 * ty][tx + 1], wy);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int row = 4 * ty + u + 1;
                const float tz = face(Kc[u], pc[u], Kn[u], pn[u], wz);
                const float yp = u < 3 ? face(Kc[u], pc[u], Kc[u < 3 ? u + 1 : 3], pc[u < 3 ? u + 1 : 3], wy)
                                       : face(Kc[3], pc[3], s.K[b][row + 1][tx + 1], s.p[b][row + 1][tx + 1], wy);
                float v = fmaf(cb[u], pc[u], carry[u]) + tz;
                v += face(Kc[u], pc[u], s.K[b][row][tx], s.p[b][row][tx], wx);
                v += face(Kc[u], pc[u], s.K[b][row][tx + 2], s.p[b][row][tx + 2], wx);
                v += ym + yp;
                ym = -yp;
                carry[u] = -tz;
                qv[u] = v;
            }
            const long long c = col + sxy * k;
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const bool act = Kc[u] >= 0.0f;
                const float po = act ? pc[u] : 0.0f, qo = act ? qv[u] : 0.0f;
                acc = fmaf(po, qo, acc);
                if (in[u]) {
                    pout[c + (long long)nx * u] = po;
                    q[c + (long long)nx * u] = qo;
                }
                pc[u] = pn[u];
                Kc[u] = Kn[u];
            }
        }
        __syncthreads();
    }
    return acc;
}

// x += alpha p, r -= alpha q, z = D^-1 r over this block's share, two cells a
// load; v accumulates r.r and r.z.  Inactive cells (dinv, p, q, r 0) keep
// their values.  The arrays that the next sweep does not read are streamed
// (evict first): z, p and q are what L2 should hold between the two.
__device__ __forceinline__ void cg64_update_cells(const Grid &g, double alpha, const double *__restrict__ dinv,
                                                  const double *pd, const double *q, double *x, double *r, double *z,
                                                  double (&v)[2])
{
    auto cell = [&](double di, double pv, double qv, double &xv, double &rv, double &zv) {
        xv = fma(alpha, pv, xv);
        rv = fma(-alpha, qv, rv);
        zv = di * rv;
        v[0] = fma(rv, rv, v[0]);
        v[1] = fma(rv, zv, v[1]);
    };
    const long long n2 = g.N / 2, stride = (long long)gridDim.x * blockDim.x;
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < n2; u += stride) {
        const double2 di = __ldcs(reinterpret_cast<const double2 *>(dinv) + u);
        const double2 pv = reinterpret_cast<const double2 *>(pd)[u];
        const double2 qv = __ldcs(reinterpret_cast<const double2 *>(q) + u);
        double2 xv = __ldcs(reinterpret_cast<double2 *>(x) + u), rv = __ldcs(reinterpret_cast<double2 *>(r) + u), zv;
        cell(di.x, pv.x, qv.x, xv.x, rv.x, zv.x);
        cell(di.y, pv.y, qv.y, xv.y, rv.y, zv.y);
        __stcs(reinterpret_cast<double2 *>(x) + u, xv);
        __stcs(reinterpret_cast<double2 *>(r) + u, rv);
        reinterpret_cast<double2 *>(z)[u] = zv;
    }
    if ((g.N & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
        const long long c = g.N - 1;
        double xv = x[c], rv = r[c], zv;
        cell(dinv[c], pd[c], q[c], xv, rv, zv);
        x[c] = xv;
        r[c] = rv;
        z[c] = zv;
    }
}

// The same in FP32, four cells a load; fresh: d is 0 and not read.
__device__ __forceinline__ void cg32_update_cells(const Grid &g, float alpha, bool fresh,
                                                  const float *__restrict__ dinv, const float *pd, const float *q,
                                                  float *d, float *r, float *z, float (&v)[2])
{
    auto cell = [&](float di, float pv, float qv, float &dv, float &rv, float &zv) {
        dv = fmaf(alpha, pv, dv);
        rv = fmaf(-alpha, qv, rv);
        zv = di * rv;
        v[0] = fmaf(rv, rv, v[0]);
        v[1] = fmaf(rv, zv, v[1]);
    };
    const long long n4 = g.N / 4, stride = (long long)gridDim.x * blockDim.x;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long u = t0; u < n4; u += stride) {
        const float4 di = __ldcs(reinterpret_cast<const float4 *>(dinv) + u);
        const float4 pv = reinterpret_cast<const float4 *>(pd)[u];
        const float4 qv = __ldcs(reinterpret_cast<const float4 *>(q) + u);
        float4 rv = reinterpret_cast<float4 *>(r)[u], zv, dv = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (!fresh) dv = __ldcs(reinterpret_cast<float4 *>(d) + u);
        cell(di.x, pv.x, qv.x, dv.x, rv.x, zv.x);
        cell(di.y, pv.y, qv.y, dv.y, rv.y, zv.y);
        cell(di.z, pv.z, qv.z, dv.z, rv.z, zv.z);
        cell(di.w, pv.w, qv.w, dv.w, rv.w, zv.w);
        __stcs(reinterpret_cast<float4 *>(d) + u, dv);
        reinterpret_cast<float4 *>(r)[u] = rv;
        reinterpret_cast<float4 *>(z)[u] = zv;
    }
    for (long long c = 4 * n4 + t0; c < g.N; c += stride) {
        float dv = fresh ? 0.0f : d[c], rv = r[c], zv;
        cell(dinv[c], pd[c], q[c], dv, rv, zv);
        d[c] = dv;
        r[c] = rv;
        z[c] = zv;
    }
}

// FP64 residual r = b - A x over this block's items as FP32 seeds r32 and
// z32 = D^-1 r32 (d32, when given, becomes 0); v accumulates r.r, b.b and r.z
// of the seeds in FP32.  b and D^-1 are loaded with the coefficients: loaded
// where they are used, behind the plane's barrier, they cost a memory latency
// a plane (384 x 320 x 64 cells, 6.1 M active: 238.6 -> 180.6 us; its 8 FP64
// instructions a cell alone take 78).
template <bool NARROW>
__device__ __forceinline__ void resid64_sweep(const Grid &g, const Tiles &tw, const Op64 &A, Sweep64Shared &s,
                                              const uint8_t *__restrict__ flags, const double *x,
                                              const double *__restrict__ b, const float *__restrict__ dinv32,
                                              float *r32, float *z32, float *d32, float (&v)[3])
{
    struct Raw {
        double x;
        uint8_t fl;
    };
    struct Own {
        double b;
        float di;
    };
    auto own = [&](long long c) { return Own{__ldcs(&b[c]), __ldcs(&dinv32[c])}; };
    // an inactive cell's head may be anything; its faces' T = 0 needs a number
    auto mix = [&](const Raw &a) { return (a.fl & FLAG_ACTIVE) ? a.x : 0.0; };
    auto load = [&](long long c) { return Raw{x[c], flags[c]}; };
    auto out = [&](long long c, double, double Ax, bool act, const Own &e) {
        float rf = 0.0f, zf = 0.0f;
        if (act) {
            const double rp = e.b - Ax;
            const float bf = ix_d2f(e.b);
            rf = ix_d2f(rp);
            zf = e.di * rf;
            v[0] = fmaf(rf, rf, v[0]);
            v[1] = fmaf(bf, bf, v[1]);
            v[2] = fmaf(rf, zf, v[2]);
        }
        r32[c] = rf;
        z32[c] = zf;
        if (d32) d32[c] = 0.0f;
    };
    if (NARROW) cells64<Own>(g, A, [&](long long c) { return mix(load(c)); }, own, out);
    else sweep64<Raw, Own>(g, tw, A, s, load, mix, own, out);
}

#endif

}  // namespace rf
