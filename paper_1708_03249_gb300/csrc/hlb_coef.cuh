// Equilibrium factor lines in double-float (FP32 groups with equilibrium
// orders up to 15): the coefficient recurrences of the half- and full-range
// projections (App. A, Eqs. "eq:hh_gk", "eq:H_gk") and their compensated dot
// products with the quadrature tables.  Used by the node pass (hlb_node.cu)
// and the persistent batched kernel (hlb_persist.cu).
#pragma once

#include <cuda_runtime.h>

#include "hlb_device.cuh"
#include "hlb_internal.h"

namespace hlb {

// The sizes factor_line_df reads, copied out of a GroupDev (a small value to
// pass to a function that is not inlined).
struct FactorDims {
    int Nx, Ny, Nz, Qx, QX2, VY, VZ, ncp, Qy, Qz, x_full;
    float2 m_om0f;
    __device__ explicit FactorDims(const GroupDev& g)
        : Nx(g.Nx), Ny(g.Ny), Nz(g.Nz), Qx(g.Qx), QX2(g.QX2), VY(g.VY), VZ(g.VZ), ncp(g.ncp), Qy(g.Qy), Qz(g.Qz),
          x_full(g.x_full), m_om0f(g.m_om0f) {}
};

// FP32 groups whose equilibrium orders are all below NM (double-float path,
// orders up to 15): one thread per node, coefficients in registers.  The FP64 prelude (erf,
// exp, sqrt) runs once per node on full warps; each role's recurrence is
// followed at once by its dot products with the quadrature tables (broadcast
// reads from shared memory); a warp's 32 factor lines are assembled in shared
// memory and written out contiguously.
template <int NM>
__device__ __forceinline__ void half_range_G_df(int r, const NodeDF& in, const float2* recf, int Nx, float2 m_om0,
                                                float2 (&G)[NM]) {
    const float2* ra = recf;
    const float2* rb = recf + Nx;
    const float2* rc = recf + 2 * Nx;
    const float2* h0 = recf + 3 * Nx;
    const float2* inv_ra = recf + 4 * Nx + 1;
    const float sg = r ? -1.0f : 1.0f;
    const float2 us = make_float2(sg * in.ux.x, sg * in.ux.y);
    const float2 half = df_add(make_float2(0.5f, 0.0f), make_float2(0.5f * sg * in.erf_z.x, 0.5f * sg * in.erf_z.y));
    G[0] = df_mul(h0[0], half);
    float2 S = make_float2(0.0f, 0.0f), gm1 = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int l = 0; l < NM - 1; ++l) {
        if (l < Nx) {
            float2 ig = df_mul(df_mul(m_om0, h0[l]), S);
            if (l) ig = df_add(ig, df_mul(gm1, inv_ra[l - 1]));
            const float2 pg = df_add(df_mul(us, G[l]), df_mul(in.T, df_add(df_mul(in.g0, h0[l]), ig)));
            G[l + 1] = df_add(df_add(df_mul(ra[l], pg), df_mul(rb[l], G[l])), df_mul(rc[l], gm1));
            S = df_add(S, df_mul(h0[l], G[l]));
            gm1 = G[l];
        }
    }
}

template <int NM>
__device__ __forceinline__ void full_range_G_df(float2 u, float2 Tm1, int N, float2 (&G)[NM]) {
    G[0] = make_float2(1.0f, 0.0f);
    G[1] = u;
#pragma unroll
    for (int l = 1; l < NM - 1; ++l)
        if (l < N) G[l + 1] = df_add(df_mul(u, G[l]), df_mul(df_mul(make_float2((float)l, 0.0f), Tm1), G[l - 1]));
}

// Two dot products at once (table rows 2k and 2k+1, one per lane of the f32x2
// registers) with the same double-float coefficients G, by the compensated
// dot product Dot2 of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26, 2005):
// TwoProduct of the high parts, TwoSum into the running sum, the rounding
// errors and the products with the low parts of the table and of G summed in
// the error term.  The result is as accurate as a double-float evaluation
// (about twice the FP32 precision, times the condition number) at a third of
// its instructions.  P[l] = (T_2k,l hi, T_2k+1,l hi, T_2k,l lo, T_2k+1,l lo).
template <int NM>
__device__ __forceinline__ void dot2_pair(const float4* P, const float2 (&G)[NM], int N, float2& r0, float2& r1) {
    float2 acc = f2(0.0f), err = f2(0.0f);
#pragma unroll
    for (int l = 0; l < NM; ++l) {
        if (l <= N) {
            const float4 t = P[l];
            const float2 th = make_float2(t.x, t.y), tl = make_float2(t.z, t.w);
            const float2 gh = f2(G[l].x), gl = f2(G[l].y);
            const float2 q = __fmul2_rn(th, f2(-G[l].x));        // -p, p = fl(th gh)
            const float2 e = __ffma2_rn(th, gh, q);               // th gh - p, exact
            const float2 sum = fsub2(acc, q);                     // acc + p
            const float2 bb = fsub2(sum, acc);
            const float2 t2 = fsub2(fsub2(acc, fsub2(sum, bb)), __fadd2_rn(q, bb));   // (acc + p) - sum, exact
            acc = sum;
            err = __fadd2_rn(err, __fadd2_rn(t2, e));
            err = __ffma2_rn(th, gl, __ffma2_rn(tl, gh, err));
        }
    }
    r0 = df_add(make_float2(acc.x, 0.0f), make_float2(err.x, 0.0f));
    r1 = df_add(make_float2(acc.y, 0.0f), make_float2(err.y, 0.0f));
}

// line[k] = (row k of a paired table . G) (times scale when given), k < nrows
template <int NM>
__device__ __forceinline__ void lines_dot2(float* line, const float4* P, int nrows, const float2 (&G)[NM], int N,
                                           const float2* scale) {
    for (int k = 0; k < nrows; k += 2) {
        float2 v0, v1;
        dot2_pair<NM>(P + (k >> 1) * (N + 1), G, N, v0, v1);
        if (scale) { v0 = df_mul(v0, *scale); v1 = df_mul(v1, *scale); }
        line[k] = v0.x + v0.y;
        if (k + 1 < nrows) line[k + 1] = v1.x + v1.y;
    }
}

// The factor line { n g_x (2Qx), g_y (VY), g_z (VZ), 1/tau, zeros to ncp } of
// one node from its n, u, T (FP64) and 1/tau; sPx, sPy, sPz the paired tables
// (dot2_pair layout), sRec the double-float recurrence table.  GD is GroupDev
// or FactorDims (the fields read here).
template <int NM, typename GD>
__device__ __forceinline__ void factor_line_df_in(const GD& g, const NodeDF& in, double itau, const float4* sPx,
                                                  const float4* sPy, const float4* sPz, const float2* sRec,
                                                  float* line) {
    const int Nx = g.Nx, Ny = g.Ny, Nz = g.Nz, Qx = g.Qx, QX2 = g.QX2, VY = g.VY, VZ = g.VZ, ncp = g.ncp;
    for (int o = QX2 + VY + VZ; o < ncp; ++o) line[o] = 0.0f;
    line[QX2 + VY + VZ] = (float)itau;
    if (itau == 0.0) {
        for (int o = 0; o < QX2 + VY + VZ; ++o) line[o] = 0.0f;
        return;
    }
    float2 G[NM];
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {                    // n g_x, p_x > 0 then p_x < 0
        if (g.x_full)                                 // full-range p_x: G_l(+-u_x)
            full_range_G_df<NM>(r ? make_float2(-in.ux.x, -in.ux.y) : in.ux, in.Tm1, Nx, G);
        else
            half_range_G_df<NM>(r, in, sRec, Nx, g.m_om0f, G);
        lines_dot2<NM>(line + r * Qx, sPx, Qx, G, Nx, &in.n);
    }
    if (g.Qy) {
        full_range_G_df<NM>(in.uy, in.Tm1, Ny, G);
        lines_dot2<NM>(line + QX2, sPy, VY, G, Ny, nullptr);
    } else {
        line[QX2] = 1.0f;
    }
    if (g.Qz) {
        full_range_G_df<NM>(in.uz, in.Tm1, Nz, G);
        lines_dot2<NM>(line + QX2 + VY, sPz, VZ, G, Nz, nullptr);
    } else {
        line[QX2 + VY] = 1.0f;
    }
}

template <int NM, typename GD>
__device__ __forceinline__ void factor_line_df(const GD& g, double n, double ux, double uy, double uz, double T,
                                               double itau, const float4* sPx, const float4* sPy, const float4* sPz,
                                               const float2* sRec, float* line) {
    NodeDF in;
    if (itau != 0.0) node_inputs_df(n, ux, uy, uz, T, g.Nx, in);
    factor_line_df_in<NM>(g, in, itau, sPx, sPy, sPz, sRec, line);
}

// s + e = a + b exactly (TwoSum), whatever the magnitudes.
__device__ __forceinline__ float2 df_two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return make_float2(s, (a - (s - bb)) + (b - bb));
}

// 1/x in double-float: the FP32 reciprocal refined by one Newton step
// (r + r (1 - x r), the residual formed exactly enough in double-float).
__device__ __forceinline__ float2 df_recip(float2 x) {
    const float r = 1.0f / x.x;
    const float2 res = df_add(make_float2(1.0f, 0.0f), df_mul(make_float2(-x.x, -x.y), make_float2(r, 0.0f)));
    return df_add(make_float2(r, 0.0f), df_mul(make_float2(r, 0.0f), res));
}

// sqrt(x) in double-float (x > 0): the FP32 root s refined by one Newton step
// s + (x - s^2) / (2 s), with s^2 by TwoProduct.
__device__ __forceinline__ float2 df_sqrt(float2 x) {
    const float s = sqrtf(x.x);
    const float p = s * s, e = fmaf(s, s, -p);
    const float2 res = df_add(x, make_float2(-p, -e));
    return df_fast_two_sum(s, res.x / (2.0f * s));
}

// exp(y) and (sqrt(pi) / 2) erf(z) / z = sum_n y^n / (n! (2n + 1)) for y = -z^2 in
// [-0.49, 0], their Taylor polynomials by Horner's rule: the flows' own range,
// |u_x| up to sqrt(2 T) 0.7, where neither needs a reduction.
// In double-float, both at once in the lanes of f32x2 registers, the terms from
// degree 9 on (5e-9 of the sum) in FP32; degree 14 leaves 1e-17.
__device__ __forceinline__ DF2 df2_exp_erf_small(float2 y) {
    const float ch[15][2] = {
        {1.0f, 1.0f}, {1.0f, 0.3333333432674408f}, {0.5f, 0.10000000149011612f}, {0.1666666716337204f,
        0.02380952425301075f}, {0.0416666679084301f, 0.004629629664123058f}, {0.008333333767950535f,
        0.0007575757335871458f}, {0.0013888889225199819f, 0.00010683760774554685f}, {0.00019841270113829523f,
        1.3227513591118623e-05f}, {2.4801587642286904e-05f, 1.4589169268219848e-06f},
        {2.7557318844628753e-06f, 1.4503852696634567e-07f}, {2.755731998149713e-07f, 1.3122533282228233e-08f},
        {2.5052107943679403e-08f, 1.0892221569136495e-09f}, {2.0876755879584152e-09f, 8.350702768167295e-11f},
        {1.6059044372074283e-10f, 5.94779390669653e-12f}, {1.147074536050896e-11f, 3.9554294626979736e-13f}};
    const float cl[9][2] = {
        {0.0f, 0.0f}, {0.0f, -9.934107758624577e-09f}, {0.0f, -1.4901161415892261e-09f},
        {-4.967053879312289e-09f, -4.434869416147791e-10f}, {-1.2417634698280722e-09f,
        -3.449342894645824e-11f}, {-4.34617203337595e-10f, 2.3988611444480945e-11f},
        {-3.3631094437103215e-11f, -9.079400100676926e-13f}, {-2.725596874933456e-12f,
        -3.6360538603445736e-13f}, {-3.40699609366682e-13f, -2.672861423565296e-14f}};
    float2 t = make_float2(ch[14][0], ch[14][1]);
#pragma unroll
    for (int n = 13; n >= 9; --n) t = __ffma2_rn(t, f2(y.x), make_float2(ch[n][0], ch[n][1]));
    const DF2 yy = df2_dup(y);
    DF2 s = {t, f2(0.0f)};
#pragma unroll
    for (int n = 8; n >= 0; --n)
        s = df2_add(df2_mul(s, yy), DF2{make_float2(ch[n][0], ch[n][1]), make_float2(cl[n][0], cl[n][1])});
    return s;
}
// In FP64 (degree 15 leaves 5e-19).
__device__ __forceinline__ void exp_erf_small(double y, double& e, double& f) {
    const double c[16] = {
        1.0 / 1.0, 1.0 / 1.0, 1.0 / 2.0, 1.0 / 6.0, 1.0 / 24.0, 1.0 / 120.0, 1.0 / 720.0, 1.0 / 5040.0, 1.0 /
        40320.0, 1.0 / 362880.0, 1.0 / 3628800.0, 1.0 / 39916800.0, 1.0 / 479001600.0, 1.0 / 6227020800.0, 1.0
        / 87178291200.0, 1.0 / 1307674368000.0};
    const double d[16] = {
        1.0 / 1.0, 1.0 / 3.0, 1.0 / 10.0, 1.0 / 42.0, 1.0 / 216.0, 1.0 / 1320.0, 1.0 / 9360.0, 1.0 / 75600.0,
        1.0 / 685440.0, 1.0 / 6894720.0, 1.0 / 76204800.0, 1.0 / 918086400.0, 1.0 / 11975040000.0, 1.0 /
        168129561600.0, 1.0 / 2528170444800.0, 1.0 / 40537905408000.0};
    e = c[15];
    f = d[15];
#pragma unroll
    for (int n = 14; n >= 0; --n) {
        e = fma(e, y, c[n]);
        f = fma(f, y, d[n]);
    }
}

// The per-node inputs of the recurrences (NodeDF) from the compensated FP32
// moment sums (running sum and error term of n, j_x, j_y, j_z, E at sm[0..4]
// and sm[8..12]): n = s + c, u = j / n, T = (E - n |u|^2) / (D n) in
// double-float, relative error about 1e-14.  The recurrence grows an error of
// its start, exp(-u_x^2 / 2T) and erf(u_x / sqrt(2T)) against the u and T it
// runs with, about threefold per order.  LOW (equilibrium orders up to 10):
// both in double-float (1e-14 stays below FP32 resolution there; FP64 where
// |u_x| / sqrt(2T) > 2.5).  Else in FP64 from the double-float u and T as they
// stand, 1 / sqrt(T) by one third-order Householder step on the FP32 root (the
// FP64 pipe runs at 1/64 of FP32 here, so it takes only what needs it).  Returns n (FP64) for 1/tau.
template <bool LOW>
__device__ inline double node_inputs_from_sums_df(const float* sm, int D, NodeDF& o) {
    const float2 n = df_two_sum(sm[0], sm[8]);
    const float2 in = df_recip(n);
    const float2 ux = df_mul(df_two_sum(sm[1], sm[9]), in), uy = df_mul(df_two_sum(sm[2], sm[10]), in),
                 uz = df_mul(df_two_sum(sm[3], sm[11]), in);
    const float2 u2 = df_add(df_add(df_mul(ux, ux), df_mul(uy, uy)), df_mul(uz, uz));
    const float2 E = df_two_sum(sm[4], sm[12]);
    float2 T = df_mul(df_add(E, df_mul(make_float2(-n.x, -n.y), u2)), in);
    if (D == 3) T = df_mul(T, make_float2(0.3333333432674408f, -9.934107758624577e-09f));   // 1/3
    else if (D == 2) T = make_float2(0.5f * T.x, 0.5f * T.y);
    o.n = n;
    o.ux = ux;
    o.uy = uy;
    o.uz = uz;
    o.T = T;
    o.Tm1 = df_add(T, make_float2(-1.0f, 0.0f));
    if constexpr (LOW) {
        const float2 irt = df_recip(df_sqrt(T));
        const float2 z = df_mul(ux, df_mul(irt, make_float2(0.7071067690849304f, 1.2101617485882343e-08f)));
        const float2 inv_sqrt2pi = make_float2(0.3989422917366028f, -1.1335170135851058e-08f);
        if (fabsf(z.x) <= 0.7f) {
            const float2 z2 = df_mul(z, z);
            const DF2 p = df2_exp_erf_small(make_float2(-z2.x, -z2.y));
            o.g0 = df_mul(df_mul(make_float2(p.h.x, p.l.x), inv_sqrt2pi), irt);
            o.erf_z = df_mul(df_mul(z, make_float2(1.128379225730896f, -5.8635382771399236e-08f)),      // 2 / sqrt(pi)
                             make_float2(p.h.y, p.l.y));
        } else if (fabsf(z.x) <= 2.5f) {
            const float2 z2 = df_mul(z, z);
            const float2 Ez = df_exp_nonpos(make_float2(-z2.x, -z2.y));
            o.erf_z = df_erf_series(z, z2, Ez);
            o.g0 = df_mul(df_mul(Ez, inv_sqrt2pi), irt);
        } else {
            const double zd = (double)z.x + (double)z.y;
            o.erf_z = df_from_double(erf(zd));
            o.g0 = df_mul(df_mul(df_from_double(exp(-zd * zd)), inv_sqrt2pi), irt);
        }
    } else {
        const double Td = (double)T.x + (double)T.y, ud = (double)ux.x + (double)ux.y;
        double r = (double)rsqrtf(T.x);
        const double e = fma(-Td * r, r, 1.0);                   // 1 - T r^2, about 1e-7
        r = fma(r * e, fma(0.375, e, 0.5), r);                   // error 5/16 e^3
        const double z = ud * r * 0.70710678118654752440;
        double E, F;
        if (fabs(z) <= 0.7) {
            exp_erf_small(-z * z, E, F);
            F *= z * 1.1283791670955125739;                      // 2 / sqrt(pi)
        } else {
            E = exp(-z * z);
            F = erf(z);
        }
        o.erf_z = df_from_double(F);
        o.g0 = df_from_double(E * (r * (1.0 / kSqrt2Pi)));
    }
    return (double)n.x + (double)n.y;
}

// ---------------------------------------------------------------------------
// The factor lines of up to NB nodes by one CTA of T threads.  The three parts
// of a line's arithmetic (inputs, recurrences, dot products) are chains of
// dependent double-float operations; with one thread per node doing all of
// them in a row the pass waits on latency (71 us for the 65536 nodes of order
// 15 of the 256^2 box, where the instructions alone take about 20).  Here thread
// t works on node t % NB, and every double-float operation on two values in
// the lanes of f32x2 registers:
//  - recurrences: G^+ with G^- (slot 0), G_y with G_z (a slot of the next warp), a
//    thread per node and pair; the coefficients go to shared memory;
//  - dot products (Dot2 of Ogita, Rump and Oishi, as in dot2_pair), items of two
//    rows over all threads of the node: n g_x of +z_k with that of -z_k (one
//    table entry for both lanes); along p_y and p_z the even orders in one lane
//    and the odd ones in the other, since He_l(-z) = (-1)^l He_l(z) makes the
//    rows of z and -z the sum and the difference of the two: half the terms.
// ---------------------------------------------------------------------------
constexpr int kNodeFields = 9;           // float2 fields of a node's inputs, [field][NB]

// Shared-memory tables (float4 each) and coefficients of node_lines, in bytes.
struct NodeTables {
    int nx, ny, nz;                      // entries: x row pairs, y and z rows of (even, odd) pairs
    int my, mz;                          // (even, odd) pairs per row
    __host__ __device__ NodeTables(const GroupDev& g) {
        my = (g.Ny + 2) >> 1;
        mz = (g.Nz + 2) >> 1;
        nx = (g.Qx >> 1) * (g.Nx + 1);
        ny = g.Qy ? (g.VY >> 1) * my : 0;
        nz = g.Qz ? (g.VZ >> 1) * mz : 0;
    }
    __host__ __device__ size_t table_bytes() const { return (size_t)(nx + ny + nz) * 16; }
    template <int NB> __host__ __device__ size_t coef_bytes(const GroupDev& g) const {
        return (size_t)NB * 16 * (g.Nx + 1 + (g.Qy ? my : 0) + (g.Qz ? mz : 0));
    }
};
__host__ __device__ inline int node_line_stride(int ncp) { return (ncp / 4) & 1 ? ncp : ncp + 4; }   // few bank conflicts

__device__ __forceinline__ void node_load_tables(const GroupDev& g, const NodeTables& nt, float4* tab, int t, int T) {
    const float2* Tx = g.Tf;
    const float2* Ty = Tx + g.Qx * (g.Nx + 1);
    const float2* Tz = Ty + g.VY * (g.Ny + 1);
    for (int i = t; i < nt.nx; i += T) {                 // rows 2 k and 2 k + 1 side by side
        const int k = i / (g.Nx + 1), l = i - k * (g.Nx + 1);
        const float2 a = Tx[2 * k * (g.Nx + 1) + l], b = Tx[(2 * k + 1) * (g.Nx + 1) + l];
        tab[i] = make_float4(a.x, b.x, a.y, b.y);
    }
    auto pairs = [&](float4* dst, const float2* src, int half, int N, int m) {     // rows half .. 2 half - 1: z > 0
        for (int i = t; i < half * m; i += T) {
            const int j = i / m, l = 2 * (i - j * m);
            const float2 a = src[(half + j) * (N + 1) + l];
            const float2 b = l < N ? src[(half + j) * (N + 1) + l + 1] : make_float2(0.0f, 0.0f);
            dst[i] = make_float4(a.x, b.x, a.y, b.y);
        }
    };
    if (nt.ny) pairs(tab + nt.nx, Ty, g.VY >> 1, g.Ny, nt.my);
    if (nt.nz) pairs(tab + nt.nx + nt.ny, Tz, g.VZ >> 1, g.Nz, nt.mz);
}

// The half-range recurrence's table for node_lines, three float4 per order l
// (at least one): (a_l, b_l), (c_l, a_l d_l), (h_l(0), a_l h_l(0)) in
// double-float, d_0 = 0 (recf: a, b, c [Nx], h(0) [Nx + 1], d_1 .. d_Nx).
__host__ __device__ inline size_t node_rec_bytes(int Nx) { return (size_t)(Nx > 0 ? Nx : 1) * 48; }
__device__ __forceinline__ void node_load_rec(const GroupDev& g, float4* rec, int t, int T) {
    const int Nx = g.Nx;
    const float2* r = g.recf;
    for (int l = t; l < (Nx > 0 ? Nx : 1); l += T) {
        const float2 h = r[3 * Nx + l], zero = make_float2(0.0f, 0.0f);
        const float2 a = Nx ? r[l] : zero, b = Nx ? r[Nx + l] : zero, c = Nx ? r[2 * Nx + l] : zero;
        const float2 ad = l ? df_mul(a, r[4 * Nx + l]) : zero, ah = df_mul(a, h);
        rec[3 * l] = make_float4(a.x, a.y, b.x, b.y);
        rec[3 * l + 1] = make_float4(c.x, c.y, ad.x, ad.y);
        rec[3 * l + 2] = make_float4(h.x, h.y, ah.x, ah.y);
    }
}

// Two dot products per lane with the coefficients G[2 l NB] (high parts) and
// G[(2 l + 1) NB] (low parts), l < n, as double-floats: of p_x rows 2 k and
// 2 k + 1 with G^+ and G^- in the lanes (x: P0 the pair's entries), or of two
// p_y or p_z rows, the even and the odd orders in the lanes.
template <int NB>
__device__ __forceinline__ void dot2_rows(bool x, const float4* P0, const float4* P1, const float2* G, int n, DF2& r0,
                                          DF2& r1) {
    float2 a0 = f2(0.0f), e0 = f2(0.0f), a1 = f2(0.0f), e1 = f2(0.0f);
#pragma unroll 2
    for (int l = 0; l < n; ++l) {
        const float2 gh = G[2 * l * NB], gl = G[(2 * l + 1) * NB];
        const float2 ng = fsub2(f2(0.0f), gh);
        auto term = [&](const float2 th, const float2 tl, float2& acc, float2& err) {
            const float2 q = __fmul2_rn(th, ng);                  // -p, p = fl(th gh)
            const float2 e = __ffma2_rn(th, gh, q);               // th gh - p, exact
            const float2 sum = fsub2(acc, q);                     // acc + p
            const float2 bb = fsub2(sum, acc);
            const float2 t2 = fsub2(fsub2(acc, fsub2(sum, bb)), __fadd2_rn(q, bb));   // (acc + p) - sum, exact
            acc = sum;
            err = __fadd2_rn(err, __fadd2_rn(t2, e));
            err = __ffma2_rn(th, gl, __ffma2_rn(tl, gh, err));
        };
        const float4 u = P0[l], w = P1[l];
        term(x ? f2(u.x) : make_float2(u.x, u.y), x ? f2(u.z) : make_float2(u.z, u.w), a0, e0);
        term(x ? f2(w.y) : make_float2(w.x, w.y), x ? f2(w.w) : make_float2(w.z, w.w), a1, e1);
    }
    r0 = df2_add(DF2{a0, f2(0.0f)}, DF2{e0, f2(0.0f)});
    r1 = df2_add(DF2{a1, f2(0.0f)}, DF2{e1, f2(0.0f)});
}

// sIn: the inputs of node k (its NodeDF; 1/tau as the .x of field 8), written
// before a CTA barrier; tab, nt: node_load_tables; rec: node_load_rec; sG:
// coef_bytes; sLine: [NB][node_line_stride(ncp)].  Ends with the first QX2 + VY
// + VZ values of every line written, before a CTA barrier.  The loops stay
// rolled: a CTA runs this code once, and unrolled it spent more time on
// fetching instructions than on running them.
template <int NB, int T>
__device__ __forceinline__ void node_lines(const GroupDev& g, const NodeTables& nt, const float2* sIn, float2* sG,
                                           float* sLine, const float4* tab, const float4* rec) {
    constexpr int SLOTS = T / NB;
    const int k = threadIdx.x % NB, slot = threadIdx.x / NB;
    const int Nx = g.Nx, Ny = g.Ny, Nz = g.Nz, Qx = g.Qx, QX2 = g.QX2, VY = g.VY, VZ = g.VZ;
    auto in = [&](int f) { return sIn[f * NB + k]; };       // NodeDF order: ux uy uz T Tm1 erf_z g0 n, then (1/tau, -)
    const bool active = in(8).x != 0.0f;
    float2* Gx = sG + k;                                    // [l][h, l][NB]: lanes (+z, -z)
    float2* Gy = Gx + 2 * (Nx + 1) * NB;                    // [pair][h, l][NB]: lanes (even, odd)
    float2* Gz = Gy + (g.Qy ? 2 * nt.my * NB : 0);
    // 1. coefficients
    if (active && slot == 0) {
        auto put = [&](int l, const DF2& v) {
            Gx[2 * l * NB] = v.h;
            Gx[(2 * l + 1) * NB] = v.l;
        };
        if (!g.x_full) {
            // half_range_G_df's recurrence with its coefficients gathered:
            //   G_{l+1} = (a_l u + b_l) G_l + (c_l + a_l d_l T) G_{l-1} + a_l h_l(0) W_l,
            //   W_l = T (g(0) - omega(0) sum_{s<l} h_s(0) G_s),
            // so that G_l enters G_{l+1} through one product and one sum
            const float2 ux = in(0), er = in(5);
            const DF2 Tn = df2_dup(in(3)), us = {make_float2(ux.x, -ux.x), make_float2(ux.y, -ux.y)};
            const DF2 kap = df2_dup(df_mul(g.m_om0f, in(3)));
            const float2 hp = df_add(make_float2(0.5f, 0.0f), make_float2(0.5f * er.x, 0.5f * er.y));
            const float2 hm = df_add(make_float2(0.5f, 0.0f), make_float2(-0.5f * er.x, -0.5f * er.y));
            const float2 h00 = make_float2(rec[2].x, rec[2].y);
            DF2 cur = df2_mul(df2_dup(h00), DF2{make_float2(hp.x, hm.x), make_float2(hp.y, hm.y)});
            DF2 W = df2_dup(df_mul(in(3), in(6))), gm1 = {f2(0.0f), f2(0.0f)};
            put(0, cur);
#pragma unroll 1
            for (int l = 0; l < Nx; ++l) {
                const float4 ab = rec[3 * l], cd = rec[3 * l + 1], hh = rec[3 * l + 2];
                const DF2 al = df2_add(df2_mul(DF2{f2(ab.x), f2(ab.y)}, us), DF2{f2(ab.z), f2(ab.w)});
                const DF2 be = df2_add(df2_mul(DF2{f2(cd.z), f2(cd.w)}, Tn), DF2{f2(cd.x), f2(cd.y)});
                const DF2 Z = df2_add(df2_mul(be, gm1), df2_mul(DF2{f2(hh.z), f2(hh.w)}, W));
                W = df2_add(W, df2_mul(df2_mul(kap, DF2{f2(hh.x), f2(hh.y)}), cur));
                gm1 = cur;
                cur = df2_add(df2_mul(al, cur), Z);
                put(l + 1, cur);
            }
        } else {
            // full-range p_x: G_l(+-u_x)
            const float2 ux = in(0);
            const DF2 u = {make_float2(ux.x, -ux.x), make_float2(ux.y, -ux.y)}, Tm1 = df2_dup(in(4));
            DF2 gm1 = {f2(1.0f), f2(0.0f)}, cur = u;
            put(0, gm1);
            if (Nx >= 1) put(1, cur);
#pragma unroll 1
            for (int l = 1; l < Nx; ++l) {
                const DF2 nxt = df2_add(df2_mul(u, cur), df2_mul(df2_mul(DF2{f2((float)l), f2(0.0f)}, Tm1), gm1));
                gm1 = cur;
                cur = nxt;
                put(l + 1, cur);
            }
        }
    } else if (active && slot == (NB < 32 ? 32 / NB : 1)) {     // in another warp than slot 0
        // G_l(u_y) with G_l(u_z); an order past an axis's last is a zero
        const float2 ua = in(1), ub = in(2);
        float* fy = reinterpret_cast<float*>(Gy);
        float* fz = reinterpret_cast<float*>(Gz);
        const int ly = g.Qy ? 2 * nt.my : 0, lz = g.Qz ? 2 * nt.mz : 0;
        auto put = [&](int l, const DF2& v) {
            const int at = 4 * (l >> 1) * NB + (l & 1);
            if (l < ly) { fy[at] = l <= Ny ? v.h.x : 0.0f; fy[at + 2 * NB] = l <= Ny ? v.l.x : 0.0f; }
            if (l < lz) { fz[at] = l <= Nz ? v.h.y : 0.0f; fz[at + 2 * NB] = l <= Nz ? v.l.y : 0.0f; }
        };
        const DF2 u = {make_float2(ua.x, ub.x), make_float2(ua.y, ub.y)}, Tm1 = df2_dup(in(4));
        DF2 gm1 = {f2(1.0f), f2(0.0f)}, cur = u;
        put(0, gm1);
        put(1, cur);
#pragma unroll 1
        for (int l = 1; l + 1 < max(ly, lz); ++l) {
            const DF2 nxt = df2_add(df2_mul(u, cur), df2_mul(df2_mul(DF2{f2((float)l), f2(0.0f)}, Tm1), gm1));
            gm1 = cur;
            cur = nxt;
            put(l + 1, cur);
        }
    }
    __syncthreads();
    // 2. dot products: items of two rows of p_x, then of p_y, then of p_z
    const int ix = Qx >> 1, iy = g.Qy ? (VY + 2) >> 2 : 1, iz = g.Qz ? (VZ + 2) >> 2 : 1;
    const DF2 n = df2_dup(in(7));
    float* line = sLine + k * node_line_stride(g.ncp);
#pragma unroll 1
    for (int it = slot; it < ix + iy + iz; it += SLOTS) {
        const bool x = it < ix, z = it >= ix + iy;
        float* o = line + (x ? 0 : QX2 + (z ? VY : 0));
        if (!x && (z ? !g.Qz : !g.Qy)) {                 // an absent axis: 1
            o[0] = active ? 1.0f : 0.0f;
            continue;
        }
        // rows j and j + 1 of p_x, or of the positive half of p_y or p_z
        const int j = 2 * (x ? it : it - ix - (z ? iy : 0)), half = x ? Qx : (z ? VZ : VY) >> 1;
        const int m = x ? Nx + 1 : (z ? nt.mz : nt.my);
        const float4* P = tab + (x ? it * m : nt.nx + (z ? nt.ny : 0) + j * m);
        float2 a = f2(0.0f), b = f2(0.0f);               // the values of +-p, rows j and j + 1
        if (active) {
            DF2 r0, r1;
            dot2_rows<NB>(x, P, !x && j + 1 < half ? P + m : P, x ? Gx : (z ? Gz : Gy), m, r0, r1);
            if (x) {
                r0 = df2_mul(r0, n);
                r1 = df2_mul(r1, n);
            } else {
                // lanes (even, odd) to the rows of z and -z: sum and difference
                r0 = df2_add(DF2{f2(r0.h.x), f2(r0.l.x)}, DF2{make_float2(r0.h.y, -r0.h.y), make_float2(r0.l.y, -r0.l.y)});
                r1 = df2_add(DF2{f2(r1.h.x), f2(r1.l.x)}, DF2{make_float2(r1.h.y, -r1.h.y), make_float2(r1.l.y, -r1.l.y)});
            }
            a = __fadd2_rn(r0.h, r0.l);
            b = __fadd2_rn(r1.h, r1.l);
        }
        const int p0 = x ? j : half + j, m0 = x ? Qx + j : half - 1 - j, dm = x ? 1 : -1;
        o[p0] = a.x;
        o[m0] = a.y;
        if (j + 1 < half) {
            o[p0 + 1] = b.x;
            o[m0 + dm] = b.y;
        }
    }
}

}  // namespace hlb
