// Node pass of an RK-3 stage (sm_103a): the quadrature sums of every node
// (Eq. "eq:fmoms"), then n, u, T, 1/tau and the per-node equilibrium factor
// line coef[node] = { n g_x (2Qx), g_y (Qy), g_z (Qz), 1/tau } (Eqs.
// "eq:hh_gk", "eq:H_gk", App. A; half-range recurrence in the orthonormal
// basis, full-range Hermite recurrence).
#include <cuda_runtime.h>

#include <cstdint>

#include "hlb_coef.cuh"
#include "hlb_device.cuh"
#include "hlb_internal.h"
#include "hlb_wall.cuh"

namespace hlb {
namespace {

// ---------------------------------------------------------------------------
// node kernels of the FP32 groups that node_df_kernel does not take (orders
// above 15, rows that are not 8, 16 or 32 values, 2D groups of at most 256
// nodes, large groups of few velocities (node_fused_pays))
// ---------------------------------------------------------------------------
// Per-node equilibrium factors, in two passes with no block-wide barrier:
//   sums_kernel   streams the stage input once (one warp per node) and writes
//                 the five quadrature sums n, j_x, j_y, j_z, E per node;
//   coef_kernel   one warp per 32 nodes, one lane per node: n, u, T, then the
//                 coefficient recurrences of all four roles, then the factor
//                 line (dot products shared across the warp).
// FP64 runs at 1/64 of FP32 here and a warp instruction costs the same
// whatever its mask, so every FP64 instruction runs on full warps; FP32
// groups with Nx <= 15 run the recurrences and dot products in double-float
// (FP64 only for erf, exp, sqrt, once per node).
__global__ void __launch_bounds__(256) sums_kernel(const GroupDev g, const float* __restrict__ fs, float* __restrict__ sums) {
    extern __shared__ __align__(16) double ssm[];
    const int QX2 = g.QX2, VY = g.VY, VZ = g.VZ, V = g.V;
    const int tid = threadIdx.x, bs = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31, nw = bs >> 5;
    float4* sM = reinterpret_cast<float4*>(ssm);         // [V]: p_x, p_y, p_z, |p|^2
    float4* sYZ = sM + V;                                // [VY * VZ]: p_y, p_z, p_y^2 + p_z^2
    const float* px = static_cast<const float*>(g.p);
    const float* py = px + QX2;
    const float* pz = py + VY;
    for (int v = tid; v < V; v += bs) {
        const int ix = v % QX2, jy = (v / QX2) % VY, kz = v / (QX2 * VY);
        const float a = px[ix], b = py[jy], c = pz[kz];
        float4 m4;
        m4.x = a; m4.y = b; m4.z = c; m4.w = a * a + b * b + c * c;
        sM[v] = m4;
    }
    for (int bq = tid; bq < VY * VZ; bq += bs) {
        const float b = py[bq % VY], c = pz[bq / VY];
        float4 y4;
        y4.x = b; y4.y = c; y4.z = b * b + c * c; y4.w = 0.0f;
        sYZ[bq] = y4;
    }
    __syncthreads();
    // 4-vector loads with eight lanes per node, four nodes per warp: they need
    // 4 | 2Qx and 2Qx | 32 (2Qx a power of two up to 32), so that the four
    // velocities of a load share (jy, kz) and a lane's p_x never change.  The
    // compensated tree then has three levels, and each shuffle serves four
    // nodes.  Other sets: one warp per node, a table of all velocities.
    const bool vec4 = (QX2 & 3) == 0 && (QX2 & (QX2 - 1)) == 0 && QX2 <= 32 && V >= 32;
    auto store = [&](int node, float a0, float a1, float a2, float a3, float a4, float c0, float c1, float c2, float c3, float c4) {
        float* o = sums + (size_t)node * kSumStride;
        o[0] = a0; o[1] = a1; o[2] = a2; o[3] = a3; o[4] = a4;
        o[8] = c0; o[9] = c1; o[10] = c2; o[11] = c3; o[12] = c4;
    };
    if (vec4) {
        const int sl = lane & 7;
        const int x0 = (4 * sl) % QX2;
        const int lg = __ffs(QX2) - 1;                   // 2Qx = 2^lg
        const float pxa = sM[x0].x, pxb = sM[x0 + 1].x, pxc = sM[x0 + 2].x, pxd = sM[x0 + 3].x;
        for (int nb = (blockIdx.x * nw + warp) * 4; nb < g.nnodes; nb += gridDim.x * nw * 4) {
            const int node = nb + (lane >> 3);
            // compensated per-lane sums (FP32 states)
            float a0 = 0, a1 = 0, a2 = 0, a3 = 0, a4 = 0, c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0;
            if (node < g.nnodes) {
                const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
                const InstDev& I = g.inst[ii];
                const float4* f4 = reinterpret_cast<const float4*>(fs + (size_t)I.f_off + (size_t)(node - I.node_off) * V);
#pragma unroll 4
                for (int q = sl; q < (V >> 2); q += 8) {
                    const float4 x = f4[q];
                    const float4 yz = sYZ[(q << 2) >> lg];
                    const float sq = (x.x + x.y) + (x.z + x.w);
                    csum_add(a0, c0, sq);
                    csum_add(a1, c1, pxa * x.x + pxb * x.y + pxc * x.z + pxd * x.w);
                    csum_add(a2, c2, yz.x * sq);
                    csum_add(a3, c3, yz.y * sq);
                    csum_add(a4, c4, pxa * pxa * x.x + pxb * pxb * x.y + pxc * pxc * x.z + pxd * pxd * x.w + yz.z * sq);
                }
            }
            // compensated tree over the eight lanes of each node
            auto tree8 = [](float& sa, float& ca) {
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    const float s2 = __shfl_xor_sync(0xffffffffu, sa, o), c2 = __shfl_xor_sync(0xffffffffu, ca, o);
                    csum_add(sa, ca, s2);
                    ca += c2;
                }
            };
            tree8(a0, c0); tree8(a1, c1); tree8(a2, c2); tree8(a3, c3); tree8(a4, c4);
            if (sl == 0 && node < g.nnodes) store(node, a0, a1, a2, a3, a4, c0, c1, c2, c3, c4);
        }
        return;
    }
    for (int node = blockIdx.x * nw + warp; node < g.nnodes; node += gridDim.x * nw) {
        const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
        const InstDev& I = g.inst[ii];
        const float* f = fs + (size_t)I.f_off + (size_t)(node - I.node_off) * V;
        // compensated per-lane sums (FP32 states), compensated warp tree
        float a0 = 0, a1 = 0, a2 = 0, a3 = 0, a4 = 0, c0 = 0, c1 = 0, c2 = 0, c3 = 0, c4 = 0;
        for (int v = lane; v < V; v += 32) {
            const float val = f[v];
            const float4 mw = sM[v];
            csum_add(a0, c0, val);
            csum_add(a1, c1, mw.x * val);
            csum_add(a2, c2, mw.y * val);
            csum_add(a3, c3, mw.z * val);
            csum_add(a4, c4, mw.w * val);
        }
        csum_warp(a0, c0); csum_warp(a1, c1); csum_warp(a2, c2); csum_warp(a3, c3); csum_warp(a4, c4);
        if (lane == 0) store(node, a0, a1, a2, a3, a4, c0, c1, c2, c3, c4);
    }
}

__global__ void __launch_bounds__(32) coef_kernel(const GroupDev g, const float* __restrict__ sums) {
    extern __shared__ __align__(16) double csm[];
    const int Nx = g.Nx, Ny = g.Ny, Nz = g.Nz;
    const int nrec = 5 * Nx + 1;
    const int nT = g.Qx * (Nx + 1) + g.VY * (Ny + 1) + g.VZ * (Nz + 1);
    const int ncoef = 2 * (Nx + 1) + (Ny + 1) + (Nz + 1);
    const int QX2 = g.QX2, VY = g.VY, VZ = g.VZ;
    const int tid = threadIdx.x, bs = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31, nw = bs >> 5;
    const bool df = g.use_df != 0;
    double* sRec = csm;
    double* sT = sRec + nrec;
    double* sW = sT + nT;                                // per warp: [32][ncoef] coefficients + [32] state
    const int per_warp = 32 * ncoef + 32 * 2 + 32 * (int)(sizeof(NodeDF) / 8);
    double* sG = sW + warp * per_warp;
    double* sNT = sG + 32 * ncoef;                       // [32][2]: n, 1/tau
    NodeDF* sIn = reinterpret_cast<NodeDF*>(sNT + 64);   // [32]
    float2* sRecF = reinterpret_cast<float2*>(sRec);
    float2* sTF = reinterpret_cast<float2*>(sT);
    float2* sGF = reinterpret_cast<float2*>(sG);
    if (df) {
        for (int i = tid; i < nrec; i += bs) sRecF[i] = g.recf[i];
        for (int i = tid; i < nT; i += bs) sTF[i] = g.Tf[i];
    } else {
        for (int i = tid; i < nrec; i += bs) sRec[i] = g.rec[i];
        for (int i = tid; i < nT; i += bs) sT[i] = g.Td[i];
    }
    __syncthreads();
    const double* sTx = sT;
    const double* sTy = sTx + g.Qx * (Nx + 1);
    const double* sTz = sTy + VY * (Ny + 1);
    const float2* sTxF = sTF;
    const float2* sTyF = sTxF + g.Qx * (Nx + 1);
    const float2* sTzF = sTyF + VY * (Ny + 1);
    float* coef = static_cast<float*>(g.coef);
    const int nf = QX2 + VY + VZ;
    const int nbatches = (g.nnodes + 31) / 32;
    for (int bt = blockIdx.x * nw + warp; bt < nbatches; bt += gridDim.x * nw) {
        const int base = bt * 32;
        const int nb = min(32, g.nnodes - base);
        // 1. lane = node: n, u, T, 1/tau; the recurrences' FP64 inputs
        bool active = false;
        if (lane < nb) {
            const int node = base + lane;
            const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
            const double inv_Kn = g.inst[ii].inv_Kn;
            const float* sm = sums + (size_t)node * kSumStride;
            active = inv_Kn != 0.0;
            // n, u, T in FP64 from the compensated sums (one division)
            const double n = (double)sm[0] + (double)sm[8], in = 1.0 / n;
            const double ux = ((double)sm[1] + (double)sm[9]) * in, uy = ((double)sm[2] + (double)sm[10]) * in,
                         uz = ((double)sm[3] + (double)sm[11]) * in;
            const double T = ((double)sm[4] + (double)sm[12] - n * (ux * ux + uy * uy + uz * uz)) * in *
                             (g.D == 3 ? 1.0 / 3.0 : (g.D == 2 ? 0.5 : 1.0));
            sNT[2 * lane] = n;
            sNT[2 * lane + 1] = n * inv_Kn;
            if (active) {
                if (df) {
                    node_inputs_df(n, ux, uy, uz, T, Nx, sIn[lane]);
                    for (int role = 0; role < 4; ++role)
                        node_coefficients_df(g, role, sIn[lane], sRecF, sGF + lane * ncoef);
                } else {
                    for (int role = 0; role < 4; ++role) {
                        node_coefficients(g, role, ux, uy, uz, T, sRec, sG + lane * ncoef);
                    }
                }
            }
        }
        __syncwarp();
        // 2. factor lines: lanes over (node, output), one loop per output kind
        //    so that the lanes of a warp follow the same path
        for (int t = lane; t < nb * QX2; t += 32) {          // n g_x
            const int k = t / QX2, o = t - k * QX2;
            float* line = coef + (size_t)(base + k) * g.ncp;
            if (sNT[2 * k + 1] == 0.0) { line[o] = 0.0f; continue; }
            const int kk = o % g.Qx, sg = o / g.Qx;
            if (df) {
                const float2* Gs = sGF + k * ncoef + sg * (Nx + 1);
                const float2* Tr = sTxF + kk * (Nx + 1);
                float2 acc = df_mul(Tr[0], Gs[0]);
                for (int l = 1; l <= Nx; ++l) acc = df_add(acc, df_mul(Tr[l], Gs[l]));
                acc = df_mul(acc, sIn[k].n);
                line[o] = acc.x + acc.y;
            } else {
                const double* Gs = sG + k * ncoef + sg * (Nx + 1);
                const double* Tr = sTx + kk * (Nx + 1);
                double acc = 0.0;
                for (int l = 0; l <= Nx; ++l) acc += Tr[l] * Gs[l];
                line[o] = (float)(acc * sNT[2 * k]);
            }
        }
        for (int t = lane; t < nb * VY; t += 32) {           // g_y
            const int k = t / VY, j = t - k * VY;
            float* line = coef + (size_t)(base + k) * g.ncp + QX2;
            if (sNT[2 * k + 1] == 0.0) { line[j] = 0.0f; continue; }
            if (!g.Qy) { line[j] = 1.0f; continue; }
            if (df) {
                const float2* Gy = sGF + k * ncoef + 2 * (Nx + 1);
                const float2* Tr = sTyF + j * (Ny + 1);
                float2 acc = df_mul(Tr[0], Gy[0]);
                for (int l = 1; l <= Ny; ++l) acc = df_add(acc, df_mul(Tr[l], Gy[l]));
                line[j] = acc.x + acc.y;
            } else {
                const double* Gy = sG + k * ncoef + 2 * (Nx + 1);
                const double* Tr = sTy + j * (Ny + 1);
                double acc = 0.0;
                for (int l = 0; l <= Ny; ++l) acc += Tr[l] * Gy[l];
                line[j] = (float)acc;
            }
        }
        for (int t = lane; t < nb * VZ; t += 32) {           // g_z
            const int k = t / VZ, j = t - k * VZ;
            float* line = coef + (size_t)(base + k) * g.ncp + QX2 + VY;
            if (sNT[2 * k + 1] == 0.0) { line[j] = 0.0f; continue; }
            if (!g.Qz) { line[j] = 1.0f; continue; }
            if (df) {
                const float2* Gz = sGF + k * ncoef + 2 * (Nx + 1) + (Ny + 1);
                const float2* Tr = sTzF + j * (Nz + 1);
                float2 acc = df_mul(Tr[0], Gz[0]);
                for (int l = 1; l <= Nz; ++l) acc = df_add(acc, df_mul(Tr[l], Gz[l]));
                line[j] = acc.x + acc.y;
            } else {
                const double* Gz = sG + k * ncoef + 2 * (Nx + 1) + (Ny + 1);
                const double* Tr = sTz + j * (Nz + 1);
                double acc = 0.0;
                for (int l = 0; l <= Nz; ++l) acc += Tr[l] * Gz[l];
                line[j] = (float)acc;
            }
        }
        if (lane < nb) coef[(size_t)(base + lane) * g.ncp + nf] = (float)sNT[2 * lane + 1];   // 1/tau
        if (g.has_field && lane < nb) {              // a = a_uniform + a_field(node)
            const int node = base + lane;
            const InstDev& I = g.inst[g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0];
            float* fl = coef + (size_t)node * g.ncp + g.field_off;
            fl[0] = (float)(I.ax + g.afield[3 * (size_t)node]);
            fl[1] = (float)(I.ay + g.afield[3 * (size_t)node + 1]);
            fl[2] = (float)(I.az + g.afield[3 * (size_t)node + 2]);
        }
        __syncwarp();
    }
}

template <int NM>
__global__ void __launch_bounds__(128) coef_df_kernel(const GroupDev g, const float* __restrict__ sums) {
    extern __shared__ __align__(16) float2 cdf[];
    const int Nx = g.Nx, Ny = g.Ny, Nz = g.Nz, Qx = g.Qx, QX2 = g.QX2, VY = g.VY, VZ = g.VZ, ncp = g.ncp;
    const int nrec = 5 * Nx + 1;
    // the tables T_x (Qx rows), T_y (VY rows), T_z (VZ rows) of Nx+1, Ny+1,
    // Nz+1 double-float entries, re-laid as row pairs (dot2_pair); an odd last
    // row is paired with zeros
    const int px = (Qx + 1) >> 1, py = (VY + 1) >> 1, pz = (VZ + 1) >> 1;
    const int nP = px * (Nx + 1) + py * (Ny + 1) + pz * (Nz + 1);
    float4* sP = reinterpret_cast<float4*>(cdf);
    float2* sRec = reinterpret_cast<float2*>(sP + nP);
    float* sLine = reinterpret_cast<float*>(sP + nP + ((nrec + 1) >> 1)) + (threadIdx.x >> 5) * 32 * ncp;   // [32][ncp] per warp
    for (int i = threadIdx.x; i < nrec; i += blockDim.x) sRec[i] = g.recf[i];
    {
        const float2* Tx = g.Tf;
        const float2* Ty = Tx + Qx * (Nx + 1);
        const float2* Tz = Ty + VY * (Ny + 1);
        auto pairs = [&](float4* dst, const float2* T, int rows, int n1) {
            const int np = (rows + 1) >> 1;
            for (int i = threadIdx.x; i < np * n1; i += blockDim.x) {
                const int k = 2 * (i / n1), l = i % n1;
                const float2 a = T[k * n1 + l];
                const float2 b = k + 1 < rows ? T[(k + 1) * n1 + l] : make_float2(0.0f, 0.0f);
                dst[i] = make_float4(a.x, b.x, a.y, b.y);
            }
        };
        pairs(sP, Tx, Qx, Nx + 1);
        pairs(sP + px * (Nx + 1), Ty, VY, Ny + 1);
        pairs(sP + px * (Nx + 1) + py * (Ny + 1), Tz, VZ, Nz + 1);
    }
    __syncthreads();
    const float4* sPx = sP;
    const float4* sPy = sPx + px * (Nx + 1);
    const float4* sPz = sPy + py * (Ny + 1);
    const int lane = threadIdx.x & 31;
    const int base = blockIdx.x * blockDim.x + (threadIdx.x & ~31);
    const int node = base + lane;
    float* line = sLine + lane * ncp;
    if (node < g.nnodes) {
        const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
        const double inv_Kn = g.inst[ii].inv_Kn;
        const float* sm = sums + (size_t)node * kSumStride;
        bool done = false;
        if constexpr (NM <= 12) {
            if (Nx <= HLB_DF_SPECIAL_MAX_N) {
                // n, u, T and the recurrences' start in double-float (no FP64
                // pipe work but for 1/tau and the rare |z| > 2.5)
                NodeDF nin;
                const double n = node_inputs_from_sums_df<true>(sm, g.D, nin);
                factor_line_df_in<NM>(g, nin, n * inv_Kn, sPx, sPy, sPz, sRec, line);
                done = true;
            }
        }
        if (!done) {
            // n, u, T in FP64 from the compensated sums (one division)
            const double n = (double)sm[0] + (double)sm[8], in = 1.0 / n;
            const double ux = ((double)sm[1] + (double)sm[9]) * in, uy = ((double)sm[2] + (double)sm[10]) * in,
                         uz = ((double)sm[3] + (double)sm[11]) * in;
            const double T = ((double)sm[4] + (double)sm[12] - n * (ux * ux + uy * uy + uz * uz)) * in *
                             (g.D == 3 ? 1.0 / 3.0 : (g.D == 2 ? 0.5 : 1.0));
            factor_line_df<NM>(g, n, ux, uy, uz, T, (double)n * inv_Kn, sPx, sPy, sPz, sRec, line);
        }
        if (g.has_field) {                           // a = a_uniform + a_field(node)
            const InstDev& I = g.inst[ii];
            line[g.field_off] = (float)(I.ax + g.afield[3 * (size_t)node]);
            line[g.field_off + 1] = (float)(I.ay + g.afield[3 * (size_t)node + 1]);
            line[g.field_off + 2] = (float)(I.az + g.afield[3 * (size_t)node + 2]);
        }
    }
    __syncwarp();
    // the warp's lines are contiguous in the factor-line buffer
    const int nb = min(32, g.nnodes - base);
    if (nb > 0) {
        float4* dst = reinterpret_cast<float4*>(static_cast<float*>(g.coef) + (size_t)base * ncp);
        const float4* src = reinterpret_cast<const float4*>(sLine);
        for (int i = lane; i < nb * ncp / 4; i += 32) dst[i] = src[i];
    }
}


// ---------------------------------------------------------------------------
// The node pass of FP32 groups in one launch: the first g.nrows g.wchunks CTAs
// form the walls' emitted densities, every other CTA the moment sums and the
// factor lines of NB nodes (32, or 8 in small groups; node_nb).  The sums stream the state (HBM-bound), the
// lines are double-float arithmetic (issue- and latency-bound) and the walls a
// few CTAs: in one launch they share the SMs instead of running in a row, and a
// line's work is spread over the CTA (node_lines).  Per stage, against the three
// kernels: 1024 x 512 nodes of 1024 velocities 0.426 against 0.495 ms (reading
// the state alone takes 0.317), the 256^2 box of order 15 0.070 against 0.111,
// 317 x 203 nodes of order 7 0.026 against 0.043 (GB300).  32 nodes and 128
// threads at 8 CTAs per SM (7 for order 15): 10 per SM spill (0.094 for the
// box), and a resident grid that loops over the batches runs its CTAs in step,
// all streaming or all computing (0.93 ms for the large channel).
// ---------------------------------------------------------------------------
constexpr int kNodeT = 128;

struct NodeSmem {                        // byte offsets
    size_t tab, yz, rec, in, G, line, bytes;
};
template <int NB>
__host__ __device__ inline NodeSmem node_smem(const GroupDev& g) {
    const NodeTables nt(g);
    NodeSmem L;
    L.tab = 0;
    L.yz = L.tab + nt.table_bytes();
    L.rec = L.yz + (size_t)g.VY * g.VZ * 16;
    L.in = L.rec + node_rec_bytes(g.Nx);
    L.G = L.in + (size_t)NB * kNodeFields * 8;
    L.line = L.G + nt.coef_bytes<NB>(g);            // the moment sums, then the lines
    const size_t lines = (size_t)NB * node_line_stride(g.ncp) * 4, sums = (size_t)NB * kSumStride * 4;
    L.bytes = L.line + (lines > sums ? lines : sums);
    return L;
}

// The compensated moment sums of nb nodes into sum[node][kSumStride], LPN lanes
// per node (rows of 4 LPN values); z: a p_z axis.  A lane adds (n, j_x), (j_y, E)
// and j_z, two sums per packed compensated addition.
template <int LPN>
__device__ __forceinline__ void node_sums(const float* fs, const float* __restrict__ P,
                                          const float4* sYZ, const long long* sOff, float* sum, int nb, int rows, int V,
                                          bool z) {
    const int lane = threadIdx.x & 31, sl = lane % LPN;
    const float4 p = reinterpret_cast<const float4*>(P)[sl];
    const float2 pa = make_float2(p.x, p.y), pb = make_float2(p.z, p.w);
    const float2 qa = __fmul2_rn(pa, pa), qb = __fmul2_rn(pb, pb);
    // every lane of a warp takes part in the shuffles, nodes or not
    for (int k = threadIdx.x / LPN; (k & ~(32 / LPN - 1)) < nb; k += kNodeT / LPN) {
        float2 a01 = f2(0.0f), c01 = f2(0.0f), a24 = f2(0.0f), c24 = f2(0.0f);
        float a3 = 0.0f, c3 = 0.0f;
        if (k < nb) {
            const float4* f4 = reinterpret_cast<const float4*>(fs + sOff[k]) + sl;
            auto add = [&](const float4 x, const float4 yz) {
                const float2 xa = make_float2(x.x, x.y), xb = make_float2(x.z, x.w);
                const float2 s2 = __fadd2_rn(xa, xb);
                const float2 j2 = __ffma2_rn(pb, xb, __fmul2_rn(pa, xa)), e2 = __ffma2_rn(qb, xb, __fmul2_rn(qa, xa));
                const float sq = s2.x + s2.y;
                csum_add2(a01, c01, make_float2(sq, j2.x + j2.y));
                csum_add2(a24, c24, make_float2(yz.x * sq, fmaf(yz.z, sq, e2.x + e2.y)));
                if (z) csum_add(a3, c3, yz.y * sq);
            };
#pragma unroll 4
            for (int r = 0; r < rows; ++r) add(__ldcs(f4 + r * LPN), sYZ[r]);
        }
#pragma unroll
        for (int o = LPN / 2; o > 0; o >>= 1) {          // compensated tree over the lanes of a node
            auto up2 = [&](float2& s, float2& c) {
                const float2 s2 = make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o));
                const float2 c2 = make_float2(__shfl_xor_sync(0xffffffffu, c.x, o), __shfl_xor_sync(0xffffffffu, c.y, o));
                csum_add2(s, c, s2);
                c = __fadd2_rn(c, c2);
            };
            up2(a01, c01);
            up2(a24, c24);
            if (z) {
                const float s2 = __shfl_xor_sync(0xffffffffu, a3, o), c2 = __shfl_xor_sync(0xffffffffu, c3, o);
                csum_add(a3, c3, s2);
                c3 += c2;
            }
        }
        if (sl == 0 && k < nb) {
            float* o = sum + k * kSumStride;
            o[0] = a01.x; o[1] = a01.y; o[2] = a24.x; o[3] = a3; o[4] = a24.y;
            o[8] = c01.x; o[9] = c01.y; o[10] = c24.x; o[11] = c3; o[12] = c24.y;
        }
    }
}

template <int ADV, int LOWN, int NB>
__global__ void __launch_bounds__(kNodeT, LOWN ? 8 : 7) node_df_kernel(const GroupDev g, const float* fs) {
    extern __shared__ __align__(16) unsigned char nsm[];
    const int nwall = g.nrows * g.wchunks;
    if ((int)blockIdx.x < nwall) {
        pdl_wait();
        pdl_trigger();
        wall_block<float, ADV>(g, fs, blockIdx.x, reinterpret_cast<double*>(nsm));
        return;
    }
    const NodeSmem L = node_smem<NB>(g);
    float4* tab = reinterpret_cast<float4*>(nsm + L.tab);
    float4* sYZ = reinterpret_cast<float4*>(nsm + L.yz);
    float4* rec = reinterpret_cast<float4*>(nsm + L.rec);
    float2* sIn = reinterpret_cast<float2*>(nsm + L.in);
    float2* sG = reinterpret_cast<float2*>(nsm + L.G);
    float* sLine = reinterpret_cast<float*>(nsm + L.line);
    float* sSum = sLine;
    const int QX2 = g.QX2, VY = g.VY, VZ = g.VZ, V = g.V;
    const int tid = threadIdx.x;
    const NodeTables nt(g);
    const float* P = static_cast<const float*>(g.p);
    for (int b = tid; b < VY * VZ; b += kNodeT) {          // momenta of the (jy, kz) pairs
        const float y = P[QX2 + b % VY], z = P[QX2 + VY + b / VY];
        sYZ[b] = make_float4(y, z, y * y + z * z, 0.0f);
    }
    node_load_rec(g, rec, tid, kNodeT);
    node_load_tables(g, nt, tab, tid, kNodeT);
    const int base = ((int)blockIdx.x - nwall) * NB;
    const int nb = min(NB, g.nnodes - base);
    __shared__ long long sOff[NB];      // each node's values in the state
    int ii = 0;
    if (tid < nb) {
        ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, base + tid) : 0;
        sOff[tid] = g.inst[ii].f_off + (long long)(base + tid - g.inst[ii].node_off) * V;
    }
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    // 1. moment sums: 2Qx / 4 lanes per node, so that a lane's p_x never change
    // and step r of its loop is the row r of (jy, kz)
    if (QX2 == 32) node_sums<8>(fs, P, sYZ, sOff, sSum, nb, VY * VZ, V, VZ > 1);
    else if (QX2 == 16) node_sums<4>(fs, P, sYZ, sOff, sSum, nb, VY * VZ, V, VZ > 1);
    else node_sums<2>(fs, P, sYZ, sOff, sSum, nb, VY * VZ, V, VZ > 1);
    __syncthreads();
    // 2. n, u, T, 1/tau and what starts the recurrences, one thread per node
    if (tid < NB) {
        NodeDF in;
        double itau = 0.0;
        if (tid < nb) {
            const double inv_Kn = g.inst[ii].inv_Kn;
            const float* sm = sSum + tid * kSumStride;
            itau = node_inputs_from_sums_df<LOWN != 0>(sm, g.D, in) * inv_Kn;
        }
        const float2 v[kNodeFields] = {in.ux, in.uy, in.uz, in.T, in.Tm1, in.erf_z, in.g0, in.n, make_float2((float)itau, 0.0f)};
#pragma unroll
        for (int f = 0; f < kNodeFields; ++f) sIn[f * NB + tid] = v[f];
    }
    __syncthreads();
    node_lines<NB, kNodeT>(g, nt, sIn, sG, sLine, tab, rec);
    if (tid < nb) {                                      // the lines' tails: 1/tau, the field's accelerations
        float* line = sLine + tid * node_line_stride(g.ncp);
        const int t0 = QX2 + VY + VZ;
        line[t0] = sIn[8 * NB + tid].x;
        for (int o = t0 + 1; o < g.ncp; ++o) line[o] = 0.0f;
        if (g.has_field) {                           // a = a_uniform + a_field(node)
            const InstDev& I = g.inst[ii];
            const double* af = g.afield + 3 * (size_t)(base + tid);
            line[g.field_off] = (float)(I.ax + af[0]);
            line[g.field_off + 1] = (float)(I.ay + af[1]);
            line[g.field_off + 2] = (float)(I.az + af[2]);
        }
    }
    __syncthreads();
    // 3. the lines are contiguous in the factor-line buffer
    const int w4 = g.ncp / 4, s4 = node_line_stride(g.ncp) / 4;
    float4* dst = reinterpret_cast<float4*>(static_cast<float*>(g.coef) + (size_t)base * g.ncp);
    const float4* src = reinterpret_cast<const float4*>(sLine);
    for (int i = tid; i < nb * w4; i += kNodeT) {
        const int k = i / w4;
        dst[i] = src[k * s4 + (i - k * w4)];
    }
}

// ---------------------------------------------------------------------------
// The node pass of FP64 groups in one launch: the first g.nrows g.wchunks CTAs
// form the walls' emitted densities, every other CTA the moments and factor
// lines of NB nodes.  FP64 instructions run at 1/64 of FP32, per warp whatever its
// mask, and in long dependent chains (erf, exp, divisions, recurrences), so a
// small group waits on one thread's chain and a large one on the pipe: the
// roles of the recurrences run in different threads (p_x in warp 0, p_y and
// p_z in warp 1), the dot products over the whole CTA; one node per CTA where
// that leaves at most two CTAs per SM, sixteen, whose recurrences and short rows
// fill the lanes of a warp, in groups of more than 16 nodes per SM, eight
// between and in the order-200 sets, whose long rows want the lanes.  Per
// stage (GB300): 5795 nodes of 128 velocities 30 us; 72 nodes of 400 velocities,
// order 20, 14.7 us with one node per CTA, 47 with eight; the 64 nodes of the
// FP64 channel (moments, lines and walls in three kernels before) take 9 of the
// 17 us that a stage is now.  Sixteen against eight: 100000 nodes of 32 velocities
// 158 / 277 us, of 128 259 / 371, 5000 of 32 19 / 24; 1200 of 128 18.5 / 16.7; 2400 of
// order 200 463 / 423 (with the quadrature).
// ---------------------------------------------------------------------------
constexpr int kNode64T = 128;

__host__ __device__ inline size_t node64_smem(const GroupDev& g, int NB) {
    const int ncoef = 2 * (g.Nx + 1) + (g.Ny + 1) + (g.Nz + 1);
    return sizeof(double) * ((size_t)NB * (6 + ncoef) + 5 * g.Nx + 1 + 3 * g.VY * g.VZ + 20);
}

// The half-range coefficients of node_coefficients (role r = 0, 1) with exp and
// erf by their Taylor polynomials where the flow is slow enough.
__device__ __forceinline__ void half_range_coefficients(const GroupDev& g, int r, double ux, double T, const double* rec,
                                                        double* G) {
    const int Nx = g.Nx;
    double irt;
    if (T > 1e-30 && T < 1e30) {
        irt = (double)rsqrtf((float)T);                          // one third-order Householder step
        const double e = fma(-T * irt, irt, 1.0);
        irt = fma(irt * e, fma(0.375, e, 0.5), irt);
    } else {
        irt = 1.0 / sqrt(T);
    }
    const double z = ux * irt * 0.70710678118654752440;
    double E, F;
    if (fabs(z) <= 0.7) {
        exp_erf_small(-z * z, E, F);
        F *= z * 1.1283791670955125739;                          // 2 / sqrt(pi)
    } else {
        E = exp(-z * z);
        F = erf(z);
    }
    const double us = r ? -ux : ux, g0 = E * (irt * (1.0 / kSqrt2Pi));
    const double* rb = rec + Nx;
    const double* rc = rec + 2 * Nx;
    const double* h0 = rec + 3 * Nx;
    const double* d = rec + 4 * Nx + 1;
    G[0] = h0[0] * (0.5 + (r ? -0.5 : 0.5) * F);
    double S = 0.0, gm1 = 0.0;
    for (int l = 0; l < Nx; ++l) {
        const double ig = (l ? gm1 * d[l - 1] : 0.0) - g.om0 * h0[l] * S;
        const double pg = us * G[l] + T * (g0 * h0[l] + ig);
        G[l + 1] = rec[l] * pg + rb[l] * G[l] + rc[l] * gm1;
        S += h0[l] * G[l];
        gm1 = G[l];
    }
}

template <int ADV, int NB>
__global__ void __launch_bounds__(kNode64T) node_f64_kernel(const GroupDev g, const double* fs) {
    extern __shared__ __align__(16) double dsm[];
    constexpr int LPN = kNode64T / NB;                        // lanes per node
    const int nwall = g.nrows * g.wchunks;
    if ((int)blockIdx.x < nwall) {
        pdl_wait();
        pdl_trigger();
        wall_block<double, ADV>(g, fs, blockIdx.x, dsm);
        return;
    }
    const int Nx = g.Nx, Ny = g.Ny, Nz = g.Nz, Qx = g.Qx, QX2 = g.QX2, VY = g.VY, VZ = g.VZ, rows = VY * VZ;
    const int ncoef = 2 * (Nx + 1) + (Ny + 1) + (Nz + 1), nf = QX2 + VY + VZ;
    double* sM = dsm;                        // [NB][6]: n, u_x, u_y, u_z, T, 1/tau
    double* sG = sM + 6 * NB;                // [NB][ncoef]
    double* sRec = sG + NB * ncoef;
    double* sRow = sRec + 5 * Nx + 1;        // [rows][3]: p_y, p_z, p_y^2 + p_z^2
    double* sPart = sRow + 3 * rows;         // [4][5]: partial moments of the warps (NB = 1)
    const int tid = threadIdx.x;
    const int base = ((int)blockIdx.x - nwall) * NB;
    const int nb = min(NB, g.nnodes - base);
    const double* P = g.pd;
    for (int i = tid; i < 5 * Nx + 1; i += kNode64T) sRec[i] = g.rec[i];
    for (int r = tid; r < rows; r += kNode64T) {
        const double py = P[QX2 + r % VY], pz = P[QX2 + VY + r / VY];
        sRow[3 * r] = py;
        sRow[3 * r + 1] = pz;
        sRow[3 * r + 2] = py * py + pz * pz;
    }
    pdl_wait();
    pdl_trigger();
    __syncthreads();
    // 1. moments: each lane its own p_x, weighted once per column
    {
        const int k = tid / LPN, sl = tid % LPN;
        const int node = base + min(k, nb - 1);
        const InstDev& I = g.inst[g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0];
        const double* f = fs + I.f_off + (size_t)(node - I.node_off) * g.V;
        double m[5] = {0.0, 0.0, 0.0, 0.0, 0.0};             // n, j_x, j_y, j_z, E
        if (I.inv_Kn != 0.0) {
            for (int ix = sl; ix < QX2; ix += LPN) {
                double s0 = 0.0, sy = 0.0, sz = 0.0, s2 = 0.0;
                if (VZ == 1) {
#pragma unroll 8
                    for (int r = 0; r < rows; ++r) {
                        const double val = f[r * QX2 + ix];
                        s0 += val;
                        sy = fma(sRow[3 * r], val, sy);
                        s2 = fma(sRow[3 * r + 2], val, s2);
                    }
                } else {
#pragma unroll 8
                    for (int r = 0; r < rows; ++r) {
                        const double val = f[r * QX2 + ix];
                        s0 += val;
                        sy = fma(sRow[3 * r], val, sy);
                        sz = fma(sRow[3 * r + 1], val, sz);
                        s2 = fma(sRow[3 * r + 2], val, s2);
                    }
                }
                const double p = P[ix], ps = p * s0;
                m[0] += s0;
                m[1] += ps;
                m[2] += sy;
                m[3] += sz;
                m[4] += fma(p, ps, s2);
            }
            constexpr int W = LPN < 32 ? LPN : 32;
            const unsigned mask = W == 32 ? 0xffffffffu : ((1u << (W & 31)) - 1u) << (tid & 31 & ~(W - 1));   // a node's lanes
#pragma unroll
            for (int o = W / 2; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < 5; ++c) m[c] += __shfl_xor_sync(mask, m[c], o);
        }
        if (LPN > 32) {
            if ((tid & 31) == 0)
                for (int c = 0; c < 5; ++c) sPart[5 * (tid >> 5) + c] = m[c];
            __syncthreads();
            if (tid == 0)
                for (int w = 1; w < kNode64T / 32; ++w)
                    for (int c = 0; c < 5; ++c) m[c] += sPart[5 * w + c];
        }
        if (sl == 0) {
            const double in = 1.0 / m[0], ux = m[1] * in, uy = m[2] * in, uz = m[3] * in;
            double* o = sM + 6 * k;
            o[0] = m[0]; o[1] = ux; o[2] = uy; o[3] = uz;
            o[4] = (m[4] - m[0] * (ux * ux + uy * uy + uz * uz)) * in * (g.D == 3 ? 1.0 / 3.0 : (g.D == 2 ? 0.5 : 1.0));
            o[5] = m[0] * I.inv_Kn;
        }
    }
    __syncthreads();
    // 2. coefficients: p_x roles in warp 0, p_y and p_z roles in warp 1
    if (tid < 64 && (tid & 31) < 2 * NB) {
        const int k = (tid & 31) % NB, r = 2 * (tid >> 5) + ((tid & 31) / NB);
        const double* m = sM + 6 * k;
        double* G = sG + k * ncoef;
        if (k < nb && m[5] != 0.0) {
            if (r < 2 && g.quad_x) {         // G^{+-} by quadrature (quad_coef_kernel)
                const double* q = g.gquad + ((size_t)(base + k) * 2 + r) * (Nx + 1);
                for (int l = 0; l <= Nx; ++l) G[r * (Nx + 1) + l] = q[l];
            } else if (r < 2 && !g.x_full) {
                half_range_coefficients(g, r, m[1], m[4], sRec, G + r * (Nx + 1));
            } else {
                node_coefficients(g, r, m[1], m[2], m[3], m[4], sRec, G);
            }
        }
    }
    __syncthreads();
    // 3. lines, one output per thread and turn
    double* coef = static_cast<double*>(g.coef);
    const double* Tx = g.Td;
    const double* Ty = Tx + Qx * (Nx + 1);
    const double* Tz = Ty + VY * (Ny + 1);
    for (int i = tid; i < nb * g.ncp; i += kNode64T) {
        const int k = i / g.ncp, o = i - k * g.ncp;
        const double* m = sM + 6 * k;
        const double* G = sG + k * ncoef;
        double v = 0.0;
        if (o == nf) {
            v = m[5];
        } else if (g.has_field && o >= g.field_off && o < g.field_off + 3) {      // a = a_uniform + a_field(node)
            const InstDev& I = g.inst[g.ninst > 1 ? find_slot(g.node_start, g.ninst, base + k) : 0];
            const int c = o - g.field_off;
            v = (c == 0 ? I.ax : (c == 1 ? I.ay : I.az)) + g.afield[3 * (size_t)(base + k) + c];
        } else if (o < nf && m[5] != 0.0) {
            const double* T;
            int N = 0;
            bool absent = false;
            if (o < QX2) {
                const int sg = o >= Qx;
                T = Tx + (o - sg * Qx) * (Nx + 1);
                G += sg * (Nx + 1);
                N = Nx;
            } else if (o < QX2 + VY) {
                T = Ty + (o - QX2) * (Ny + 1);
                G += 2 * (Nx + 1);
                N = Ny;
                absent = !g.Qy;
            } else {
                T = Tz + (o - QX2 - VY) * (Nz + 1);
                G += 2 * (Nx + 1) + Ny + 1;
                N = Nz;
                absent = !g.Qz;
            }
            if (absent) {
                v = 1.0;
            } else {
                // eight table entries (global memory, one row per thread) at a time
                double a0 = 0.0, a1 = 0.0;
                for (int l = 0; l <= N; l += 8) {
                    double t[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) t[c] = l + c <= N ? T[l + c] : 0.0;
#pragma unroll
                    for (int c = 0; c < 8; c += 2) {
                        if (l + c <= N) a0 = fma(t[c], G[l + c], a0);
                        if (l + c + 1 <= N) a1 = fma(t[c + 1], G[l + c + 1], a1);
                    }
                }
                v = a0 + a1;
                if (o < QX2) v *= m[0];
            }
        }
        coef[(size_t)base * g.ncp + i] = v;
    }
}

}  // namespace

cudaError_t prepare_node() {
    cudaError_t e = cudaFuncSetAttribute(coef_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(coef_df_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(coef_df_kernel<12>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(coef_df_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
}

int sm_count() {
    static const int nsm = [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            n = 152;
        }
        return n;
    }();
    return nsm;
}

// Blocks of `func` resident on the whole GPU at once (one wave), at most
// `want`: a grid-stride kernel then has no partly filled last wave.
static int one_wave(const void* func, int block, size_t smem, int want) {
    const int nsm = sm_count();
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, func, block, smem) != cudaSuccess || per < 1) per = 1;
    return want < nsm * per ? (want > 0 ? want : 1) : nsm * per;
}

__global__ void df_special_kernel(const double* __restrict__ z, int n, double* __restrict__ erf_out,
                                  double* __restrict__ exp_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 zd = df_from_double(z[i]);
    const float2 z2 = df_mul(zd, zd);
    const float2 E = df_exp_nonpos(make_float2(-z2.x, -z2.y));
    const float2 er = df_erf_series(zd, z2, E);
    erf_out[i] = (double)er.x + (double)er.y;
    exp_out[i] = (double)E.x + (double)E.y;
}

cudaError_t launch_df_special(const double* z, int n, double* erf_out, double* exp_out) {
    if (n > 0) df_special_kernel<<<(n + 127) / 128, 128>>>(z, n, erf_out, exp_out);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : cudaDeviceSynchronize();
}

// Whether the one-launch node pass (sums, factor lines and walls) takes this
// FP32 group: rows of 8, 16 or 32 p_x values, the double-float lines, within the 48 KB
// of shared memory that a launch has without asking (the sets that march need
// 43.5 KB at most).
bool node_fused_available(int precision, const GroupDev& g) {
    return precision != HLB_FP64_ && g.use_df && max(g.Nx, max(g.Ny, g.Nz)) < 16 && (g.QX2 == 8 || g.QX2 == 16 || g.QX2 == 32) &&
           node_smem<32>(g).bytes <= 47 * 1024;
}

// Nodes per CTA of the one-launch node pass.  With rows of 32 values (the longest
// recurrences and dot products) a group of up to 64 nodes per SM waits on the
// chain of one CTA, and at 8 nodes the dot products take one turn of the CTA
// instead of three; else 32.  us per step of order-16 channels (GB300), 8
// against 32: 64 nodes 44.5 / 55.9, 1216 nodes 56 / 79, 4864 105 / 107, 9728
// 171 / 183, 19456 379 / 347; order 8: 1216 nodes 38.5 / 36.8, 4864 46.5 / 45.2.
static int node_nb(const GroupDev& g) { return g.QX2 == 32 && g.nnodes <= 64 * sm_count() ? 8 : 32; }

// Orders at which the recurrences' start is in double-float too (LOWN).
static bool node_low_order(const GroupDev& g) { return g.Nx <= HLB_DF_SPECIAL_MAX_N && max(g.Ny, g.Nz) < 12; }

// Whether the one-launch node pass is the faster one for a group that it can
// take.  It hides the sums' latency behind the lines and saves two launches; the
// separate kernels form the lines of 128 nodes per table load.  With few values
// per node the lines are the work and the launches are nothing in a large group.
// us per step, one launch against three (GB300): 32 x 1 velocities, order 7, 60000
// nodes 129 / 157, 130000 301 / 295, 400000 862 / 754, 3000000 6151 / 4852; order 15,
// 400000 1062 / 1157, 3000000 7593 / 7118; 16 x 8 velocities 400000 nodes 1192 /
// 1208, 3000000 8542 / 8275; 8 x 4 407 / 437 at 300000, 3675 / 3616 at 3000000; from
// 512 velocities on equal or faster at every size (16 x 8 x 8, 1000000 nodes, 15709 / 16013).
bool node_fused_pays(const GroupDev& g) {
    return g.V >= 512 || g.nnodes <= (g.QX2 == 32 && node_low_order(g) ? 1 << 17 : 1 << 19);
}

template <int ADV, int LOWN>
static void node_df_launch(const GroupDev& g, const float* fs, cudaStream_t st) {
    const int NB = node_nb(g);
    const size_t smem = NB == 8 ? node_smem<8>(g).bytes : node_smem<32>(g).bytes;
    const int grid = g.nrows * g.wchunks + (g.nnodes + NB - 1) / NB;
    if (NB == 8) launch_dependent(g.pdl, node_df_kernel<ADV, LOWN, 8>, grid, kNodeT, smem, st, g, fs);
    else launch_dependent(g.pdl, node_df_kernel<ADV, LOWN, 32>, grid, kNodeT, smem, st, g, fs);
}

void launch_node_fused(int adv, const GroupDev& g, const void* fs, cudaStream_t st) {
    const bool low = node_low_order(g);
    const float* f = static_cast<const float*>(fs);
    if (adv == HLB_WENO5_) low ? node_df_launch<HLB_WENO5_, 1>(g, f, st) : node_df_launch<HLB_WENO5_, 0>(g, f, st);
    else low ? node_df_launch<HLB_UPWIND2_, 1>(g, f, st) : node_df_launch<HLB_UPWIND2_, 0>(g, f, st);
}

// The FP64 node pass and walls (every FP64 group).
template <int ADV, int NB>
static void node_f64_launch(const GroupDev& g, const double* fs, cudaStream_t st) {
    const int grid = g.nrows * g.wchunks + (g.nnodes + NB - 1) / NB;
    launch_dependent(g.pdl, node_f64_kernel<ADV, NB>, grid, kNode64T, node64_smem(g, NB), st, g, fs);
}

template <int ADV>
static void node_f64_dispatch(const GroupDev& g, const double* fs, cudaStream_t st) {
    if (g.nnodes <= 2 * sm_count()) node_f64_launch<ADV, 1>(g, fs, st);
    else if (g.nnodes <= 16 * sm_count() || g.QX2 > 64) node_f64_launch<ADV, 8>(g, fs, st);
    else node_f64_launch<ADV, 16>(g, fs, st);
}

void launch_node_f64(int adv, const GroupDev& g, const void* fs, cudaStream_t st) {
    const double* f = static_cast<const double*>(fs);
    if (adv == HLB_WENO5_) node_f64_dispatch<HLB_WENO5_>(g, f, st);
    else node_f64_dispatch<HLB_UPWIND2_>(g, f, st);
}

// Node pass of a stage of the FP32 groups that the one-launch pass does not
// take: the quadrature sums of every node (in the first 8 values of each
// node's slot of g.sums), then the factor lines.
void launch_node(const GroupDev& g, const void* fs, cudaStream_t st) {
    const size_t smem_a = 4 * (g.V + g.VY * g.VZ) * sizeof(float);
    const int blocks_a = one_wave(reinterpret_cast<const void*>(&sums_kernel), 256, smem_a, (g.nnodes + 7) / 8);
    const int nrec = 5 * g.Nx + 1;
    sums_kernel<<<blocks_a, 256, smem_a, st>>>(g, (const float*)fs, (float*)g.sums);
    const int nmax = max(g.Nx, max(g.Ny, g.Nz));
    if (g.use_df && nmax < 16) {
        const int nP = (g.Qx + 1) / 2 * (g.Nx + 1) + (g.VY + 1) / 2 * (g.Ny + 1) + (g.VZ + 1) / 2 * (g.Nz + 1);
        const size_t smem_c = 16 * ((size_t)nP + (nrec + 1) / 2) + 4 * 32 * (size_t)g.ncp * 4;
        const int blocks_c = (g.nnodes + 127) / 128;
        if (nmax < 8) coef_df_kernel<8><<<blocks_c, 128, smem_c, st>>>(g, (const float*)g.sums);
        else if (nmax < 12) coef_df_kernel<12><<<blocks_c, 128, smem_c, st>>>(g, (const float*)g.sums);
        else coef_df_kernel<16><<<blocks_c, 128, smem_c, st>>>(g, (const float*)g.sums);
    } else {
        const int nT = g.Qx * (g.Nx + 1) + g.VY * (g.Ny + 1) + g.VZ * (g.Nz + 1);
        const int ncoef = 2 * (g.Nx + 1) + (g.Ny + 1) + (g.Nz + 1);
        const size_t smem_b = 8 * (nrec + nT) + 8 * (32 * ncoef + 64) + 32 * sizeof(NodeDF);
        coef_kernel<<<(g.nnodes + 31) / 32, 32, smem_b, st>>>(g, (const float*)g.sums);
    }
}

}  // namespace hlb
