// Device kernels of libhlb (sm_103a).
//
// Per RK-3 stage (Eq. "eq:rk3") these kernels run (the marching kernels of
// hlb_march.cu, hlb_pair.cuh, hlb_line.cuh take the stage kernel's place
// where they apply):
//   quad_coef_kernel  FP64 half-range groups above order 12: the half-range
//                 equilibrium coefficients of every collisional node by
//                 quadrature of the projection integrals (see below).
//   wall_kernel   (where the node pass does not hold it) one or a few CTAs per (instance, y-row): incident fluxes at
//                 both wall faces from the quadratically extrapolated ghosts
//                 (Sec. IV.C.3), summed in FP64, give the emitted densities
//                 n_w = -sum_inc F / sum_emit p_x g^w (Eq. "eq:nplus_def").
//   stage_kernel  fused per node: moments (Eq. "eq:fmoms") by a block
//                 reduction and the equilibrium factors g_x, g_y, g_z (FP64
//                 recurrences, App. A; FP64 groups read both from the node
//                 pass of hlb_node.cu), the force term sum_a a_a K_a f
//                 (Eqs. "eq:hh_Kk_hh", "eq:H_Kk"; a the uniform acceleration
//                 plus the node's field value), BGK with tau = Kn/n,
//                 WENO-5 / upwind2 fluxes along x (walls: Eq.
//                 "eq:weno_populate" ghosts) and y (periodic), and the RK-3
//                 combination; writes the stage output.  It serves the
//                 shapes the marching kernels do not, among them the
//                 half-range sets beyond Qx = 32 in 2D: there K_x stays in
//                 global memory, its cross-half blocks enter as their rank-one
//                 factor, and a node's velocities are split over several CTAs.
//   stage_wide_kernel  the same stage for the sets beyond Qx = 32 in 1D (the
//                 HHLB(20;200) model of Sec. V).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "hlb_internal.h"
#include "hlb_device.cuh"
#include "hlb_wall.cuh"

namespace hlb {

namespace {

// Shared-memory layout of the stage kernel (sizes in elements).
struct SmemLayout {
    int nK, nP, nT, nG;
    size_t offK, offP, offT, offF, offG;      // in R elements
    size_t offD;                              // in bytes (8-aligned)
    int nRec, nCoef;
    int nJ;                                   // doubles: per-fibre cross-half sums (kx_global)
    size_t bytes;
};

template <typename R>
__host__ __device__ inline SmemLayout smem_layout(const GroupDev& g, int nwarps) {
    SmemLayout L;
    L.nK = (g.kx_global ? 0 : g.QX2 * g.QX2) + g.VY * g.VY + g.VZ * g.VZ;
    L.nP = g.QX2 + g.VY + g.VZ;
    L.nT = g.Qx * (g.Nx + 1) + g.VY * (g.Ny + 1) + g.VZ * (g.Nz + 1);
    L.nG = g.QX2 + g.VY + g.VZ;
    L.offK = 0;
    L.offP = L.offK + L.nK;
    L.offT = L.offP + L.nP;
    L.offF = L.offT + L.nT;
    L.offG = L.offF + g.V;
    size_t rbytes = (L.offG + L.nG) * sizeof(R);
    L.offD = (rbytes + 15) & ~size_t(15);
    L.nRec = 5 * g.Nx + 1;
    L.nCoef = 2 * (g.Nx + 1) + (g.Ny + 1) + (g.Nz + 1);
    L.nJ = g.kx_global ? 2 * g.VY * g.VZ : 0;
    // doubles: rec, coef, 8 scalars, 5 * nwarps reduction slots, cross-half sums
    L.bytes = L.offD + sizeof(double) * (L.nRec + L.nCoef + 8 + 5 * nwarps + L.nJ);
    return L;
}

// Value of velocity v at x-position pos of a row (ghost rules at the walls).
template <typename R>
__device__ __forceinline__ R x_value(const R* __restrict__ frow, int pos, int nx, int V, int v,
                                     bool px_pos, R nwl_g, R nwr_g) {
    if (pos >= 0 && pos < nx) return frow[(size_t)pos * V + v];
    if (pos < 0) {
        if (px_pos) return nwl_g;                        // emitted: n_w g^w (3 ghosts)
        const R f0 = frow[v], f1 = frow[(size_t)V + v], f2 = frow[2 * (size_t)V + v];
        if (pos == -1) return R(3) * f0 - R(3) * f1 + f2;            // paper's cell 0
        return R(6) * f0 - R(8) * f1 + R(3) * f2;                     // paper's cell -1
    }
    if (!px_pos) return nwr_g;
    const R f0 = frow[(size_t)(nx - 1) * V + v], f1 = frow[(size_t)(nx - 2) * V + v],
            f2 = frow[(size_t)(nx - 3) * V + v];
    if (pos == nx) return R(3) * f0 - R(3) * f1 + f2;
    return R(6) * f0 - R(8) * f1 + R(3) * f2;
}

// Fluxes at the faces x+1/2 and x-1/2 (per unit velocity) from a 6-cell
// window; w[] holds cells x-3..x+2 for v > 0 and x-2..x+3 for v < 0.
template <typename R, int ADV>
__device__ __forceinline__ void face_pair(const R* w, bool pos, R& Fp, R& Fm) {
    if constexpr (ADV == HLB_WENO5_ && sizeof(R) == 8) {
        double u[6], F[2];
#pragma unroll
        for (int j = 0; j < 6; ++j) u[j] = pos ? w[j] : w[5 - j];
        weno5_faces64<2>(u, F);
        Fp = pos ? F[1] : F[0];
        Fm = pos ? F[0] : F[1];
    } else if (ADV == HLB_WENO5_) {
        if (pos) {
            Fp = weno5_face(w[1], w[2], w[3], w[4], w[5]);
            Fm = weno5_face(w[0], w[1], w[2], w[3], w[4]);
        } else {
            Fp = weno5_face(w[5], w[4], w[3], w[2], w[1]);
            Fm = weno5_face(w[4], w[3], w[2], w[1], w[0]);
        }
    } else {
        if (pos) {
            Fp = upwind2_face(w[2], w[3]);
            Fm = upwind2_face(w[1], w[2]);
        } else {
            Fp = upwind2_face(w[4], w[3]);
            Fm = upwind2_face(w[3], w[2]);
        }
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// stage kernel
// ---------------------------------------------------------------------------
// CTAs per SM the generic stage kernel is compiled for: two, at most 128
// registers per thread.  us per stage against one (GB300): 24 x 6 cells of 400
// FP64 velocities 60 / 78, 24 x 40 314 / 357; 64 x 64 of 1024 FP32 velocities with a
// force along p_z 548 / 875.
constexpr int kStageMinBlocks = 2;
template <typename R, int ADV>
__global__ void __launch_bounds__(256, kStageMinBlocks)
stage_kernel(const GroupDev g, const R* __restrict__ fs, const R* __restrict__ fn,
             R* __restrict__ fo, int stage) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nwarps = blockDim.x >> 5;
    const SmemLayout L = smem_layout<R>(g, nwarps);
    R* sR = reinterpret_cast<R*>(smem_raw);
    R* sK = sR + L.offK;
    R* sP = sR + L.offP;
    R* sT = sR + L.offT;
    R* sF = sR + L.offF;
    R* sG = sR + L.offG;
    double* sD = reinterpret_cast<double*>(smem_raw + L.offD);
    double* sRec = sD;
    double* sCoef = sRec + L.nRec;
    double* sScal = sCoef + L.nCoef;
    double* sRed = sScal + 8;
    double* sJ = sRed + 5 * nwarps;           // [fibre][2]: sum_{k' in half} d_k' f_k'

    const int tid = threadIdx.x, bs = blockDim.x, lane = tid & 31, warp = tid >> 5;
    // Kx stays in global memory (read through KxT) when it exceeds the
    // shared-memory budget; sK then holds Ky and Kz only
    const R* gK = static_cast<const R*>(g.K) + (g.kx_global ? g.QX2 * g.QX2 : 0);
    const R* gP = static_cast<const R*>(g.p);
    const R* gT = static_cast<const R*>(g.Tt);
    for (int i = tid; i < L.nK; i += bs) sK[i] = gK[i];
    for (int i = tid; i < L.nP; i += bs) sP[i] = gP[i];
    if (sizeof(R) == 4) {                     // FP64 groups read the node pass's lines instead
        for (int i = tid; i < L.nT; i += bs) sT[i] = gT[i];
        for (int i = tid; i < L.nRec; i += bs) sRec[i] = g.rec[i];
    }
    __syncthreads();

    const int V = g.V, QX2 = g.QX2, VY = g.VY, VZ = g.VZ, Qx = g.Qx;
    const R* sKx = sK;
    const R* sKy = sK + (g.kx_global ? 0 : QX2 * QX2);
    const R* sKz = sKy + VY * VY;
    const R* sPx = sP;
    const R* sPy = sP + QX2;
    const R* sPz = sPy + VY;
    const R* sTx = sT;
    const R* sTy = sT + Qx * (g.Nx + 1);
    const R* sTz = sTy + VY * (g.Ny + 1);
    const R* gw = static_cast<const R*>(g.gw);

    // work items: (node, velocity range); one range per node unless Kx is
    // read from global memory (vchunks > 1)
    const int nvc = g.vchunks;
    for (int item = blockIdx.x; item < g.nnodes * nvc; item += gridDim.x) {
        const int node = item / nvc, chunk = item - node * nvc;
        const int v0 = (int)((long long)chunk * V / nvc), v1 = (int)((long long)(chunk + 1) * V / nvc);
        const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
        const InstDev I = g.inst[ii];
        const int local = node - I.node_off;
        const int nx = I.nx;
        const int y = local / nx, x = local - y * nx;
        const size_t row_off = (size_t)I.f_off + (size_t)y * nx * V;
        const R* frow = fs + row_off;

        // Collisionless instances (Kn = +inf) have no BGK term at all: no
        // moments and no equilibrium are formed for them.
        const bool collide = I.inv_Kn != 0.0;
        // FP64 groups: the node pass has formed the factors and 1/tau
        // (node_f64_kernel); FP32 groups form them here, per node
        const R* line = static_cast<const R*>(g.coef) + (size_t)node * g.ncp;
        const bool form = collide && sizeof(R) == 4;
        if (collide && sizeof(R) == 8)
            for (int t = tid; t < QX2 + VY + VZ; t += bs) sG[t] = line[t];
        // 1. node values and moment partial sums, accumulated in FP64 for
        // either state precision (T = (E - n|u|^2)/(D n) cancels digits, and
        // the FP32 state's sums are not compensated here)
        double a0 = 0, a1 = 0, a2 = 0, a3 = 0, a4 = 0;
        for (int v = tid; v < V; v += bs) {
            const R val_r = frow[(size_t)x * V + v];
            sF[v] = val_r;
            if (!form) continue;
            const int ix = v % QX2, jy = (v / QX2) % VY, kz = v / (QX2 * VY);
            const double px = sPx[ix], py = sPy[jy], pz = sPz[kz], val = val_r;
            a0 += val;
            a1 += px * val;
            a2 += py * val;
            a3 += pz * val;
            a4 += (px * px + py * py + pz * pz) * val;
        }
        if (form) {
        a0 = warp_sum(a0); a1 = warp_sum(a1); a2 = warp_sum(a2); a3 = warp_sum(a3); a4 = warp_sum(a4);
        if (lane == 0) {
            sRed[warp * 5 + 0] = a0; sRed[warp * 5 + 1] = a1; sRed[warp * 5 + 2] = a2;
            sRed[warp * 5 + 3] = a3; sRed[warp * 5 + 4] = a4;
        }
        __syncthreads();
        if (tid < 4) {
            double m[5] = {0, 0, 0, 0, 0};
            for (int w = 0; w < nwarps; ++w)
                for (int k = 0; k < 5; ++k) m[k] += sRed[w * 5 + k];
            const double n = m[0];
            const double ux = m[1] / n, uy = m[2] / n, uz = m[3] / n;
            const double T = (m[4] - n * (ux * ux + uy * uy + uz * uz)) / (g.D * n);
            if (tid == 0) {
                sScal[0] = n;
                sScal[1] = n * I.inv_Kn;     // 1/tau
            }
            node_coefficients(g, tid, ux, uy, uz, T, sRec, sCoef);
        }
        __syncthreads();
        // 2. equilibrium factors g_x (times n), g_y, g_z
        {
            const int nf = QX2 + VY + VZ;
            for (int t = tid; t < nf; t += bs) {
                double acc = 0.0;
                if (t < QX2) {
                    const int k = t % Qx, sg = t / Qx;
                    const double* G = sCoef + sg * (g.Nx + 1);
                    for (int l = 0; l <= g.Nx; ++l) acc += (double)sTx[k * (g.Nx + 1) + l] * G[l];
                    acc *= sScal[0];
                } else if (t < QX2 + VY) {
                    const int j = t - QX2;
                    if (g.Qy) {
                        const double* G = sCoef + 2 * (g.Nx + 1);
                        for (int l = 0; l <= g.Ny; ++l) acc += (double)sTy[j * (g.Ny + 1) + l] * G[l];
                    } else {
                        acc = 1.0;
                    }
                } else {
                    const int k = t - QX2 - VY;
                    if (g.Qz) {
                        const double* G = sCoef + 2 * (g.Nx + 1) + (g.Ny + 1);
                        for (int l = 0; l <= g.Nz; ++l) acc += (double)sTz[k * (g.Nz + 1) + l] * G[l];
                    } else {
                        acc = 1.0;
                    }
                }
                sG[t] = (R)acc;
            }
        }
        }  // form
        __syncthreads();
        if (g.kx_global) {
            // K^h = blockdiag(same-half blocks) + the rank-one jump term
            // c_k d_k' in every block (Eq. "eq:hh_Kk_hh"): the cross-half
            // blocks enter through one sum per fibre and half
            const double* jd = g.KxJ + QX2;
            const int nfib = VY * VZ;
            for (int fh = warp; fh < 2 * nfib; fh += nwarps) {
                const int fb = fh >> 1, h = fh & 1;
                const R* fr = sF + (size_t)fb * QX2 + h * Qx;
                double acc = 0.0;
                for (int i = lane; i < Qx; i += 32) acc += jd[h * Qx + i] * (double)fr[i];
                acc = warp_sum(acc);
                if (lane == 0) sJ[fh] = acc;
            }
            __syncthreads();
        }

        const R inv_tau = !collide ? R(0) : (sizeof(R) == 8 ? line[QX2 + VY + VZ] : (R)sScal[1]);
        const R dt = (R)I.dt;
        const R inv_dx = (R)(1.0 / g.dx[I.dx_off + x]);
        const R inv_dy = (R)I.inv_dy;
        // the uniform acceleration plus the node's field value (hlb_set_force_field)
        const double* af = g.has_field ? g.afield + 3 * (size_t)node : nullptr;
        const R ax = (R)(I.ax + (af ? af[0] : 0.0)), ay = (R)(I.ay + (af ? af[1] : 0.0)),
                az = (R)(I.az + (af ? af[2] : 0.0));
        const double nwl = g.nw[(size_t)(I.row_off + y) * 2 + 0];
        const double nwr = g.nw[(size_t)(I.row_off + y) * 2 + 1];
        const R* gwl = gw + I.gw_off;
        const R* gwr = gwl + V;
        const int ny = I.ny;

        // 3. per velocity of the range
        for (int v = v0 + tid; v < v1; v += bs) {
            const int ix = v % QX2, jy = (v / QX2) % VY, kz = v / (QX2 * VY);
            const R f = sF[v];
            const R feq = collide ? sG[ix] * sG[QX2 + jy] * sG[QX2 + VY + kz] : R(0);
            // force: sum_a a_a (K_a f)
            R force = 0;
            if (ax != R(0)) {
                const R* fr = sF + (v - ix);
                R acc = 0;
                if (g.kx_global) {
                    // own half: column ix of Kx^T (consecutive threads read
                    // consecutive entries; four partial sums shorten the
                    // dependent chain); other half: c_ix times its fibre sum
                    const int h = ix < Qx ? 0 : 1;
                    const double* Kc = g.KxT + (size_t)h * Qx * QX2 + ix;
                    const R* fh = fr + h * Qx;
                    R a4[4] = {0, 0, 0, 0};
                    int i = 0;
                    for (; i + 4 <= Qx; i += 4) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) a4[q] += (R)Kc[(size_t)(i + q) * QX2] * fh[i + q];
                    }
                    for (; i < Qx; ++i) a4[0] += (R)Kc[(size_t)i * QX2] * fh[i];
                    const int fb = (v - ix) / QX2;
                    acc = (a4[0] + a4[1]) + (a4[2] + a4[3]) + (R)(g.KxJ[ix] * sJ[2 * fb + (1 - h)]);
                } else {
                    const R* Kr = sKx + ix * QX2;
                    for (int i = 0; i < QX2; ++i) acc += Kr[i] * fr[i];
                }
                force += ax * acc;
            }
            if (ay != R(0) && g.Qy) {
                const R* Kr = sKy + jy * VY;
                const R* fr = sF + (v - jy * QX2);
                R acc = 0;
                for (int j = 0; j < VY; ++j) acc += Kr[j] * fr[j * QX2];
                force += ay * acc;
            }
            if (az != R(0) && g.Qz) {
                const R* Kr = sKz + kz * VZ;
                const R* fr = sF + (v - kz * QX2 * VY);
                R acc = 0;
                for (int k = 0; k < VZ; ++k) acc += Kr[k] * fr[(size_t)k * QX2 * VY];
                force += az * acc;
            }
            // advection along x
            const R vx = sPx[ix];
            const bool xpos = ix < Qx;
            R w[6];
            const int base = xpos ? x - 3 : x - 2;
            const R nwl_g = (R)nwl * gwl[v], nwr_g = (R)nwr * gwr[v];
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = x_value(frow, base + k, nx, V, v, xpos, nwl_g, nwr_g);
            R Fp, Fm;
            face_pair<R, ADV>(w, xpos, Fp, Fm);
            R Lval = -vx * (Fp - Fm) * inv_dx;
            // advection along y (periodic)
            if (ny > 1) {
                const R vy = sPy[jy];
                const bool ypos = vy > R(0);
                const int yb = ypos ? y - 3 : y - 2;
                const R* fcol = fs + (size_t)I.f_off + (size_t)x * V + v;
                const size_t rstride = (size_t)nx * V;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    int yy = yb + k;
                    yy += (yy < 0) ? ny : 0;
                    yy -= (yy >= ny) ? ny : 0;
                    w[k] = fcol[(size_t)yy * rstride];
                }
                R Gp, Gm;
                face_pair<R, ADV>(w, ypos, Gp, Gm);
                Lval -= vy * (Gp - Gm) * inv_dy;
            }
            Lval -= force;
            if (collide) Lval -= (f - feq) * inv_tau;
            R out;
            bool done = false;
            if constexpr (sizeof(R) == 4) {
                if (g.sround) {      // stochastic rounding of the stage output (hlb_device.cuh)
                    R* dst = fo + row_off + (size_t)x * V + v;
                    *dst = rk3_out_sr(stage, f, -(dt * Lval), stage > 0 ? fn[row_off + (size_t)x * V + v] : R(0),
                                      sr_key(dst));
                    done = true;
                }
            }
            if (!done) {
                if (stage == 0) {
                    out = f + dt * Lval;
                } else {
                    const R fnv = fn[row_off + (size_t)x * V + v];
                    // c f^n + (1 - c) f' as f' + c (f^n - f'): the weights sum to
                    // 1 exactly whatever the rounding of c
                    const R fp = f + dt * Lval;
                    out = fp + (stage == 1 ? R(0.75) : R(1.0 / 3.0)) * (fnv - fp);
                }
                fo[row_off + (size_t)x * V + v] = out;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// stage kernel of the wide FP64 sets (K_x in global memory) without a y axis in
// space: the HHLB(20;200) runs
// ---------------------------------------------------------------------------
// One thread per velocity and pair of neighbouring cells, the (pair, velocity)
// list cut into CTAs of 64 whatever fibre they fall in.  The FP64 pipe is the
// bound (a warp's instruction takes 64 cycles of its SM quarter), so what counts
// is the number of FP64 operations and an even number of full warps per
// quarter: two cells share the faces between them (three instead of four, at a
// common scale) and every K_x entry read from L2, and no warp is cut short at a
// node's end (400 velocities are 12.5 warps; in seven CTAs of 64 per node they
// took 14 and 4.4 rounds of the resident CTAs, here 12.5 and 2).  Per stage
// (GB300): eight ballistic cases 43.6 us against 63.9 in the generic kernel.
//   A group of few cells leaves SM quarters idle that way (one transition-regime
// run of 72 cells: 450 warps for 608 quarters), and is spread at one cell per
// thread (NC = 1).
constexpr int kWideThreads = 64;
template <int NC>
struct alignas(8 * NC) CellVals {            // one population's values at a thread's cells
    double c[NC];
};
template <int ADV, int NC>
__global__ void __launch_bounds__(kWideThreads, 4)
stage_wide_kernel(const GroupDev g, const double* __restrict__ fs, const double* __restrict__ fn,
                  double* __restrict__ fo, int stage) {
    extern __shared__ __align__(16) unsigned char wsm[];
    const int V = g.V, QX2 = g.QX2, Qx = g.Qx, VY = g.VY, VZ = g.VZ, nfib = VY * VZ;
    CellVals<NC>* sF = reinterpret_cast<CellVals<NC>*>(wsm);         // [2 fibres][QX2]
    CellVals<NC>* sJ = sF + 2 * QX2;                                      // [2 fibres][2 halves]: sum_{k' in half} d_k' f_k'
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int* start = NC == 2 ? g.pair_start : g.node_start;        // cell pairs or cells before each instance
    const long long total = (long long)(NC == 2 ? g.npairs : g.nnodes) * V;
    const long long e0 = (long long)blockIdx.x * kWideThreads;
    const long long fib0 = e0 / QX2;                                 // first fibre of the CTA, over all pairs
    const long long last = min(total, e0 + kWideThreads) - 1;
    const int nfb = (int)(last / QX2 - fib0) + 1;                    // one or two (QX2 > 64)
    for (int a = 0; a < nfb; ++a) {
        const int pair = (int)((fib0 + a) / nfib), fb = (int)((fib0 + a) - (long long)pair * nfib);
        const int ii = g.ninst > 1 ? find_slot(start, g.ninst, pair) : 0;
        const InstDev& I = g.inst[ii];
        const int x0 = NC * (pair - start[ii]);
        const double* f = fs + I.f_off + (size_t)x0 * V + (size_t)fb * QX2;
        const bool two = NC == 2 && x0 + 1 < I.nx;
        for (int i = tid; i < QX2; i += kWideThreads) {
            CellVals<NC> val;
            val.c[0] = f[i];
            if (NC == 2) val.c[NC - 1] = two ? f[V + i] : 0.0;
            sF[a * QX2 + i] = val;
        }
    }
    __syncthreads();
    {
        // the cross-half blocks of K^h are rank one, c_k d_k': one sum per fibre,
        // half and cell (only of halves that a thread of the CTA needs)
        const double* jd = g.KxJ + QX2;
        for (int j = warp; j < 2 * nfb; j += kWideThreads / 32) {
            const int a = j >> 1, h = j & 1;
            const long long b = (fib0 + a) * QX2 + (h ? 0 : Qx);     // the other half's values
            if (b > last || b + Qx <= e0) continue;
            CellVals<NC> s = {};
            for (int i = lane; i < Qx; i += 32) {
                const double d = jd[h * Qx + i];
                const CellVals<NC> f = sF[a * QX2 + h * Qx + i];
#pragma unroll
                for (int c = 0; c < NC; ++c) s.c[c] = fma(d, f.c[c], s.c[c]);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) s.c[c] = warp_sum(s.c[c]);
            if (lane == 0) sJ[j] = s;
        }
    }
    __syncthreads();
    const long long e = e0 + tid;
    if (e >= total) return;
    const int a = (int)(e / QX2 - fib0), ix = (int)(e % QX2);
    const int pair = (int)(e / V), v = (int)(e - (long long)pair * V);
    const int jy = (v / QX2) % VY, kz = v / (QX2 * VY);
    const int ii = g.ninst > 1 ? find_slot(start, g.ninst, pair) : 0;
    const InstDev& I = g.inst[ii];
    const int nx = I.nx, x0 = NC * (pair - start[ii]);
    const bool two = NC == 2 && x0 + 1 < nx, xpos = ix < Qx;
    const double* frow = fs + I.f_off;
    // fluxes per unit velocity at x0 - 1/2, x0 + 1/2 (and x0 + 3/2)
    constexpr int NF = NC + 1;
    double Fx[NF];
    {
        const double* gw = static_cast<const double*>(g.gw) + I.gw_off;
        const double nwl_g = g.nw[(size_t)I.row_off * 2 + 0] * gw[v], nwr_g = g.nw[(size_t)I.row_off * 2 + 1] * gw[V + v];
        double w[NF + 4];
        const int base = xpos ? x0 - 3 : x0 - 2;
#pragma unroll
        for (int k = 0; k < NF + 4; ++k) w[k] = x_value(frow, base + k, nx, V, v, xpos, nwl_g, nwr_g);
        if (ADV == HLB_WENO5_) {
            double u[NF + 4], F[NF];
#pragma unroll
            for (int k = 0; k < NF + 4; ++k) u[k] = xpos ? w[k] : w[NF + 3 - k];
            weno5_faces64<NF>(u, F);
#pragma unroll
            for (int k = 0; k < NF; ++k) Fx[k] = xpos ? F[k] : F[NF - 1 - k];
        } else {
#pragma unroll
            for (int k = 0; k < NF; ++k)
                Fx[k] = xpos ? upwind2_face(w[k + 1], w[k + 2]) : upwind2_face(w[k + 3], w[k + 2]);
        }
    }
    // a_x K_x f + a_y K_y f + a_z K_z f at the cells (accelerations; at the last cell c1 too)
    const int node0 = I.node_off + x0;
    constexpr int c1 = NC - 1;
    double acc3[3][NC] = {};
    double acl[NC][3];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const double* af = g.has_field && (c == 0 || two) ? g.afield + 3 * (size_t)(node0 + c) : nullptr;
        acl[c][0] = I.ax + (af ? af[0] : 0.0);
        acl[c][1] = I.ay + (af ? af[1] : 0.0);
        acl[c][2] = I.az + (af ? af[2] : 0.0);
    }
    if (acl[0][0] != 0.0 || acl[c1][0] != 0.0) {
        // own half: column ix of Kx^T (consecutive threads read consecutive
        // entries), eight entries ahead of the sums; other half: c_ix times its sum
        const int h = xpos ? 0 : 1;
        const double* Kc = g.KxT + (size_t)h * Qx * QX2 + ix;
        const CellVals<NC>* fh = sF + a * QX2 + h * Qx;
        double p[NC][2] = {};
        constexpr int U = 8;
        double kc[U];
        const int n8 = Qx / U * U;
#pragma unroll
        for (int j = 0; j < U; ++j) kc[j] = Kc[(size_t)j * QX2];
        for (int i = 0; i < n8; i += U) {
            double kn[U];
            const bool more = i + U < n8;
#pragma unroll
            for (int j = 0; j < U; ++j) kn[j] = more ? Kc[(size_t)(i + U + j) * QX2] : 0.0;
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const CellVals<NC> f0 = fh[i + j];
#pragma unroll
                for (int c = 0; c < NC; ++c) p[c][j & 1] = fma(kc[j], f0.c[c], p[c][j & 1]);
            }
#pragma unroll
            for (int j = 0; j < U; ++j) kc[j] = kn[j];
        }
        for (int i = n8; i < Qx; ++i) {
            const double k = Kc[(size_t)i * QX2];
            const CellVals<NC> f0 = fh[i];
#pragma unroll
            for (int c = 0; c < NC; ++c) p[c][0] = fma(k, f0.c[c], p[c][0]);
        }
        const CellVals<NC> J = sJ[2 * a + 1 - h];
        const double cj = g.KxJ[ix];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc3[0][c] = fma(cj, J.c[c], p[c][0] + p[c][1]);
    }
    const double* f0p = frow + (size_t)x0 * V;
    const double* Ky = static_cast<const double*>(g.K) + (size_t)QX2 * QX2;
    if (g.Qy && (acl[0][1] != 0.0 || acl[c1][1] != 0.0))
        for (int j = 0; j < VY; ++j) {
            const double k = Ky[jy * VY + j];
            const size_t o = (size_t)(kz * VY + j) * QX2 + ix;
            acc3[1][0] = fma(k, f0p[o], acc3[1][0]);
            if (two) acc3[1][c1] = fma(k, f0p[V + o], acc3[1][c1]);
        }
    if (g.Qz && (acl[0][2] != 0.0 || acl[c1][2] != 0.0))
        for (int j = 0; j < VZ; ++j) {
            const double k = Ky[VY * VY + kz * VZ + j];
            const size_t o = (size_t)(j * VY + jy) * QX2 + ix;
            acc3[2][0] = fma(k, f0p[o], acc3[2][0]);
            if (two) acc3[2][c1] = fma(k, f0p[V + o], acc3[2][c1]);
        }
    const double vx = g.pd[ix], dt = I.dt;
    const double* idx = static_cast<const double*>(g.inv_dx) + I.dx_off + x0;
    const CellVals<NC> fc = sF[a * QX2 + ix];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        if (c == 1 && !two) break;
        double force = acl[c][0] * acc3[0][c];
        if (g.Qy) force = fma(acl[c][1], acc3[1][c], force);
        if (g.Qz) force = fma(acl[c][2], acc3[2][c], force);
        const double f = fc.c[c];
        double L = -vx * (Fx[c + 1] - Fx[c]) * idx[c] - force;
        if (I.inv_Kn != 0.0) {
            const double* line = static_cast<const double*>(g.coef) + (size_t)(node0 + c) * g.ncp;
            L -= (f - line[ix] * line[QX2 + jy] * line[QX2 + VY + kz]) * line[QX2 + VY + VZ];
        }
        const size_t o = (size_t)I.f_off + (size_t)(x0 + c) * V + v;
        double out = fma(dt, L, f);
        // c f^n + (1 - c) f' as f' + c (f^n - f'): the weights sum to 1 exactly
        if (stage > 0) out = fma(stage == 1 ? 0.75 : 1.0 / 3.0, fn[o] - out, out);
        fo[o] = out;
    }
}

// ---------------------------------------------------------------------------
// wall kernel: emitted densities of both walls of one (instance, y) row
// ---------------------------------------------------------------------------
template <typename R, int ADV>
__global__ void __launch_bounds__(256)
wall_kernel(const GroupDev g, const R* __restrict__ fs) {
    __shared__ double red[16];
    wall_block<R, ADV>(g, fs, blockIdx.x, red);
}

// ---------------------------------------------------------------------------
// The half-range equilibrium coefficients of FP64 groups above the
// recurrence's stable order: G^{+-}_l = int_0^inf g(+-p) h_l(p) dp (l <= Nx),
// g the Gaussian of the node's u_x and T (Sec. IV.B, the projection of Eq.
// "eq:hh_gk"), by composite Gauss-Legendre quadrature over [0, |u_x| +
// 13 sqrt(T)] in panels of 1.5 sqrt(T) (kQuadNodes = 24 points each: 216 to 240
// points while |u_x| <= 2 sqrt(T); beyond the end g h_l is below 1e-17 of its
// maximum for l <= 31; 3.7e-15 of max |G| at order 20 against a 30-point rule on
// panels of 0.1 sqrt(T) in extended precision, 3.8e-15 with 20 points on panels of
// sqrt(T); 2.6e-14 at orders 20 and 31 over T from 0.05 to 30 and |u_x| up to 5, the
// rounding of the FP64 recurrence), h_l(p) by the three-term recurrence of the orthonormal basis
// (forward evaluation at a point is stable).  The integration-by-parts
// recurrence of node_coefficients carries its rounding (and that of its erf
// and exp start) along a solution that grows about threefold per order:
// 5e-7 of max g at N = 20.  One CTA per node and sign (72 nodes fill 144 of 152
// SMs; both signs in one CTA save the second evaluation of h_l(p), 2 of 5
// operations per point and order, but leave half the SMs idle), 128 threads of
// two points each (one warp per SM quarter: the FP64 pipe is the bound, and 260 to
// 300 points would take every quarter a third round), their sums over the CTA
// through shared memory (the FP64 adds of a full-warp butterfly for every order
// cost as much as the points).  72 nodes at order 20: 18.7 us per stage, 25 with
// three rounds and two more divisions, 44 with one CTA of 256 threads per node and
// butterflies (GB300).
// ---------------------------------------------------------------------------
constexpr int kQuadThreads = 128;
template <int NMAX>
__global__ void __launch_bounds__(kQuadThreads) quad_coef_kernel(const GroupDev g, const double* __restrict__ fs) {
    __shared__ double part[NMAX][kQuadThreads + 1];
    __shared__ double red[kQuadThreads / 32][5];
    __shared__ double sMom[2];
    const int node = blockIdx.x >> 1, sg = blockIdx.x & 1;
    const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
    const InstDev& I = g.inst[ii];
    if (I.inv_Kn == 0.0) return;                // collisionless: no equilibrium is formed
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kQuadThreads / 32;
    const int V = g.V, QX2 = g.QX2, VY = g.VY, Nx = g.Nx;
    const double* f = fs + I.f_off + (size_t)(node - I.node_off) * V;
    // moments of the node
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0, a4 = 0.0;
#pragma unroll 4
    for (int v = tid; v < V; v += kQuadThreads) {
        const double val = f[v];
        const double px = g.pd[v % QX2], pv = px * val;
        a0 += val;
        a1 += pv;
        a4 = fma(px, pv, a4);
        if (V > QX2) {                          // p_y, p_z
            const double py = g.pd[QX2 + (v / QX2) % VY], pz = g.pd[QX2 + VY + v / (QX2 * VY)];
            a2 = fma(py, val, a2);
            a3 = fma(pz, val, a3);
            a4 = fma(fma(py, py, pz * pz), val, a4);
        }
    }
    a0 = warp_sum(a0); a1 = warp_sum(a1); a4 = warp_sum(a4);
    if (V > QX2) { a2 = warp_sum(a2); a3 = warp_sum(a3); }
    if (lane == 0) { red[warp][0] = a0; red[warp][1] = a1; red[warp][2] = a2; red[warp][3] = a3; red[warp][4] = a4; }
    __syncthreads();
    if (tid == 0) {
        double m[5] = {0, 0, 0, 0, 0};
        for (int w = 0; w < nw; ++w)
            for (int k = 0; k < 5; ++k) m[k] += red[w][k];
        const double n = m[0], in = 1.0 / n, ux = m[1] * in, uy = m[2] * in, uz = m[3] * in;
        sMom[0] = ux;
        sMom[1] = (m[4] - n * (ux * ux + uy * uy + uz * uz)) * in * (g.D == 3 ? 1.0 / 3.0 : (g.D == 2 ? 0.5 : 1.0));
    }
    __syncthreads();
    const double ux = sMom[0], T = sMom[1];
    const double sT = sqrt(T), isT = 1.0 / sT, width = kQuadWidth * sT;
    const int panels = (int)ceil(fma(fabs(ux), isT, 13.0) * (1.0 / kQuadWidth));
    const int npts = panels * kQuadNodes;
    const double norm = isT * (1.0 / kSqrt2Pi), i2T = 0.5 * isT * isT, u = sg ? -ux : ux;
    const double* ra = g.rec;
    const double* rb = g.rec + Nx;
    const double* rc = g.rec + 2 * Nx;
    const double h00 = g.rec[3 * Nx];
    double G[NMAX];
#pragma unroll
    for (int l = 0; l < NMAX; ++l) G[l] = 0.0;
    for (int k = tid; k < npts; k += kQuadThreads) {
        const int pnl = k / kQuadNodes, i = k - pnl * kQuadNodes;
        const double p = (pnl + 0.5 * (1.0 + g.glrule[i])) * width;
        const double d = p - u;
        const double w = 0.5 * width * g.glrule[kQuadNodes + i] * norm * exp(-d * d * i2T);
        double hm = 0.0, h = w * h00;            // the weight times h_l(p): the recurrence is linear
        G[0] += h;
#pragma unroll
        for (int l = 0; l < NMAX - 1; ++l) {
            if (l < Nx) {
                const double hn = fma(fma(ra[l], p, rb[l]), h, rc[l] * hm);
                hm = h;
                h = hn;
                G[l + 1] += h;
            }
        }
    }
#pragma unroll
    for (int l = 0; l < NMAX; ++l)
        if (l <= Nx) part[l][tid] = G[l];
    __syncthreads();
    double* out = g.gquad + ((size_t)node * 2 + sg) * (Nx + 1);
    // four threads per order, 32 partial sums each
    static_assert(4 * NMAX <= kQuadThreads, "four threads per order");
    if (tid < 4 * NMAX) {                        // whole warps: NMAX is a multiple of 8
        const int l = min(tid >> 2, Nx), q = tid & 3;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll 4
        for (int i = q; i < kQuadThreads; i += 16) {
            s0 += part[l][i];
            s1 += part[l][i + 4];
            s2 += part[l][i + 8];
            s3 += part[l][i + 12];
        }
        double acc = (s0 + s1) + (s2 + s3);
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (q == 0 && (tid >> 2) <= Nx) out[l] = acc;
    }
}

// ---------------------------------------------------------------------------
// state initialisation, moments (FP64 output), residual
// ---------------------------------------------------------------------------
template <typename R>
__global__ void broadcast_kernel(R* __restrict__ f, const R* __restrict__ g, long long nvalues, int V) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nvalues;
         i += (long long)gridDim.x * blockDim.x)
        f[i] = g[i % V];
}

// One warp per node, one pass over the node's values: the raw quadrature sums
// n, j, P_xa = sum p_x p_a f, E = sum |p|^2 f and Q = sum p_x |p|^2 f, from which
// (FP64, per node)
//   u = j/n,  T = (E - n|u|^2)/(D n),
//   q_x = (1/2) sum (p_x - u_x)|p - u|^2 f
//       = (1/2) [Q - 2 (u_x P_xx + u_y P_xy + u_z P_xz) - u_x E + 2 n u_x |u|^2].
// Lanes and the warp tree accumulate in the state's precision, compensated for
// FP32 states (sum and error term); the per-node combination is FP64.  With
// 4 | 2Q_x and 2Q_x | 128 the lanes read 4-vectors whose p_x are fixed per
// lane (as in sums_kernel); otherwise a shared table of (p_x, p_y, p_z) per
// velocity (up to kMomentTableMax velocities) or per-value index arithmetic.
template <typename R, typename R4>
__device__ __forceinline__ R4 velocity_of(const R* P, int v, int QX2, int VY) {
    R4 m;
    m.x = P[v % QX2]; m.y = P[QX2 + (v / QX2) % VY]; m.z = P[QX2 + VY + v / (QX2 * VY)]; m.w = R(0);
    return m;
}

constexpr int kMomentTableMax = 1536;

template <typename R, bool kTable>
__global__ void __launch_bounds__(256)
moments_kernel(const GroupDev g, const R* __restrict__ fs, double* n_out, double* u_out,
               double* T_out, double* q_out, int node_base, const long long* __restrict__ gnode) {
    using R4 = typename std::conditional<sizeof(R) == 4, float4, double4>::type;
    extern __shared__ __align__(16) unsigned char mom_smem[];
    R4* sP = reinterpret_cast<R4*>(mom_smem);            // [V]: p_x, p_y, p_z   (kTable)
    R4* sYZ = sP + (kTable ? g.V : 0);                   // [VY VZ]: p_y, p_z, p_y^2 + p_z^2
    const int V = g.V, QX2 = g.QX2, VY = g.VY, VZ = g.VZ;
    const R* P = static_cast<const R*>(g.p);
    const bool vec4 = (QX2 & 3) == 0 && (QX2 & (QX2 - 1)) == 0 && QX2 <= 128;
    if (kTable) {
        for (int v = threadIdx.x; v < V; v += blockDim.x) sP[v] = velocity_of<R, R4>(P, v, QX2, VY);
        for (int k = threadIdx.x; k < VY * VZ; k += blockDim.x) {
            R4 y;
            y.x = P[QX2 + k % VY]; y.y = P[QX2 + VY + k / VY]; y.z = y.x * y.x + y.y * y.y; y.w = R(0);
            sYZ[k] = y;
        }
        __syncthreads();
    }
    // Nodes go to warps in batches of 32: the warp forms the sums of each node
    // of its batch together (butterfly sums leave them in every lane) and lane
    // k keeps node k's; then every lane finishes its own node in FP64 (on full
    // warps: a lone lane's FP64 instruction costs a whole warp's) and the
    // outputs are written coalesced.
    const int warps = (blockDim.x >> 5) * gridDim.x;
    const int lane = threadIdx.x & 31;
    // 4-vector path with 2Q_x <= 32 (FP64; FP32 states go to moments_rows_kernel):
    // eight lanes per node, four nodes of the batch at a time; each lane's p_x
    // stay fixed (its 4-vectors are 8 apart).
    const bool quad = kTable && sizeof(R) == 8 && vec4 && QX2 <= 32;
    for (int base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < g.nnodes; base += warps * 32) {
        const int nb = min(32, g.nnodes - base);
        R mine[9], mine_c[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) mine[k] = mine_c[k] = R(0);
        if (quad) {
            const int sl = lane & 7, lg = __ffs(QX2) - 1;
            const int x0 = (4 * sl) & (QX2 - 1);
            R px[4], px2[4], px3[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                px[e] = P[x0 + e]; px2[e] = px[e] * px[e]; px3[e] = px2[e] * px[e];
            }
            for (int b = 0; 4 * b < nb; ++b) {
                const int node = base + 4 * b + (lane >> 3);
                // n, j_x, j_y, j_z, P_xx, E - P_xx, P_xy, P_xz, Q
                R a[9] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
                R c[9] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
                if (node < base + nb) {
                    const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
                    const InstDev& I = g.inst[ii];
                    const R4* f4 = reinterpret_cast<const R4*>(fs + (size_t)I.f_off + (size_t)(node - I.node_off) * V);
#pragma unroll 4
                    for (int k = sl; k < (V >> 2); k += 8) {
                        const R4 x = f4[k];
                        const R4 yz = sYZ[k >> (lg - 2)];
                        const R sm = (x.x + x.y) + (x.z + x.w);
                        const R jx = px[0] * x.x + px[1] * x.y + px[2] * x.z + px[3] * x.w;
                        const R pxx = px2[0] * x.x + px2[1] * x.y + px2[2] * x.z + px2[3] * x.w;
                        const R pxxx = px3[0] * x.x + px3[1] * x.y + px3[2] * x.z + px3[3] * x.w;
                        csum_add(a[0], c[0], sm); csum_add(a[1], c[1], jx);
                        csum_add(a[2], c[2], yz.x * sm); csum_add(a[3], c[3], yz.y * sm);
                        csum_add(a[4], c[4], pxx); csum_add(a[5], c[5], yz.z * sm);
                        csum_add(a[6], c[6], yz.x * jx); csum_add(a[7], c[7], yz.y * jx);
                        csum_add(a[8], c[8], pxxx + yz.z * jx);
                    }
                }
                // eight-lane trees; lane L keeps node L's sums (lane 8 (L & 3) of sub-batch L >> 2)
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    csum_warp<R, 4>(a[k], c[k]);
                    const R s2 = __shfl_sync(0xffffffffu, a[k], 8 * (lane & 3));
                    const R c2 = __shfl_sync(0xffffffffu, c[k], 8 * (lane & 3));
                    if ((lane >> 2) == b) { mine[k] = s2; mine_c[k] = c2; }
                }
            }
        }
        for (int kn = 0; kn < (quad ? 0 : nb); ++kn) {
            const int node = base + kn;
            const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
            const InstDev& I = g.inst[ii];
            const R* f = fs + (size_t)I.f_off + (size_t)(node - I.node_off) * V;
            // n, j_x, j_y, j_z, P_xx, E - P_xx, P_xy, P_xz, Q
            // compensated per-lane sums (FP32 states)
            R a[9] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
            R c[9] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
            if (kTable && vec4) {
                const R4* f4 = reinterpret_cast<const R4*>(f);
                const int x0 = (4 * lane) % QX2;
                R px[4], px2[4], px3[4];
    #pragma unroll
                for (int e = 0; e < 4; ++e) {
                    px[e] = P[x0 + e]; px2[e] = px[e] * px[e]; px3[e] = px2[e] * px[e];
                }
    #pragma unroll 4
                for (int k = lane; k < (V >> 2); k += 32) {
                    const R4 x = f4[k];
                    const R4 yz = sYZ[(k << 2) / QX2];
                    const R sm = (x.x + x.y) + (x.z + x.w);
                    const R jx = px[0] * x.x + px[1] * x.y + px[2] * x.z + px[3] * x.w;
                    const R pxx = px2[0] * x.x + px2[1] * x.y + px2[2] * x.z + px2[3] * x.w;
                    const R pxxx = px3[0] * x.x + px3[1] * x.y + px3[2] * x.z + px3[3] * x.w;
                    csum_add(a[0], c[0], sm); csum_add(a[1], c[1], jx);
                    csum_add(a[2], c[2], yz.x * sm); csum_add(a[3], c[3], yz.y * sm);
                    csum_add(a[4], c[4], pxx); csum_add(a[5], c[5], yz.z * sm);
                    csum_add(a[6], c[6], yz.x * jx); csum_add(a[7], c[7], yz.y * jx);
                    csum_add(a[8], c[8], pxxx + yz.z * jx);
                }
            } else {
                for (int v = lane; v < V; v += 32) {
                    const R val = f[v];
                    const R4 p = kTable ? sP[v] : velocity_of<R, R4>(P, v, QX2, VY);
                    const R jx = p.x * val, yz2 = p.y * p.y + p.z * p.z;
                    csum_add(a[0], c[0], val); csum_add(a[1], c[1], jx);
                    csum_add(a[2], c[2], p.y * val); csum_add(a[3], c[3], p.z * val);
                    csum_add(a[4], c[4], p.x * jx); csum_add(a[5], c[5], yz2 * val);
                    csum_add(a[6], c[6], p.y * jx); csum_add(a[7], c[7], p.z * jx);
                    csum_add(a[8], c[8], (p.x * p.x + yz2) * jx);
                }
            }
            // warp sums in the state's precision (FP64 adds run at 1/64 of FP32 here)
    #pragma unroll
            for (int k = 0; k < 9; ++k) {
                csum_warp(a[k], c[k]);
                if (lane == kn) { mine[k] = a[k]; mine_c[k] = c[k]; }
            }
        }
        if (lane < nb) {
            const int node = base + lane;
            double d[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) d[k] = (double)mine[k] + (double)mine_c[k];
            const double n = d[0];
            const double ux = d[1] / n, uy = d[2] / n, uz = d[3] / n;
            const double u2 = ux * ux + uy * uy + uz * uz;
            const double E = d[4] + d[5];
            const double Tn = (E - n * u2) / (g.D * n);
            const double qx = 0.5 * (d[8] - 2.0 * (ux * d[4] + uy * d[6] + uz * d[7]) - ux * E + 2.0 * n * ux * u2);
            long long o = node_base + node;
            if (gnode) {                    // the caller's layout: instance by instance
                const int k = find_slot(g.node_start, g.ninst, node);
                o = gnode[k] + (node - g.node_start[k]);
            }
            if (n_out) n_out[o] = n;
            if (u_out) { u_out[3 * o] = ux; u_out[3 * o + 1] = uy; u_out[3 * o + 2] = uz; }
            if (T_out) T_out[o] = Tn;
            if (q_out) q_out[o] = qx;
            if (!(isfinite(n) && isfinite(Tn))) *g.nonfinite = 1;
        }
    }
}

// The moments of FP32 groups with 2Q_x a power of two up to 32: 32 nodes per CTA
// of 128 threads, the nine sums of a node by eight lanes as in moments_kernel's
// 4-vector path (the same loop, lane by lane: how the compiler joins its packed
// products and sums shows in the last digits of u and q), then one thread per
// node in FP64.  HBM-bound work: what counts is enough loads in flight, so the
// sums of finished nodes wait in shared memory and the kernel stays at 80
// registers, 24 warps per SM (moments_kernel keeps them in registers: 104, 16
// warps of 256-thread CTAs, 30 % of the DRAM rate).  1024 x 512 nodes of 1024
// velocities (GB300): 0.459 ms against 0.771; reading the state alone takes 0.317.
constexpr int kMomNodes = 32, kMomThreads = 128;
__global__ void __launch_bounds__(kMomThreads, 6)
moments_rows_kernel(const GroupDev g, const float* __restrict__ fs, double* n_out, double* u_out, double* T_out,
                    double* q_out, int node_base, const long long* __restrict__ gnode) {
    extern __shared__ __align__(16) unsigned char mom_smem[];
    __shared__ long long sOff[kMomNodes];
    __shared__ float sSum[kMomNodes][21];                // nine sums, nine error terms (padded)
    float4* sYZ = reinterpret_cast<float4*>(mom_smem);   // [VY VZ]: p_y, p_z, p_y^2 + p_z^2
    const int V = g.V, QX2 = g.QX2, VY = g.VY, rows = g.VY * g.VZ;
    const float* P = static_cast<const float*>(g.p);
    const int tid = threadIdx.x, base = blockIdx.x * kMomNodes, nb = min(kMomNodes, g.nnodes - base);
    int ii = 0;
    if (tid < nb) {
        ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, base + tid) : 0;
        sOff[tid] = g.inst[ii].f_off + (long long)(base + tid - g.inst[ii].node_off) * V;
    }
    for (int k = tid; k < rows; k += kMomThreads) {
        float4 y;
        y.x = P[QX2 + k % VY]; y.y = P[QX2 + VY + k / VY]; y.z = y.x * y.x + y.y * y.y; y.w = 0.0f;
        sYZ[k] = y;
    }
    __syncthreads();
    const int lane = tid & 31, sl = lane & 7, lg = __ffs(QX2) - 1;
    const int x0 = (4 * sl) & (QX2 - 1);
    float px[4], px2[4], px3[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        px[e] = P[x0 + e]; px2[e] = px[e] * px[e]; px3[e] = px2[e] * px[e];
    }
    for (int kn = tid >> 3; (kn & ~3) < nb; kn += kMomThreads / 8) {
        float2 s2[5], c2[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) s2[q] = c2[q] = make_float2(0.0f, 0.0f);
        if (kn < nb) {
            const float4* f4 = reinterpret_cast<const float4*>(fs + sOff[kn]);
            float2 pjx[4], p13[4];                   // (p_x, p_x^2), (1, p_x^3) per element
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                pjx[e] = make_float2((float)px[e], (float)px2[e]);
                p13[e] = make_float2(1.0f, (float)px3[e]);
            }
#pragma unroll 4
            for (int k = sl; k < (V >> 2); k += 8) {
                const float4 x = __ldcs(f4 + k);
                const float4 yz = sYZ[k >> (lg - 2)];
                const float xe[4] = {x.x, x.y, x.z, x.w};
                float2 jp = make_float2(0.0f, 0.0f), sq = make_float2(0.0f, 0.0f);   // (j_x, P_xx), (n, Q_x)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    jp = __ffma2_rn(pjx[e], f2(xe[e]), jp);
                    sq = __ffma2_rn(p13[e], f2(xe[e]), sq);
                }
                const float2 yzv = make_float2(yz.x, yz.y);
                csum_add2(s2[0], c2[0], make_float2(sq.x, jp.x));
                csum_add2(s2[1], c2[1], __fmul2_rn(yzv, f2(sq.x)));
                csum_add2(s2[2], c2[2], make_float2(jp.y, yz.z * sq.x));
                csum_add2(s2[3], c2[3], __fmul2_rn(yzv, f2(jp.x)));
                csum_add2(s2[4], c2[4], make_float2(fmaf(yz.z, jp.x, sq.y), 0.0f));
            }
        }
        float a[9], c[9];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            a[2 * q] = s2[q].x; c[2 * q] = c2[q].x;
            if (q < 4) { a[2 * q + 1] = s2[q].y; c[2 * q + 1] = c2[q].y; }
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            csum_warp<float, 4>(a[k], c[k]);
            if (sl == 0 && kn < nb) {
                sSum[kn][k] = a[k];
                sSum[kn][10 + k] = c[k];
            }
        }
    }
    __syncthreads();
    if (tid < nb) {
        const int node = base + tid;
        double d[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) d[k] = (double)sSum[tid][k] + (double)sSum[tid][10 + k];
        const double n = d[0];
        const double ux = d[1] / n, uy = d[2] / n, uz = d[3] / n;
        const double u2 = ux * ux + uy * uy + uz * uz;
        const double E = d[4] + d[5];
        const double Tn = (E - n * u2) / (g.D * n);
        const double qx = 0.5 * (d[8] - 2.0 * (ux * d[4] + uy * d[6] + uz * d[7]) - ux * E + 2.0 * n * ux * u2);
        const long long o = gnode ? gnode[ii] + (node - g.node_start[ii]) : (long long)node_base + node;
        if (n_out) n_out[o] = n;
        if (u_out) { u_out[3 * o] = ux; u_out[3 * o + 1] = uy; u_out[3 * o + 2] = uz; }
        if (T_out) T_out[o] = Tn;
        if (q_out) q_out[o] = qx;
        if (!(isfinite(n) && isfinite(Tn))) *g.nonfinite = 1;
    }
}

__device__ __forceinline__ void atomic_max_nonneg(double* addr, double v) {
    atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

// Per instance: max |a - b| and max |b| (non-negative doubles order like their bits).
template <typename R>
__global__ void residual_kernel(const GroupDev g, const R* __restrict__ a, const R* __restrict__ b,
                                double* out /* [ninst][2] */) {
    const int warps = (blockDim.x >> 5) * gridDim.x;
    const int lane = threadIdx.x & 31;
    for (int node = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); node < g.nnodes; node += warps) {
        const int ii = g.ninst > 1 ? find_slot(g.node_start, g.ninst, node) : 0;
        const InstDev I = g.inst[ii];
        const size_t off = (size_t)I.f_off + (size_t)(node - I.node_off) * g.V;
        double md = 0.0, mb = 0.0;
        for (int v = lane; v < g.V; v += 32) {
            const double bv = b[off + v];
            md = fmax(md, fabs(bv - (double)a[off + v]));
            mb = fmax(mb, fabs(bv));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            md = fmax(md, __shfl_xor_sync(0xffffffffu, md, o));
            mb = fmax(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        }
        if (lane == 0) {
            atomic_max_nonneg(out + 2 * ii, md);
            atomic_max_nonneg(out + 2 * ii + 1, mb);
        }
    }
}

// ---------------------------------------------------------------------------
// host-side launchers (non-template entry points used by hlb_api.cu)
// ---------------------------------------------------------------------------
size_t stage_smem_bytes(const GroupDev& g, int precision, int block) {
    return precision == HLB_FP64_ ? smem_layout<double>(g, block / 32).bytes
                                  : smem_layout<float>(g, block / 32).bytes;
}

template <typename R, int ADV>
static cudaError_t set_attr(size_t smem) {
    return cudaFuncSetAttribute(stage_kernel<R, ADV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

cudaError_t prepare_stage(int precision, int adv, size_t smem) {
    if (precision == HLB_FP64_) return adv == HLB_WENO5_ ? set_attr<double, HLB_WENO5_>(smem) : set_attr<double, HLB_UPWIND2_>(smem);
    return adv == HLB_WENO5_ ? set_attr<float, HLB_WENO5_>(smem) : set_attr<float, HLB_UPWIND2_>(smem);
}

cudaError_t stage_occupancy(int precision, int adv, int block, size_t smem, int* blocks_per_sm) {
    const void* fn;
    if (precision == HLB_FP64_) fn = adv == HLB_WENO5_ ? (const void*)stage_kernel<double, HLB_WENO5_> : (const void*)stage_kernel<double, HLB_UPWIND2_>;
    else fn = adv == HLB_WENO5_ ? (const void*)stage_kernel<float, HLB_WENO5_> : (const void*)stage_kernel<float, HLB_UPWIND2_>;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, block, smem);
}

void launch_stage(int precision, int adv, const GroupDev& g, const void* fs, const void* fn, void* fo,
                  int stage, int grid, int block, size_t smem, cudaStream_t st) {
    if (precision == HLB_FP64_) {
        if (adv == HLB_WENO5_) stage_kernel<double, HLB_WENO5_><<<grid, block, smem, st>>>(g, (const double*)fs, (const double*)fn, (double*)fo, stage);
        else stage_kernel<double, HLB_UPWIND2_><<<grid, block, smem, st>>>(g, (const double*)fs, (const double*)fn, (double*)fo, stage);
    } else {
        if (adv == HLB_WENO5_) stage_kernel<float, HLB_WENO5_><<<grid, block, smem, st>>>(g, (const float*)fs, (const float*)fn, (float*)fo, stage);
        else stage_kernel<float, HLB_UPWIND2_><<<grid, block, smem, st>>>(g, (const float*)fs, (const float*)fn, (float*)fo, stage);
    }
}

template <int ADV>
static void stage_wide_launch(const GroupDev& g, const double* fs, const double* fn, double* fo, int stage, cudaStream_t st) {
    const long long pairs = (long long)g.npairs * g.V, cells = (long long)g.nnodes * g.V;
    // Two cells per thread once their CTAs give every SM two (each quarter a
    // warp); below, one.  us per step, one cell against two (GB300): 72 cells of 400
    // velocities 209 / 228, 144 279 / 275, 288 479 / 437, 576 930 / 898.
    if (pairs <= 2LL * sm_count() * kWideThreads) {
        const int grid = (int)((cells + kWideThreads - 1) / kWideThreads);
        stage_wide_kernel<ADV, 1><<<grid, kWideThreads, (2 * (size_t)g.QX2 + 4) * sizeof(CellVals<1>), st>>>(g, fs, fn, fo, stage);
    } else {
        const int grid = (int)((pairs + kWideThreads - 1) / kWideThreads);
        stage_wide_kernel<ADV, 2><<<grid, kWideThreads, (2 * (size_t)g.QX2 + 4) * sizeof(CellVals<2>), st>>>(g, fs, fn, fo, stage);
    }
}

void launch_stage_wide(int adv, const GroupDev& g, const void* fs, const void* fn, void* fo, int stage, cudaStream_t st) {
    if (adv == HLB_WENO5_) stage_wide_launch<HLB_WENO5_>(g, (const double*)fs, (const double*)fn, (double*)fo, stage, st);
    else stage_wide_launch<HLB_UPWIND2_>(g, (const double*)fs, (const double*)fn, (double*)fo, stage, st);
}

void launch_quad_coef(const GroupDev& g, const void* fs, cudaStream_t st) {
    if (g.Nx < 24) quad_coef_kernel<24><<<2 * g.nnodes, kQuadThreads, 0, st>>>(g, (const double*)fs);
    else quad_coef_kernel<32><<<2 * g.nnodes, kQuadThreads, 0, st>>>(g, (const double*)fs);
}

void launch_wall(int precision, int adv, const GroupDev& g, const void* fs, cudaStream_t st) {
    const int block = 128;
    if (precision == HLB_FP64_) {
        if (adv == HLB_WENO5_) wall_kernel<double, HLB_WENO5_><<<g.nrows * g.wchunks, block, 0, st>>>(g, (const double*)fs);
        else wall_kernel<double, HLB_UPWIND2_><<<g.nrows * g.wchunks, block, 0, st>>>(g, (const double*)fs);
    } else {
        if (adv == HLB_WENO5_) wall_kernel<float, HLB_WENO5_><<<g.nrows * g.wchunks, block, 0, st>>>(g, (const float*)fs);
        else wall_kernel<float, HLB_UPWIND2_><<<g.nrows * g.wchunks, block, 0, st>>>(g, (const float*)fs);
    }
}

void launch_broadcast(int precision, void* f, const void* gvec, long long nvalues, int V, cudaStream_t st) {
    const int block = 256;
    long long blocks = (nvalues + block - 1) / block;
    const int grid = (int)(blocks < 65535LL * 16 ? blocks : 65535LL * 16);
    if (precision == HLB_FP64_) broadcast_kernel<double><<<grid, block, 0, st>>>((double*)f, (const double*)gvec, nvalues, V);
    else broadcast_kernel<float><<<grid, block, 0, st>>>((float*)f, (const float*)gvec, nvalues, V);
}

void launch_moments(int precision, const GroupDev& g, const void* fs, double* n, double* u, double* T,
                    double* q, int node_base, cudaStream_t st, const long long* gnode) {
    const int block = 256;                               // 8 warps, 32 nodes per warp and batch
    const int grid = (g.nnodes + 255) / 256 < 152 * 8 ? (g.nnodes + 255) / 256 : 152 * 8;
    const bool table = g.V + g.VY * g.VZ <= kMomentTableMax;
    if (precision != HLB_FP64_ && table && (g.QX2 & 3) == 0 && (g.QX2 & (g.QX2 - 1)) == 0 && g.QX2 <= 32) {
        moments_rows_kernel<<<(g.nnodes + kMomNodes - 1) / kMomNodes, kMomThreads, g.VY * g.VZ * sizeof(float4), st>>>(
            g, (const float*)fs, n, u, T, q, node_base, gnode);
        return;
    }
    if (precision == HLB_FP64_) {
        if (table) moments_kernel<double, true><<<grid, block, (g.V + g.VY * g.VZ) * sizeof(double4), st>>>(g, (const double*)fs, n, u, T, q, node_base, gnode);
        else moments_kernel<double, false><<<grid, block, 0, st>>>(g, (const double*)fs, n, u, T, q, node_base, gnode);
    } else {
        if (table) moments_kernel<float, true><<<grid, block, (g.V + g.VY * g.VZ) * sizeof(float4), st>>>(g, (const float*)fs, n, u, T, q, node_base, gnode);
        else moments_kernel<float, false><<<grid, block, 0, st>>>(g, (const float*)fs, n, u, T, q, node_base, gnode);
    }
}

void launch_residual(int precision, const GroupDev& g, const void* a, const void* b, double* out, cudaStream_t st) {
    const int block = 256;
    const int grid = (g.nnodes + 7) / 8 < 4096 ? (g.nnodes + 7) / 8 : 4096;
    if (precision == HLB_FP64_) residual_kernel<double><<<grid, block, 0, st>>>(g, (const double*)a, (const double*)b, out);
    else residual_kernel<float><<<grid, block, 0, st>>>(g, (const float*)a, (const float*)b, out);
}

}  // namespace hlb

// ---------------------------------------------------------------------------
// FP32 FMA throughput of the device (the ALU roof of the FP32 stage kernels):
// every thread runs kFmaChains independent chains of dependent FMAs (scalar
// fmaf, or packed f32x2 __ffma2_rn counting two FMAs each), enough warps per SM
// to cover the pipeline latency; the result is written so that no chain is
// dropped.
// ---------------------------------------------------------------------------
namespace hlb {
namespace {
constexpr int kFmaChains = 8, kFmaIters = 4096;

__global__ void __launch_bounds__(256) fma_peak_kernel(float* out, float a, float b) {
    float x[kFmaChains];
#pragma unroll
    for (int c = 0; c < kFmaChains; ++c) x[c] = threadIdx.x * 1e-7f + c;
#pragma unroll 16
    for (int i = 0; i < kFmaIters; ++i)
#pragma unroll
        for (int c = 0; c < kFmaChains; ++c) x[c] = fmaf(x[c], a, b);
    float s = 0.0f;
#pragma unroll
    for (int c = 0; c < kFmaChains; ++c) s += x[c];
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

__global__ void __launch_bounds__(256) fma2_peak_kernel(float* out, float a, float b) {
    float2 x[kFmaChains / 2];
#pragma unroll
    for (int c = 0; c < kFmaChains / 2; ++c) x[c] = make_float2(threadIdx.x * 1e-7f + c, c + 0.5f);
    const float2 a2 = make_float2(a, a), b2 = make_float2(b, b);
#pragma unroll 16
    for (int i = 0; i < kFmaIters; ++i)
#pragma unroll
        for (int c = 0; c < kFmaChains / 2; ++c) x[c] = __ffma2_rn(x[c], a2, b2);
    float s = 0.0f;
#pragma unroll
    for (int c = 0; c < kFmaChains / 2; ++c) s += x[c].x + x[c].y;
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}
}  // namespace

cudaError_t measure_fp32_peak(int packed, double* tflops) {
    int dev = 0, nsm = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int block = 256, grid = nsm * 8;          // 64 warps per SM
    float* out = nullptr;
    e = cudaMalloc(&out, (size_t)grid * block * sizeof(float));
    if (e != cudaSuccess) return e;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 0.0f;
    for (int rep = 0; rep < 4; ++rep) {             // the first launch is a warm-up
        cudaEventRecord(e0);
        if (packed) fma2_peak_kernel<<<grid, block>>>(out, 0.999f, 1e-3f);
        else fma_peak_kernel<<<grid, block>>>(out, 0.999f, 1e-3f);
        cudaEventRecord(e1);
        e = cudaEventSynchronize(e1);
        if (e != cudaSuccess) break;
        float ms = 0.0f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (rep > 0 && (best == 0.0f || ms < best)) best = ms;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(out);
    if (e != cudaSuccess) return e;
    const double flops = 2.0 * kFmaChains * (double)kFmaIters * grid * block;
    *tflops = flops / (best * 1e-3) / 1e12;
    return cudaSuccess;
}
}  // namespace hlb
