// The walls of one (instance, y) row (sm_103a): the emitted densities of both
// walls from the incident fluxes (Sec. IV.C.3, Eq. "eq:nplus_def").  One CTA's
// work, run by the wall kernel (hlb_kernels.cu) and by the one-launch node pass
// (hlb_node.cu).
#pragma once

#include <cuda_runtime.h>

#include "hlb_device.cuh"
#include "hlb_internal.h"

namespace hlb {

// Block `block` of g.nrows g.wchunks; red: shared memory for two doubles per warp.
template <typename R, int ADV>
__device__ __forceinline__ void wall_block(const GroupDev& g, const R* fs, int block, double* red) {
    const int nw = (blockDim.x + 31) >> 5;
    const int row = block / g.wchunks, chunk = block - row * g.wchunks;
    if (row >= g.nrows) return;
    const int ii = g.ninst > 1 ? find_slot(g.row_start, g.ninst, row) : 0;
    const InstDev I = g.inst[ii];
    const int y = row - I.row_off;
    const int nx = I.nx, V = g.V, QX2 = g.QX2;
    const R* frow = fs + (size_t)I.f_off + (size_t)y * nx * V;
    double accL = 0.0, accR = 0.0;
    const int Vc = (V + g.wchunks - 1) / g.wchunks, v0 = chunk * Vc, v1 = min(V, v0 + Vc);
    for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
        const int ix = v % QX2;
        const double px = g.pd[ix];
        const size_t a = px < 0 ? 0 : (size_t)(nx - 1) * V, step = px < 0 ? (size_t)V : (size_t)0 - (size_t)V;
        // incident on the left wall (face -1/2) or on the right one (face nx-1/2):
        // f0 the wall cell, f1 and f2 the next two inward
        double F;
        if constexpr (sizeof(R) == 4) {
            // the stage kernels' FP32 face: stencil scaled by 1/w, ghosts
            // extrapolated from the scaled values
            const float sv = static_cast<const float*>(g.wscale)[v];
            const float f0 = frow[a + v] * sv, f1 = frow[a + step + v] * sv, f2 = frow[a + 2 * step + v] * sv;
            float face;
            if (ADV == HLB_WENO5_) {
                face = weno5_scaled(f2, f1, f0, wall_ghost1(f0, f1, f2), wall_ghost2(f0, f1, f2));
            } else {
                face = upwind2_face<float>(f1, f0);
            }
            F = (double)(((float)px * (1.0f / sv)) * face);
        } else {
            const double f0 = frow[a + v], f1 = frow[a + step + v], f2 = frow[a + 2 * step + v];
            if (ADV == HLB_WENO5_) {
                const double d = 3.0 * f0 - 3.0 * f1 + f2, e = 6.0 * f0 - 8.0 * f1 + 3.0 * f2;
                F = px * weno5_face<double>(f2, f1, f0, d, e);
            } else {
                F = px * upwind2_face<double>(f1, f0);
            }
        }
        if (px < 0) accL += F; else accR += F;
    }
    accL = warp_sum(accL);
    accR = warp_sum(accR);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { red[warp] = accL; red[nw + warp] = accR; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sl = 0.0, sr = 0.0;
        for (int w = 0; w < nw; ++w) { sl += red[w]; sr += red[nw + w]; }
        if (g.wchunks > 1) {
            // this chunk's partial sums; the row's last CTA adds them in chunk
            // order (the same result whatever order the CTAs finish in)
            double* part = g.wpart + (size_t)row * g.wchunks * 2;
            part[2 * chunk] = sl;
            part[2 * chunk + 1] = sr;
            __threadfence();
            if (atomicAdd(g.wcount + row, 1u) != (unsigned)(g.wchunks - 1)) return;
            __threadfence();
            sl = sr = 0.0;
            for (int c = 0; c < g.wchunks; ++c) {
                sl += __ldcg(part + 2 * c);
                sr += __ldcg(part + 2 * c + 1);
            }
            atomicExch(g.wcount + row, 0u);
        }
        g.nw[(size_t)row * 2 + 0] = -sl / I.den_left;
        g.nw[(size_t)row * 2 + 1] = -sr / I.den_right;
    }
}

}  // namespace hlb
