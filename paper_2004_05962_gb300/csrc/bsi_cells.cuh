// bsi_cells.cuh -- Eq. 1 and its transpose on x-cells of any width (see CellPlan
// in bsi_geometry.h): non-integer spacing num/den with lattice shift off/den,
// and integer x-spacings above kMaxSpecializedDx (den = 1).
//
// The weights of a lane's voxels are the same in every row of its strip, so
// they live in registers (run x 4, computed when a warp's strip changes); the y
// and z weights of a unit's rows and planes are computed once per unit, one row
// per lane, into shared memory.  Rows move between HBM and shared memory in
// blocks of rb rows: lane r handles row r's bulk copy, so the address
// arithmetic of a block's copies, the fence, the barrier and the wait are paid
// once per block and not once per row.  Rows may start on any 4-byte boundary:
// a staged row keeps its address modulo 16.
#pragma once

#include "bsi_kernels.cuh"
#include "bsi_launch.h"

namespace bsi {

// The four cubic B-spline weights at offset u (FP32, Horner with FMAs).
__device__ __forceinline__ void bspline4(float u, float B[4]) {
    const float s = 1.f - u;
    const float u2 = u * u;
    constexpr float k6 = 1.f / 6.f;
    B[0] = s * s * s * k6;
    B[1] = fmaf(fmaf(3.f, u, -6.f), u2, 4.f) * k6;
    B[2] = fmaf(fmaf(fmaf(-3.f, u, 3.f), u, 3.f), u, 1.f) * k6;
    B[3] = u2 * u * k6;
}

// The four weights of voxel x of cell f on one axis.  Integer spacing (den = 1)
// reads the table (FP64, rounded once).
__device__ __forceinline__ void cell_weights(int x, int f, int num, int den, int off, float B[4]) {
    const int r = x * den + off - f * num;
    if (den == 1) {
        const int o = weight_base(num) + 4 * r;
#pragma unroll
        for (int l = 0; l < 4; ++l) B[l] = c_lut.w[o + l];
    } else {
        bspline4(__fdiv_rn((float)r, (float)num), B);
    }
}

// The y weights of a unit's rows and the z weights of its planes, one per lane.
// (The caller has a warp barrier before: the previous unit's are read.)
__device__ __forceinline__ void unit_weights(const RatDesc& d, const CellPlan& c, const CellUnit& u, float4* yw,
                                             float4* zw, int lane, unsigned* err) {
    BSI_GUARD(u.y1 - u.y0 <= c.ymax && u.z1 - u.z0 <= c.zmax, kErrStage, err) {
        for (int i = lane; i < u.y1 - u.y0; i += kLanes) {
            float B[4];
            cell_weights(u.y0 + i, u.jy, d.num[1], d.den[1], d.off[1], B);
            yw[i] = make_float4(B[0], B[1], B[2], B[3]);
        }
        for (int i = lane; i < u.z1 - u.z0; i += kLanes) {
            const int z = u.z0 + i;
            const int kz = (int)(((long long)z * d.den[2] + d.off[2]) / d.num[2]);
            float B[4];
            cell_weights(z, kz, d.num[2], d.den[2], d.off[2], B);
            zw[i] = make_float4(B[0], B[1], B[2], B[3]);
        }
    }
    __syncwarp();
}

// The x weights of voxel i of a lane's run: zeros past its end.
__device__ __forceinline__ void run_weights(const RatDesc& d, const CellRun& r, int i, float (&B)[4]) {
    B[0] = B[1] = B[2] = B[3] = 0.f;
    if (i < r.cnt) cell_weights(r.xa + i, r.col, d.num[0], d.den[0], d.off[0], B);
}

// Packed FP32x2 arithmetic (sm_100-class GPUs).  These kernels keep their
// weights in registers, where a packed operand is two neighbouring registers:
// the pairs run along taps, rows or voxels, whose weights differ and lie side
// by side, and the one value they share is doubled.
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// Byte offset, from the lane's run in a staged row, of voxel i of the run, when
// it may be missing: regular strips hold runs of RUN - 1 or RUN voxels, so that
// only the last voxel needs a look (its own address `last`: the spare run when
// missing); in the irregular ones (cells cut by the volume's ends) every voxel
// does.
template <int RUN, bool IRR>
__device__ __forceinline__ uint32_t run_addr(int i, uint32_t sv, uint32_t last, uint32_t spare, int cnt) {
    if (IRR) return i < cnt ? sv + 12u * i : spare;
    return i < RUN - 1 ? sv + 12u * i : last;
}

}  // namespace bsi
