// bsi_cells_forward.cu -- Eq. 1 on x-cells of any width (see bsi_cells.cuh).
//
// Bound by its rows' instructions and HBM writes (512 x 512 x 300 at spacing 4.7:
// 0.158 ms, 5.97 TB/s; 0.204 ms with the weights in shared memory and a copy per
// row).  12 warps of 168 registers and blocks of whole y-cells beat 16 of 128
// with shorter blocks (0.165 against 0.184 ms); pairing voxels instead of
// channels in the packed x-stage was slower (0.189 ms).
#include "bsi_cells.cuh"

namespace bsi {

static __device__ unsigned g_err;

// x-stage of a lane's run into one staged row: voxel i = sum_l W_l(i) p_l, the
// weights doubled for channels 0 and 1 (combine4's packed form).  VEC: the run
// is 4 voxels on a 16-byte boundary.
template <int RUN, bool IRR, bool VEC>
__device__ __forceinline__ void emit_run(const float2 (&W)[RUN][4], const float (&p0)[3], const float (&p1)[3],
                                         const float (&p2)[3], const float (&p3)[3], uint32_t sv, uint32_t last,
                                         uint32_t spare, int cnt) {
    float v[VEC ? 3 * RUN : 3];
#pragma unroll
    for (int i = 0; i < RUN; ++i) {
        float2 t = __fmul2_rn(W[i][0], make_float2(p0[0], p0[1]));
        t = __ffma2_rn(W[i][1], make_float2(p1[0], p1[1]), t);
        t = __ffma2_rn(W[i][2], make_float2(p2[0], p2[1]), t);
        t = __ffma2_rn(W[i][3], make_float2(p3[0], p3[1]), t);
        const float t2 = fmaf(W[i][3].x, p3[2], fmaf(W[i][2].x, p2[2], fmaf(W[i][1].x, p1[2], W[i][0].x * p0[2])));
        if (VEC) {
            v[3 * i] = t.x;
            v[3 * i + 1] = t.y;
            v[3 * i + 2] = t2;
        } else {
            const uint32_t a = run_addr<RUN, IRR>(i, sv, last, spare, cnt);
            sts_f32(a, t.x);
            sts_f32(a + 4, t.y);
            sts_f32(a + 8, t2);
        }
    }
    if (VEC) {
#pragma unroll
        for (int i = 0; i < (VEC ? 3 * RUN / 4 : 0); ++i)
            sts_v4_f32(sv + 16 * i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
}

constexpr int kCellFwdWarps = 4;   // per CTA, three CTAs per SM

// YSPLIT: units may be parts of y-cells (small volumes; finding one costs 0.5% of 512 x
// 512 x 300 at spacing 4.7, whose units are whole y-cells).
template <int RUN, bool WIDE, bool VEC, bool YSPLIT>
__global__ void __launch_bounds__(kCellFwdWarps * kLanes, 3)
    bsi_cells_forward_kernel(const __grid_constant__ RatDesc d, const __grid_constant__ CellPlan c) {
    extern __shared__ __align__(128) unsigned char csmem[];
    const int lane = threadIdx.x & (kLanes - 1);
    const int warp = threadIdx.x >> 5;
    const int wpc = blockDim.x >> 5;
    unsigned char* wsm = csmem + (size_t)warp * c.warp_bytes;
    float4* yw = reinterpret_cast<float4*>(wsm + kCellWeightOff);
    float4* zw = yw + c.ymax;
    unsigned char* ring = wsm + c.head_bytes;
    const uint32_t spare = smem_u32(wsm + kCellSpareOff);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the previous kernel's writes are visible
    const uintptr_t row_pitch = (uintptr_t)12 * d.X, plane_pitch = row_pitch * d.Y;
    const uintptr_t fbase = reinterpret_cast<uintptr_t>(d.field);
    const int lc = WIDE ? lane / c.parts : lane;   // this lane's cell in the strip
    int lxs = -1;
    CellStrip st = {};
    CellRun run = {};
    bool irr = false;
    float2 W[RUN][4];   // each weight twice
    int buf = 0;
    for (long long un = (long long)blockIdx.x * wpc + warp; un < c.units; un += (long long)gridDim.x * wpc) {
        const CellUnit u = cell_unit<YSPLIT>(d, c, un);
        __syncwarp();   // the previous unit's weights are read
        unit_weights(d, c, u, yw, zw, lane, &g_err);
        if (u.xs != lxs) {   // warp-uniform: this warp's strip changed
            lxs = u.xs;
            st = cell_strip(d, c, u.xs);
            run = cell_run(d, c, st, lane);
#pragma unroll
            for (int i = 0; i < RUN; ++i) {
                float B[4];
                run_weights(d, run, i, B);
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    W[i][l] = dup2(B[l]);
                    asm volatile("" : "+f"(W[i][l].y));   // a register of its own: a packed operand without a move per use
                }
            }
            irr = __any_sync(kFull, run.cnt > 0 && run.cnt < RUN - 1);
        }
        // this lane's grid column
        const int col = st.c0 + lane;
        float ph[4][4][3];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const long long e0 = (((long long)(u.kz0 + n) * d.ny + u.jy) * d.nx + col) * 3;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const long long e = e0 + m * 3LL * d.nx;
                ph[n][m][0] = ph[n][m][1] = ph[n][m][2] = 0.f;
                if (lane < st.cells + kHalo) {
                    BSI_GUARD(e >= 0 && e + 3 <= 3LL * d.nx * d.ny * d.nz, kErrPhiRead, &g_err) {
                        const float* p = d.phi + e;
                        ph[n][m][0] = __ldg(p);
                        ph[n][m][1] = __ldg(p + 1);
                        ph[n][m][2] = __ldg(p + 2);
                    }
                }
            }
        }
        const int nbytes = 12 * (st.sx1 - st.sx0);
        const int nyu = u.y1 - u.y0;
        const bool owns = run.cnt > 0, full = run.cnt >= RUN;
        const uint32_t xoff = 12u * (uint32_t)(run.xa - st.sx0);
        const uint32_t stride = owns ? (uint32_t)c.slot : 0u, lstride = full ? (uint32_t)c.slot : 0u;
        BSI_GUARD((int)xoff + 12 * run.cnt + 15 <= c.slot && nbytes + 15 <= c.slot, kErrStage, &g_err) {}
        uintptr_t gz = fbase + 12 * (((uintptr_t)u.z0 * d.Y + u.y0) * d.X + st.sx0);   // row 0 of the plane
        for (int z = u.z0; z < u.z1; ++z, gz += plane_pitch) {
            const float4 wz = zw[z - u.z0];
            float pz[4][3];
#pragma unroll
            for (int m = 0; m < 4; ++m)
                combine4<3, true>(pz[m], wz.x, wz.y, wz.z, wz.w, ph[0][m], ph[1][m], ph[2][m], ph[3][m]);
            for (int r0 = 0; r0 < nyu; r0 += c.rb) {
                const int rows = imin(c.rb, nyu - r0);
                unsigned char* blk = ring + buf * c.stage_bytes;
                buf = buf + 1 == kCellStages ? 0 : buf + 1;
                // (the block is free: each lane waited for its copies of it before the last barrier)
                const uintptr_t g = gz + (uintptr_t)r0 * row_pitch;
                const uint32_t b0 = smem_u32(blk) + xoff;
                uint32_t sv = owns ? b0 : spare;
                uint32_t last = full ? b0 + 12u * (RUN - 1) : spare;
                uint32_t ph16 = (uint32_t)g & 15u;
                for (int r = 0; r < rows; ++r) {
                    const float4 wy = yw[r0 + r];
                    float t[3], p0[3], p1[3], p2[3], p3[3];
                    combine4<3, true>(t, wy.x, wy.y, wy.z, wy.w, pz[0], pz[1], pz[2], pz[3]);
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        if (WIDE) {
                            p0[ch] = __shfl_sync(kFull, t[ch], lc);
                            p1[ch] = __shfl_sync(kFull, t[ch], lc + 1);
                            p2[ch] = __shfl_sync(kFull, t[ch], lc + 2);
                            p3[ch] = __shfl_sync(kFull, t[ch], lc + 3);
                        } else {
                            p0[ch] = t[ch];
                            p1[ch] = __shfl_down_sync(kFull, t[ch], 1);
                            p2[ch] = __shfl_down_sync(kFull, t[ch], 2);
                            p3[ch] = __shfl_down_sync(kFull, t[ch], 3);
                        }
                    }
                    if (VEC) {
                        emit_run<RUN, false, VEC>(W, p0, p1, p2, p3, sv, last, spare, run.cnt);
                    } else {
                        if (irr) emit_run<RUN, true, VEC>(W, p0, p1, p2, p3, sv + ph16, last + ph16, spare, run.cnt);
                        else emit_run<RUN, false, VEC>(W, p0, p1, p2, p3, sv + ph16, last + ph16, spare, run.cnt);
                        last += lstride;
                        ph16 = (ph16 + (uint32_t)row_pitch) & 15u;
                    }
                    sv += stride;
                }
                fence_proxy_async_smem();   // this lane's staging writes before the bulk copies read them
                __syncwarp();
                // lane r hands row r's 16-byte-aligned body to the bulk-copy engine; eight lanes per
                // row store the up to 3 + 3 values around it
                BSI_GUARD(g >= fbase && g + (uintptr_t)(rows - 1) * row_pitch + nbytes <=
                                            fbase + (uintptr_t)(12LL * d.X * d.Y * d.Z), kErrFieldWrite, &g_err) {
                    if (lane < rows) {
                        const uintptr_t gr = g + (uintptr_t)lane * row_pitch;
                        const int shift = (int)(gr & 15), head = imin((16 - shift) & 15, nbytes);
                        const int body = (nbytes - head) & ~15;
                        if (body > 0)
                            bulk_store(reinterpret_cast<void*>(gr + head), blk + lane * c.slot + shift + head, (uint32_t)body);
                    }
                    bulk_commit();
                    // (none where every row starts and ends on a 16-byte boundary; warp-uniform)
                    if ((((uint32_t)g | (uint32_t)row_pitch | (uint32_t)nbytes) & 15u) != 0)
                    for (int r = lane >> 3; r < rows; r += 4) {
                        const uintptr_t gr = g + (uintptr_t)r * row_pitch;
                        const int shift = (int)(gr & 15), head = imin((16 - shift) & 15, nbytes);
                        const int e = lane & 7;
                        const int off = e < 4 ? 4 * e : head + ((nbytes - head) & ~15) + 4 * (e - 4);
                        if (off < (e < 4 ? head : nbytes))
                            *reinterpret_cast<float*>(gr + off) = *reinterpret_cast<const float*>(blk + r * c.slot + shift + off);
                    }
                }
                bulk_wait_read<kCellStages - 1>();   // the block staged next has been read
                __syncwarp();
            }
        }
    }
    // the ring must outlive every bulk copy that reads it
    bulk_wait_all<0>();
    __syncwarp();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // this CTA's rows are written
}

template <int RUN, bool WIDE, bool VEC>
static cudaError_t launch_cells_fwd_t(const RatDesc& d, const CellPlan& c, cudaStream_t s) {
    auto kern = c.ysplit > 1 ? bsi_cells_forward_kernel<RUN, WIDE, VEC, true> : bsi_cells_forward_kernel<RUN, WIDE, VEC, false>;
    const int wpc = imin(kCellFwdWarps, kSmemBudget / c.warp_bytes);
    const int threads = wpc * kLanes, smem = wpc * c.warp_bytes;
    KernelFacts f;
    cudaError_t e = kernel_facts(reinterpret_cast<const void*>(kern), threads, smem, &f);
    if (e != cudaSuccess) return e;
    const long long want = cdiv(c.units, wpc);
    const long long cap = (long long)f.sms * f.ctas_per_sm;
    const int grid = (int)(want < cap ? want : cap);
    if (grid <= 0) return cudaSuccess;
    return launch_pdl(kern, grid, threads, smem, s, d, c);
}

cudaError_t launch_cells_forward(const RatDesc& d, const CellPlan& c, cudaStream_t s) {
    if (c.vec) return launch_cells_fwd_t<4, true, true>(d, c, s);
    if (c.parts == 1) {
        switch (c.run) {
            case 1: return launch_cells_fwd_t<1, false, false>(d, c, s);
            case 2: return launch_cells_fwd_t<2, false, false>(d, c, s);
            case 3: return launch_cells_fwd_t<3, false, false>(d, c, s);
            case 4: return launch_cells_fwd_t<4, false, false>(d, c, s);
            case 5: return launch_cells_fwd_t<5, false, false>(d, c, s);
            case 6: return launch_cells_fwd_t<6, false, false>(d, c, s);
            case 7: return launch_cells_fwd_t<7, false, false>(d, c, s);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (c.run) {   // 8 <= width: runs of 4 to 7
        case 4: return launch_cells_fwd_t<4, true, false>(d, c, s);
        case 5: return launch_cells_fwd_t<5, true, false>(d, c, s);
        case 6: return launch_cells_fwd_t<6, true, false>(d, c, s);
        case 7: return launch_cells_fwd_t<7, true, false>(d, c, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t cells_forward_err_read_clear(unsigned* out, cudaStream_t s) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_err, sizeof(unsigned), 0, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_err);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(p, 0, sizeof(unsigned), s);
}

}  // namespace bsi
