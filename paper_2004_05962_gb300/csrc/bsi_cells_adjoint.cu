// bsi_cells_adjoint.cu -- the transpose of Eq. 1 on x-cells of any width (see
// bsi_cells.cuh): partial sums per unit, then one sum per control point.
//
// Bound by HBM reads on large volumes (512 x 512 x 300 at spacing 4.7: 0.161 ms
// alone for 944 MB, 78% of the DRAM peak, 100 M warp instructions; re-reading
// every voxel's weights from shared memory and copying row by row took 240 M and
// 0.313 ms), by the rows' latency on small ones.  12 warps of 168 registers, which
// hold the rolling z window (48 sums per lane) and the weights; where lanes share
// a cell, whose rows are summed per tap (48 sums more), 16 to 156 bytes per thread
// spill.  Two stages of blocks; three (fewer rows each) measured 0.192 against
// 0.181 ms.
#include "bsi_cells.cuh"

namespace bsi {

static __device__ unsigned g_err;

constexpr int kCellAdjWarps = 4;   // per CTA, three CTAs per SM

// One grid plane of a unit's partial sums; h holds pairs of grid rows.
__device__ __forceinline__ void cell_flush(const CellPlan& c, long long un, int pz, float* part,
                                           const float2 (&h)[2][3], int lane, unsigned* err) {
    if (lane < c.nc) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const long long e = cell_part(c, un, pz, m, lane);
            BSI_GUARD(e >= 0 && e + 3 <= c.part_floats, kErrPartWrite, err) {
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) part[e + ch] = m & 1 ? h[m >> 1][ch].y : h[m >> 1][ch].x;
            }
        }
    }
}

// x-transpose of a lane's run in one staged row: q_l = sum B_l(x) G(x), in order;
// W and q hold pairs of taps.  VEC: the run is 4 voxels on a 16-byte boundary.
template <int RUN, bool IRR, bool VEC>
__device__ __forceinline__ void gather_run(float2 (&q)[2][3], const float2 (&W)[RUN][2], uint32_t sv, uint32_t last,
                                           uint32_t spare, int cnt) {
    float v[VEC ? 3 * RUN : 1];
    if (VEC) {
#pragma unroll
        for (int i = 0; i < (VEC ? 3 * RUN / 4 : 0); ++i)
            lds_v4_f32(sv + 16 * i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
#pragma unroll
    for (int i = 0; i < RUN; ++i) {
        const uint32_t a = run_addr<RUN, IRR>(i, sv, last, spare, cnt);
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            const float2 g = dup2(VEC ? v[VEC ? 3 * i + ch : 0] : lds_f32(a + 4 * ch));
#pragma unroll
            for (int l = 0; l < 2; ++l) q[l][ch] = i == 0 ? __fmul2_rn(W[i][l], g) : __ffma2_rn(W[i][l], g, q[l][ch]);
        }
    }
}

template <int RUN, bool WIDE, bool VEC>
__global__ void __launch_bounds__(kCellAdjWarps * kLanes, 3)
    bsi_cells_adjoint_kernel(const __grid_constant__ RatDesc d, const __grid_constant__ CellPlan c,
                             const float* __restrict__ grad, float* __restrict__ part) {
    extern __shared__ __align__(128) unsigned char csmem[];
    const int lane = threadIdx.x & (kLanes - 1);
    const int warp = threadIdx.x >> 5;
    const int wpc = blockDim.x >> 5;
    unsigned char* wsm = csmem + (size_t)warp * c.warp_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(wsm);
    float4* yw = reinterpret_cast<float4*>(wsm + kCellWeightOff);
    float4* zw = yw + c.ymax;
    unsigned char* ring = wsm + c.head_bytes;
    const uint32_t spare = smem_u32(wsm + kCellSpareOff);
    sts_f32(spare + 4u * lane, 0.f);   // the spare run: zeros, also 12 bytes past it
    if (lane == 0) {
        for (int s = 0; s < kCellStages; ++s) mbar_init(bars + s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the previous kernel's writes are visible
    const uintptr_t gbase = reinterpret_cast<uintptr_t>(grad);
    const uintptr_t A0 = ceil16(gbase);
    const uintptr_t A1 = floor16(gbase + (uintptr_t)(12LL * d.X * d.Y * d.Z));
    const uintptr_t row_pitch = (uintptr_t)12 * d.X, plane_pitch = row_pitch * d.Y;
    const int per = kLanes / c.parts, lp = lane % c.parts;   // cells a warp could hold; this lane's part
    bool ok_all = true;
    int lxs = -1;
    CellStrip st = {};
    CellRun run = {};
    bool irr = false;
    float2 W[RUN][2];
    unsigned q = 0;
    for (long long un = (long long)blockIdx.x * wpc + warp; ok_all && un < c.units; un += (long long)gridDim.x * wpc) {
        const CellUnit u = cell_unit<false>(d, c, un);
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
                W[i][0] = make_float2(B[0], B[1]);
                W[i][1] = make_float2(B[2], B[3]);
            }
            irr = __any_sync(kFull, run.cnt > 0 && run.cnt < RUN - 1);
        }
        const int nbytes = 12 * (st.sx1 - st.sx0);
        const int nyu = u.y1 - u.y0, nblk = (nyu + c.rb - 1) / c.rb;
        const int planes = u.z1 - u.z0, blocks = planes * nblk;
        const uintptr_t g0 = gbase + 12 * (((uintptr_t)u.z0 * d.Y + u.y0) * d.X + st.sx0);
        // only a unit holding the first or last row of the array has bytes outside the bulk copies
        const bool unit_edge =
            g0 < A0 || g0 + (uintptr_t)(planes - 1) * plane_pitch + (uintptr_t)(nyu - 1) * row_pitch + nbytes > A1;
        const unsigned q0 = q;

        // producer (the whole warp): block ik of the unit, rows ii rb .. of plane ip, into
        // stage (q0 + ik) % kCellStages; lane r copies row r
        int ik = 0, ii = 0;
        uintptr_t gp = g0;   // row 0 of that plane
        auto issue = [&]() {
            const unsigned s = (q0 + (unsigned)ik) % kCellStages;
            const int r0 = ii * c.rb, n = imin(c.rb, nyu - r0);
            uint32_t bytes = 0;
            RowLoad L = {};
            if (lane < n) {
                L = row_load(reinterpret_cast<const unsigned char*>(gp + (uintptr_t)(r0 + lane) * row_pitch), nbytes, A0, A1);
                if (L.s1 > L.s0) bytes = (uint32_t)(L.s1 - L.s0);
            }
            const uint32_t total = __reduce_add_sync(kFull, bytes);
            if (lane == 0) {
                if (total > 0) mbar_arrive_expect_tx(bars + s, total);
                else mbar_arrive(bars + s);
            }
            __syncwarp();
            BSI_GUARD((L.s0 - L.lo) + bytes <= (uintptr_t)c.slot && lane < kLanes && n <= c.rb, kErrStage, &g_err) {
                if (bytes > 0)
                    bulk_load(ring + s * c.stage_bytes + lane * c.slot + (L.s0 - L.lo),
                              reinterpret_cast<const void*>(L.s0), bytes, bars + s);
            }
            ++ik;
            if (++ii == nblk) {
                ii = 0;
                gp += plane_pitch;
            }
        };
        while (ik < blocks && ik < kCellStages) issue();

        float2 hz[4][2][3];   // four grid planes x pairs of grid rows
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) hz[n][m][ch] = dup2(0.f);
        const bool owns = run.cnt > 0;
        const uint32_t xoff = 12u * (uint32_t)(run.xa - st.sx0);
        const uint32_t stride = owns ? (uint32_t)c.slot : 0u, lstride = run.cnt >= RUN ? (uint32_t)c.slot : 0u;
        uintptr_t gz = g0;   // consumer: row 0 of the current plane
        int k = 0;
        for (int kz = u.kz0; ok_all && kz < u.kz1; ++kz) {
            const int zb = imax(u.z0, cell_first(kz, d.num[2], d.den[2], d.off[2]));
            const int ze = imin(u.z1, cell_first(kz + 1, d.num[2], d.den[2], d.off[2]));
            for (int z = zb; ok_all && z < ze; ++z, gz += plane_pitch) {
                // narrow cells: hy[row pair], each row's column sums taken at once.  WIDE: the rows
                // are summed per lane and tap (hq[row][tap pair]) and the lanes of a cell
                // combined once per plane, which keeps the shuffles out of the rows.
                float2 hy[2][3], hq[WIDE ? 4 : 1][2][3];
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        hy[m][ch] = dup2(0.f);
#pragma unroll
                        for (int n = 0; n < (WIDE ? 4 : 1); ++n) hq[n][m][ch] = dup2(0.f);
                    }
                for (int i = 0; i < nblk; ++i, ++k) {
                    const unsigned qq = q0 + (unsigned)k, s = qq % kCellStages;
                    if (!mbar_wait_bounded(bars + s, (qq / kCellStages) & 1u)) {
                        // a bulk copy never completed: record it, give the copies still in
                        // flight a bounded chance to land, and stop this warp
                        if (lane == 0) atomicOr(&g_err, kErrTimeout);
                        for (int p = k + 1; p < ik; ++p) {
                            const unsigned qp = q0 + (unsigned)p;
                            (void)mbar_wait_bounded(bars + qp % kCellStages, (qp / kCellStages) & 1u);
                        }
                        ok_all = false;
                        break;
                    }
                    const int r0 = i * c.rb, rows = imin(c.rb, nyu - r0);
                    unsigned char* blk = ring + s * c.stage_bytes;
                    uintptr_t g = gz + (uintptr_t)r0 * row_pitch;
                    if (unit_edge) {   // elements outside the bulk copies: first or last row of the array
                        for (int r = 0; r < rows; ++r) {
                            const uintptr_t gr = g + (uintptr_t)r * row_pitch;
                            if (gr >= A0 && gr + (uintptr_t)nbytes <= A1) continue;
                            const RowLoad L = row_load(reinterpret_cast<const unsigned char*>(gr), nbytes, A0, A1);
                            float* sb = reinterpret_cast<float*>(blk + r * c.slot + (gr & 15));
                            for (int e = lane; e < nbytes / 4; e += kLanes) {
                                const uintptr_t a = gr + 4u * (uintptr_t)e;
                                if (a < L.s0 || a >= L.s1) sb[e] = *reinterpret_cast<const float*>(a);
                            }
                        }
                        __syncwarp();
                    }
                    const uint32_t b0 = smem_u32(blk) + xoff;
                    uint32_t sv = owns ? b0 : spare;
                    uint32_t last = run.cnt >= RUN ? b0 + 12u * (RUN - 1) : spare;
                    uint32_t ph = (uint32_t)g & 15u;
                    BSI_GUARD((int)xoff + 12 * run.cnt + 12 <= c.slot && rows * c.slot <= c.stage_bytes, kErrStage, &g_err) {}
                    for (int r = 0; r < rows; ++r) {
                        float2 q2[2][3];
                        if (VEC) {
                            gather_run<RUN, false, VEC>(q2, W, sv, last, spare, run.cnt);
                        } else {
                            if (irr) gather_run<RUN, true, VEC>(q2, W, sv + ph, last + ph, spare, run.cnt);
                            else gather_run<RUN, false, VEC>(q2, W, sv + ph, last + ph, spare, run.cnt);
                            last += lstride;
                            ph = (ph + (uint32_t)row_pitch) & 15u;
                        }
                        sv += stride;
                        const float4 wy = yw[r0 + r];
                        if (!WIDE) {
                            // column sums: column c0 + lane collects tap l of the cell l below
#pragma unroll
                            for (int ch = 0; ch < 3; ++ch) {
                                const float t1 = __shfl_up_sync(kFull, q2[0][ch].y, 1);
                                const float t2 = __shfl_up_sync(kFull, q2[1][ch].x, 2);
                                const float t3 = __shfl_up_sync(kFull, q2[1][ch].y, 3);
                                const float2 h = dup2(q2[0][ch].x + (lane >= 1 ? t1 : 0.f) + (lane >= 2 ? t2 : 0.f) +
                                                      (lane >= 3 ? t3 : 0.f));
                                hy[0][ch] = __ffma2_rn(make_float2(wy.x, wy.y), h, hy[0][ch]);
                                hy[1][ch] = __ffma2_rn(make_float2(wy.z, wy.w), h, hy[1][ch]);
                            }
                        } else {
                            const float By[4] = {wy.x, wy.y, wy.z, wy.w};
#pragma unroll
                            for (int m = 0; m < (WIDE ? 4 : 0); ++m)
#pragma unroll
                                for (int l = 0; l < 2; ++l)
#pragma unroll
                                    for (int ch = 0; ch < 3; ++ch)
                                        hq[m][l][ch] = __ffma2_rn(dup2(By[m]), q2[l][ch], hq[m][l][ch]);
                        }
                    }
                    // the stage may be refilled once every lane has read it
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (ik < blocks) issue();
                }
                if (!ok_all) break;
                if (WIDE) {
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        // the cell's sums over its parts land on its first lane
                        for (int step = 1; step < c.parts; step <<= 1)
#pragma unroll
                            for (int m = 0; m < (WIDE ? 4 : 0); ++m)
#pragma unroll
                                for (int l = 0; l < 2; ++l) {
                                    const float tx = __shfl_down_sync(kFull, hq[m][l][ch].x, step);
                                    const float ty = __shfl_down_sync(kFull, hq[m][l][ch].y, step);
                                    if (lp + step < c.parts) {
                                        hq[m][l][ch].x += tx;
                                        hq[m][l][ch].y += ty;
                                    }
                                }
                        // column c0 + lane collects tap l of the cell l below
#pragma unroll
                        for (int m = 0; m < (WIDE ? 4 : 0); ++m) {
                            float h = 0.f;
#pragma unroll
                            for (int l = 0; l < 4; ++l) {
                                const bool has = lane >= l && lane - l < per;
                                const float t = __shfl_sync(kFull, l & 1 ? hq[m][l >> 1][ch].y : hq[m][l >> 1][ch].x,
                                                            has ? (lane - l) * c.parts : 0);
                                if (has) h += t;
                            }
                            if (m & 1) hy[m >> 1][ch].y = h;
                            else hy[m >> 1][ch].x = h;
                        }
                    }
                }
                const float4 wz = zw[z - u.z0];
                const float Bz[4] = {wz.x, wz.y, wz.z, wz.w};
#pragma unroll
                for (int n = 0; n < 4; ++n)
#pragma unroll
                    for (int m = 0; m < 2; ++m)
#pragma unroll
                        for (int ch = 0; ch < 3; ++ch) hz[n][m][ch] = __ffma2_rn(dup2(Bz[n]), hy[m][ch], hz[n][m][ch]);
            }
            if (!ok_all) break;
            // grid plane kz is complete for this unit: write it, roll the window by one plane
            cell_flush(c, un, kz - u.kz0, part, hz[0], lane, &g_err);
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) {
#pragma unroll
                    for (int n = 0; n < 3; ++n) hz[n][m][ch] = hz[n + 1][m][ch];
                    hz[3][m][ch] = dup2(0.f);
                }
        }
        q = q0 + (unsigned)blocks;
        if (!ok_all) break;
        // planes kz1 .. kz1 + 2 get contributions from this unit's last cells only
#pragma unroll
        for (int n = 0; n < 3; ++n) cell_flush(c, un, u.kz1 - u.kz0 + n, part, hz[n], lane, &g_err);
    }
    __syncwarp();
    if (lane == 0)
        for (int s = 0; s < kCellStages; ++s) mbar_inval(bars + s);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // this CTA's partial sums are written
}

// One thread per stored control point (gx, gy, gz), a block per run of kReduceX
// points of a grid row (the row is decoded once per block).  The units that
// cover it are the z-units whose planes hold gz, y-cells gy - m (m = 0..3), and
// the strips whose columns [xs sc, xs sc + cells + 3) hold gx; their offsets
// differ by constants of the plan, so one 64-bit offset per point and adds give
// them all, and the 12 loads of a (z-unit, strip) pair are issued together.
// Where z-cells are split (few, large cells: few points, many units each) SLICES
// groups of threads take the z-units in turn and their sums are added in order.
constexpr int kReduceX = 64;

template <int SLICES>
__global__ void __launch_bounds__(kReduceX * SLICES)
    bsi_cells_reduce_kernel(const __grid_constant__ RatDesc d, const __grid_constant__ CellPlan c,
                            const float* __restrict__ part, float* __restrict__ dphi) {
    __shared__ float sum[SLICES > 1 ? SLICES : 1][3][kReduceX];
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the partial sums are visible
    const int nb = (d.nx + kReduceX - 1) / kReduceX;
    const long long blocks = (long long)d.ny * d.nz * nb;
    const int zdiv = c.zsplit > 1 ? c.zsplit : 1;   // z-units per z-chunk
    const int nch = c.zsplit > 1 ? c.ncz : c.nzu;   // z-chunks of zc cells
    const long long uf = cell_part(c, 1, 0, 0, 0);                             // floats of one unit
    const long long sm = (long long)c.nsx * uf - cell_part(c, 0, 0, 1, 0);     // one y-cell less, one row more
    const long long szu = (long long)c.ncy * c.nsx * uf;                       // one z-unit
    for (long long b = blockIdx.x; b < blocks; b += gridDim.x) {
        const long long row = b / nb;
        const int gx = (int)(b - row * nb) * kReduceX + threadIdx.x;
        const int gz = (int)(row / d.ny), gy = (int)(row - (long long)gz * d.ny);
        float s[3] = {0.f, 0.f, 0.f};
        if (gx < d.nx) {
            const int xh = imin(c.nsx - 1, gx / c.sc);
            int k = 0;
            for (int ch = imin(nch - 1, gz / c.zc); ch >= 0; --ch) {
                const int pz = gz - ch * c.zc;                            // plane slot within the chunk
                if (pz >= imin(c.zc, c.ncz - ch * c.zc) + kHalo) break;   // beyond its planes (and every earlier chunk's)
                // tap m = 0, strip xh, first z-unit of the chunk
                const long long e0 = cell_part(c, ((long long)ch * zdiv * c.ncy + gy) * c.nsx + xh, pz, 0, gx - xh * c.sc);
                for (int z = 0; z < zdiv; ++z, ++k) {
                    if (SLICES > 1 && k % SLICES != (int)threadIdx.y) continue;
                    long long ex = e0 + z * szu;
                    for (int xs = xh; xs >= 0; --xs, ex -= uf - 3LL * c.sc) {
                        if (gx - xs * c.sc >= imin(c.sc, c.ncx - xs * c.sc) + kHalo) break;
                        float v[4][3];
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            v[m][0] = v[m][1] = v[m][2] = 0.f;
                            if (gy - m >= 0 && gy - m < c.ncy) {
                                const long long e = ex - m * sm;
                                BSI_GUARD(e >= 0 && e + 3 <= c.part_floats, kErrPartRead, &g_err) {
                                    v[m][0] = __ldcs(part + e);
                                    v[m][1] = __ldcs(part + e + 1);
                                    v[m][2] = __ldcs(part + e + 2);
                                }
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 3; ++i) s[i] += (v[3][i] + v[2][i]) + (v[1][i] + v[0][i]);
                    }
                }
            }
        }
        if (SLICES > 1) {
#pragma unroll
            for (int i = 0; i < 3; ++i) sum[threadIdx.y][i][threadIdx.x] = s[i];
            __syncthreads();
            if (threadIdx.y == 0)
#pragma unroll
                for (int k = 1; k < SLICES; ++k)
#pragma unroll
                    for (int i = 0; i < 3; ++i) s[i] += sum[SLICES > 1 ? k : 0][i][threadIdx.x];
        }
        if (gx < d.nx && threadIdx.y == 0) {
            float* o = dphi + 3 * (row * d.nx + gx);
            o[0] = s[0];
            o[1] = s[1];
            o[2] = s[2];
        }
        if (SLICES > 1) __syncthreads();   // the sums are read before the next block's
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <int SLICES>
static cudaError_t launch_cells_reduce(const RatDesc& d, const CellPlan& c, const float* part, float* dphi,
                                       cudaStream_t s) {
    auto kern = bsi_cells_reduce_kernel<SLICES>;
    KernelFacts f;
    const cudaError_t e = kernel_facts(reinterpret_cast<const void*>(kern), kReduceX * SLICES, 0, &f);
    if (e != cudaSuccess) return e;
    const long long want = (long long)d.ny * d.nz * cdiv(d.nx, kReduceX), cap = (long long)f.sms * f.ctas_per_sm * 64;
    const int grid = (int)(want < cap ? want : cap);
    if (grid <= 0) return cudaSuccess;
    return launch_pdl(kern, dim3((unsigned)grid), dim3(kReduceX, SLICES), 0, s, d, c, part, dphi);
}

template <int RUN, bool WIDE, bool VEC>
static cudaError_t launch_cells_adj_t(const RatDesc& d, const CellPlan& c, const float* grad, float* part,
                                      cudaStream_t s) {
    auto kern = bsi_cells_adjoint_kernel<RUN, WIDE, VEC>;
    const int wpc = imin(kCellAdjWarps, kSmemBudget / c.warp_bytes);
    const int threads = wpc * kLanes, smem = wpc * c.warp_bytes;
    KernelFacts f;
    cudaError_t e = kernel_facts(reinterpret_cast<const void*>(kern), threads, smem, &f);
    if (e != cudaSuccess) return e;
    const long long want = cdiv(c.units, wpc);
    const long long cap = (long long)f.sms * f.ctas_per_sm;
    const int grid = (int)(want < cap ? want : cap);
    if (grid <= 0) return cudaSuccess;
    return launch_pdl(kern, grid, threads, smem, s, d, c, grad, part);
}

static cudaError_t launch_cells_partials(const RatDesc& d, const CellPlan& c, const float* grad, float* part,
                                         cudaStream_t s) {
    if (c.vec) return launch_cells_adj_t<4, true, true>(d, c, grad, part, s);
    if (c.parts == 1) {
        switch (c.run) {
            case 1: return launch_cells_adj_t<1, false, false>(d, c, grad, part, s);
            case 2: return launch_cells_adj_t<2, false, false>(d, c, grad, part, s);
            case 3: return launch_cells_adj_t<3, false, false>(d, c, grad, part, s);
            case 4: return launch_cells_adj_t<4, false, false>(d, c, grad, part, s);
            case 5: return launch_cells_adj_t<5, false, false>(d, c, grad, part, s);
            case 6: return launch_cells_adj_t<6, false, false>(d, c, grad, part, s);
            case 7: return launch_cells_adj_t<7, false, false>(d, c, grad, part, s);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (c.run) {   // 8 <= width: runs of 4 to 7
        case 4: return launch_cells_adj_t<4, true, false>(d, c, grad, part, s);
        case 5: return launch_cells_adj_t<5, true, false>(d, c, grad, part, s);
        case 6: return launch_cells_adj_t<6, true, false>(d, c, grad, part, s);
        case 7: return launch_cells_adj_t<7, true, false>(d, c, grad, part, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_cells_adjoint(const RatDesc& d, const CellPlan& c, const float* grad, float* dphi, float* part,
                                 cudaStream_t s) {
    const cudaError_t e = launch_cells_partials(d, c, grad, part, s);
    if (e != cudaSuccess) return e;
    return c.zsplit > 1 ? launch_cells_reduce<8>(d, c, part, dphi, s) : launch_cells_reduce<1>(d, c, part, dphi, s);
}

cudaError_t cells_adjoint_err_read_clear(unsigned* out, cudaStream_t s) {
    cudaError_t e = cudaMemcpyFromSymbolAsync(out, g_err, sizeof(unsigned), 0, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_err);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(p, 0, sizeof(unsigned), s);
}

}  // namespace bsi
