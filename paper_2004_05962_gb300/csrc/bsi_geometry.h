// bsi_geometry.h -- index arithmetic shared by the kernels and the host.
//
// Every global or shared-memory range a kernel touches is computed by one of
// these functions.  They compile for the device (kernels) and for the host
// (launch set-up and bsi_selfcheck_ranges, which walks every unit of a launch
// on the CPU and checks each range against its buffer before anything runs).
//
// Work decomposition (Sec. 2.1.1: a tile is one control cell of dx*dy*dz
// voxels, and all voxels of a tile share the same 4x4x4 control points):
//  * a warp owns a UNIT: a strip of up to 29 x-neighbouring tiles of one
//    tile-row (jy) and one tile-plane (kz) -- forward -- or of a chunk of
//    tile-planes -- adjoint.  Lane l holds one column of control points, so a
//    warp holds 32 columns and completes 32 - 3 = 29 tiles (forward) or the
//    full sums of 29 columns (adjoint); the 3 extra lanes are the halo of the
//    4-wide neighbourhood.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define BSI_HD __host__ __device__ __forceinline__
#else
#define BSI_HD inline
#endif

namespace bsi {

constexpr int kLanes = 32;
constexpr int kHalo = 3;                       // neighbourhood width 4 = 1 + kHalo
constexpr int kGroupCells = kLanes - kHalo;    // tiles (forward) or columns (adjoint) per warp
constexpr int kMaxSpacing = 64;
constexpr int kMaxSpecializedDx = 8;           // x-spacings with a compile-time inner loop
constexpr int kMaxBatch = 64;                  // instances per launch (kernel parameters)

// One volume as the kernels see it.  Filled on the host from bsi_geom.
struct InstDesc {
    int X, Y, Z;
    int dx, dy, dz;
    int nx, ny, nz;      // stored control grid
    int ncx, ncy, ncz;   // tiles per axis (0 for an empty volume)
    int nxg;             // x-groups: ceil(ncx/29) forward, ceil(nx/29) adjoint
    int nzc;             // adjoint: tile-plane chunks
    int zchunk;          // adjoint: tile-planes per chunk
    int gcells;          // forward: tiles per warp strip (<= 29; see fwd_strip_tiles)
    int zparts;          // forward: units per tile-plane of a strip (see fwd_zparts)
    int warps_req;       // requested warps per CTA from the tile-config table (0: automatic)
    int tma_rows;        // adjoint tensor-copy path: rows per block (tma_block_rows), else 0
    int jrows;           // adjoint: tile-rows per unit (1, or 2 on the tensor-copy path)
    int ncyu;            // adjoint: unit rows, ceil(ncy / jrows)
    int row_block;       // adjoint row-copy path: rows per block (row_block_rows)
    long long units;        // units of this instance
    long long unit_begin;   // first global unit index of this instance in its launch
    long long point_begin;  // adjoint reduce: first global grid point of this instance
    long long part_off;     // adjoint: float offset of this instance's partials in the workspace
    const float* phi;
    void* field;
    const float* grad;
    float* dphi;
    // resampling of a floating image by the field (bsi_resample_*)
    const float* image;     // floating image [fZ][fY][fX]
    const float* gwarp;     // gradient mode: dL/dwarped [Z][Y][X]
    int fX, fY, fZ;
};

template <int MAXB>
struct Batch {
    int n;
    int buf_bytes;          // bytes of one staging row slot (stage_buf_bytes of the largest dx); adjoint: of a ring stage
    int warps_req;          // requested warps per CTA (0: as many as shared memory allows, <= 8)
    int stages;             // adjoint tensor-copy path: ring stages per warp (else 0)
    long long total_units;
    long long total_points;
    InstDesc inst[MAXB];
};

// Index of instance i in a launch's descriptor array: the constant 0 when the
// launch holds one instance (MAXB == 1), so that the descriptor's fields are
// constant-bank operands rather than loads indexed by a register.
template <int MAXB>
BSI_HD int inst_index(int i) { return MAXB == 1 ? 0 : i; }

BSI_HD long long cdiv(long long a, long long b) { return (a + b - 1) / b; }
BSI_HD int imin(int a, int b) { return a < b ? a : b; }
BSI_HD int imax(int a, int b) { return a > b ? a : b; }

// Offset of the 4*d weights of spacing d in the weight table: sum_{e<d} 4e.
BSI_HD constexpr int weight_base(int d) { return 2 * d * (d - 1); }
constexpr int kWeightCount = weight_base(kMaxSpacing + 1);

// Element (float or bf16) offset of voxel (x, y, z) channel 0 in a field.
BSI_HD long long field_elem(const InstDesc& d, int z, int y, int x) {
    return (((long long)z * d.Y + y) * d.X + x) * 3;
}

// Float offset of stored control point (gx, gy, gz) channel 0.
BSI_HD long long phi_elem(const InstDesc& d, int gz, int gy, int gx) {
    return (((long long)gz * d.ny + gy) * d.nx + gx) * 3;
}

// Unit taken by slot (cta, warp) in round r of a persistent launch of `ctas`
// CTAs x `wpc` warps over `total` units, or -1 when the slot has none.  Full
// rounds are CTA-major (the warps of a CTA take neighbouring units, which share
// control points in L1 and, in a batch, a kernel specialisation); the last,
// partial round is dealt warp-major across the CTAs (spread_tail) so that every
// SM gets an even share of it -- worth it for the adjoint's few long units,
// not for the forward's many short ones.
BSI_HD long long slot_unit(long long r, int cta, int warp, int ctas, int wpc, long long total,
                           bool spread_tail = true) {
    const long long W = (long long)ctas * wpc;
    const long long base = r * W;
    if (base >= total) return -1;
    if (total - base >= W || !spread_tail) {
        const long long u = base + (long long)cta * wpc + warp;
        return u < total ? u : -1;
    }
    const long long p = (long long)warp * ctas + cta;
    return p < total - base ? base + p : -1;
}

// ---------------------------------------------------------------- forward

struct FwdUnit {
    int kz, jy, xg;
    int rz0, rz1;   // planes of the tile-plane the unit takes
    int cell0;   // first tile of the strip; lane l holds grid column cell0 + l
    int ncell;   // tiles the warp outputs (<= 29)
    int x0;      // first voxel of the strip
    int nvox;    // voxels per row of the strip
};

// Tiles per forward strip.  When a row of the field is a multiple of 16 bytes
// (X % 4 == 0 for FP32 output, X % 8 == 0 for BF16), a strip of g tiles whose
// byte width 3 g dx ES is a multiple of 16 starts every row segment on a
// 16-byte boundary, so each row leaves as one aligned bulk copy with no
// unaligned head or tail: the largest such g <= 29 (FP32: 28 or 29; BF16 at
// even dx: 28 or 29).  BF16 at odd dx would need g = 24, whose idle lanes cost
// more than the unaligned ends save (512 x 512 x 300 at spacing 5: 0.172 ->
// 0.181 ms): 29, as when rows are unaligned anyway.  (One channel of 4 or 2
// bytes gives the same conditions.)
BSI_HD int fwd_strip_tiles(int X, int dx, bool bf16) {
    const int q = bf16 ? 8 : 4;   // g dx must be a multiple of q
    if (X % q != 0 || (bf16 && dx % 2 != 0)) return kGroupCells;
    for (int g = kGroupCells; g > 1; --g)
        if ((g * dx) % q == 0) return g;
    return kGroupCells;
}

// Shared memory of one warp of the resampling: its lanes' control points, then a
// staging row.
constexpr int kPhBytes = 48 * kLanes * 4;
BSI_HD int resample_warp_smem(int buf_bytes) { return kPhBytes + buf_bytes; }

// Units per tile-plane of a strip, one volume of `units` whole ones on `slots`
// resident warps: a volume of fewer strips than warps is bound by the serial walk
// of a unit's dy dz rows, not by bandwidth, and its tile-planes are split so that
// every warp gets a part (one volume per call; us for whole tile-planes -> parts:
// 64^3 at spacing 5 10.6 -> 4.2, at 8 34.0 -> 6.8; 128^3 at 5 10.6 -> 7.8; 160 x
// 192 x 192 at 8 34.3 -> 14.2).  From as many units as warps on, parts only add
// their start, 48 loads of control points: 160 x 192 x 192 at 5 22.7 us whole, 21.4
// and 22.9 in 2 and 5 parts, 256^3 at 5 36.4, 37.7 and 45.5.
BSI_HD int fwd_zparts(long long units, long long slots, int dz) {
    if (units <= 0 || units >= slots) return 1;
    const long long p = slots / units;
    return p < dz ? (int)p : dz;
}

// Tiles per strip of the resampling.  Its rows are sampled 32 voxels at a time, so a
// strip of 29 tiles that ends just past such a run wastes most of one, and most of
// all in gradient mode, which keeps one sample per lane in flight: there, and at
// x-spacing 8 (232 voxels: 7 runs and 8 voxels), strips of equal width of at most 128
// voxels, unless they are more than half as many again (each costs its z and y
// stages).  Measured (us, 29 tiles -> these): gradient mode and adjoint of 512 x 512 x
// 300 at 5 942 -> 885, 192 x 192 x 160 at 5 112 -> 101, 317 x 203 x 155 at (4, 5, 7) 176 ->
// 159, 512 x 512 x 256 at 8 1001 -> 898; value mode at 8 638 -> 524, 301 x 222 x 131 97 ->
// 81.  Value mode at 5 and 7 keeps 29 (539 against 597, 78 against 92).  Its stores
// are not bulk copies: the strips need not start on 16-byte boundaries (512 x 512 x
// 256 at 3, 28 -> 29 tiles: 592 -> 569).
inline int resample_strip_tiles(int ncx, int dx, bool grad) {
    const int most = 128 / dx;
    if (dx <= 4 || dx > kMaxSpecializedDx || !(grad || dx == 8)) return kGroupCells;
    const long long wide = cdiv(ncx, kGroupCells), n = cdiv(ncx, most);
    return 2 * n <= 3 * wide ? (int)cdiv(ncx, n) : kGroupCells;
}

// Units per tile-plane of a strip for the resampling, by a model of the rounds over
// the resident warps (a round that is not full costs 0.75 + 0.25 x its fill, none
// less than one) x the rows of a unit and 1.5 for its start.  Its rows cost more
// than the forward's and its time is their latency, so a nearly empty last round
// or a few long units decide at every size: 160 x 192 x 192 at spacing 5 in gradient
// mode, 2496 units on 2432 warps, 103 us whole and 84 in fifths; 131 x 222 x 301 at 8
// 153 -> 79 us (value) and 325 -> 145 (gradient); 256 x 512 x 512 at 8 851 -> 638 and 1096 ->
// 877.  512 x 512 x 300 at 5, 6.8 rounds, 536 us whole and 596 in fifths.
inline int resample_zparts(long long units, long long slots, int dz, int dy) {
    int best = 1;
    double best_t = -1;
    for (int p = 1; p <= dz && units > 0 && slots > 0; ++p) {
        const double n = (double)units * p / slots, full = (double)(long long)n, f = n - full;
        const double rounds = full + (f > 1e-9 ? 0.75 + 0.25 * f : 0.0);
        const double t = (rounds < 1.0 ? 1.0 : rounds) * ((dz + p - 1) / p * dy + 1.5);
        if (best_t < 0 || t < best_t) {
            best = p;
            best_t = t;
        }
    }
    return best;
}

// The same for value mode where whole tile-planes make units for half to three quarters
// of the warps: two CTAs per SM already run its gathers at their rate, so what counts there
// is the CTAs of the fullest SM (one alone takes 0.8 of the time of two, each after the third
// about half), and parts that only fill more warps lose.  Measured (us, the model above -> this):
// 64 x 290 x 97 at (6, 3, 4) 23.4 -> 16.6, 96 x 167 x 354 at (8, 5, 5) 47.8 -> 39.5; 192 x 192 x
// 160 at 5 keeps fifths, 55 against 67 whole.  Of 600 random volumes 22 were more than 5% slower
// than whole, 1.41 times at most; with this 3, 1.19 times.  Below half the model above
// is as good, from three quarters on better.
inline int resample_zparts_sm(long long units, int sms, int wpc, int dz, int dy) {
    int best = 1;
    double best_t = -1;
    for (int p = 1; p <= dz; ++p) {
        const long long k = cdiv(cdiv(units * p, wpc), sms);
        const double g = k <= 1 ? 0.8 : k == 2 ? 1.0 : 1.5 + 0.48 * (double)(k - 3);
        const double t = g * ((dz + p - 1) / p * dy + 1.0);
        if (best_t < 0 || t < best_t) {
            best = p;
            best_t = t;
        }
    }
    return best;
}

template <bool PARTS = true>
BSI_HD FwdUnit fwd_unit(const InstDesc& d, long long ul) {
    FwdUnit u;
    if (d.units <= 0x7fffffffLL) {   // 32-bit division (64-bit division is a long sequence)
        const unsigned t = (unsigned)ul / (unsigned)d.nxg;
        u.xg = (int)((unsigned)ul - t * (unsigned)d.nxg);
        u.jy = (int)(t % (unsigned)d.ncy);
        u.kz = (int)(t / (unsigned)d.ncy);
    } else {
        u.xg = (int)(ul % d.nxg);
        const long long t = ul / d.nxg;
        u.jy = (int)(t % d.ncy);
        u.kz = (int)(t / d.ncy);
    }
    u.rz0 = 0;
    u.rz1 = d.dz;
    if (PARTS && d.zparts > 1) {
        const int zp = u.kz;
        u.kz = zp / d.zparts;
        const int p = zp - u.kz * d.zparts;
        u.rz0 = d.dz * p / d.zparts;
        u.rz1 = d.dz * (p + 1) / d.zparts;
    }
    u.cell0 = u.xg * d.gcells;
    u.ncell = imin(d.gcells, d.ncx - u.cell0);
    u.x0 = u.cell0 * d.dx;
    u.nvox = imin(u.ncell * d.dx, d.X - u.x0);
    return u;
}

// ---------------------------------------------------------------- adjoint

struct AdjUnit {
    int zc, jy, xg;   // jy: the unit's first tile-row (it takes jrows of them)
    int col0;    // first complete column; lane l holds tile / column col0 - 3 + l
    int xs;      // first voxel read by the warp
    int nvox;    // voxels per row read by the warp
    int kz0, kz1;
};

BSI_HD AdjUnit adj_unit(const InstDesc& d, long long ul) {
    AdjUnit u;
    u.xg = (int)(ul % d.nxg);
    const long long t = ul / d.nxg;
    u.jy = (int)(t % d.ncyu) * d.jrows;
    u.zc = (int)(t / d.ncyu);
    u.col0 = u.xg * kGroupCells;
    const int c_lo = imax(0, u.col0 - kHalo);
    const int c_hi = imin(d.ncx, u.col0 + kGroupCells);
    u.xs = c_lo * d.dx;
    u.nvox = c_hi > c_lo ? imin(d.X, c_hi * d.dx) - u.xs : 0;
    u.kz0 = u.zc * d.zchunk;
    u.kz1 = imin(d.ncz, u.kz0 + d.zchunk);
    return u;
}

// Floats of partial sums one adjoint unit writes: (zchunk + 3) planes x
// (jrows + 3) grid rows x 29 columns x 3 channels.
BSI_HD long long adj_unit_floats(const InstDesc& d) {
    return (long long)(d.zchunk + kHalo) * (d.jrows + kHalo) * kGroupCells * 3;
}

// Partial sum of a unit: grid plane pz of its window, grid row m (0 .. jrows + 2,
// from its first tile-row), column j.
BSI_HD long long part_elem(const InstDesc& d, long long ul, int pz, int m, int j) {
    return d.part_off + ul * adj_unit_floats(d) + (((long long)pz * (d.jrows + kHalo) + m) * kGroupCells + j) * 3;
}

// Staging buffer bytes for a largest x-spacing dxmax: one row segment of up to
// 32 tiles x dxmax voxels x 3 FP32 channels, plus up to 15 bytes of alignment
// shift on each side (the adjoint's bulk loads cover the 16-byte-aligned
// superset of a row segment).
BSI_HD int stage_buf_bytes(int dxmax) {
    const int b = 32 + kLanes * dxmax * 3 * 4;
    return (b + 15) & ~15;
}

constexpr int kStoreStages = 3;   // forward: ring of staging buffers per warp (bulk stores in flight)
constexpr int kLoadStages = 2;    // adjoint row-copy path: ring of blocks per warp

// Shared memory of one warp: forward -- the store ring; adjoint row-copy path --
// a head (the stages' mbarriers, then 128 bytes of zeros), then the load ring.
// A ring stage holds a block of rows of the instance's own x-spacing; with 9.25
// KB stages twelve warps (three 4-warp CTAs) share an SM's shared memory.  Of the
// generic kernel's rows it may hold one only.
constexpr int kRowSpareOff = 64;
constexpr int kRowHeadBytes = 256;
constexpr int kRowStageBytes = 9472;
BSI_HD int fwd_warp_smem(int buf_bytes) { return kStoreStages * buf_bytes; }
BSI_HD int adj_warp_smem(int stage_bytes) { return kRowHeadBytes + kLoadStages * stage_bytes; }
// Bytes of a ring stage in a launch of x-spacings up to dxmax.  deep: two rows of the
// widest spacing at least (the generic kernel's rows of 13 and more voxels per tile),
// where the warps that this costs are not missed (plan_row_stages).
BSI_HD int row_stage_bytes(int dxmax, bool deep) {
    return imax(kRowStageBytes, (deep ? 2 : 1) * stage_buf_bytes(dxmax));
}
// Zero voxels written after a staged row for the tile that the volume's end cuts:
// what that tile lacks and no more.  Where it is the last of a strip of 32 tiles it
// ends with the row's slot, and the next row's slot follows.
BSI_HD int row_tail_voxels(const InstDesc& d) { return d.ncx * d.dx - d.X; }
// Rows per block at spacing (dx, dy): as many as fit a stage, in even blocks.
BSI_HD int row_block_rows(int dx, int dy, int stage_bytes) {
    const int rb = imax(1, imin(imin(dy, kLanes), stage_bytes / stage_buf_bytes(dx)));
    return (int)cdiv(dy, cdiv(dy, rb));
}

// Forward on the tensor-store path (one volume, three channels): when every row
// of the field is a multiple of 16 bytes and every strip starts on a 16-byte
// boundary, a warp stages rb rows of its strip (a block) and writes the block
// with one tensor store instead of one bulk copy per row.  The box is the
// strip's row as 8-byte elements (at most 256) x rb rows x 1 plane; rb divides
// the y-spacing, so that a block never reaches into the next tile-row, and the
// warp's kStoreStages blocks (128-byte aligned, plus a 128-byte slot the halo
// lanes stage into) fit 1/16 of an SM's shared memory (two 8-warp CTAs).
constexpr int kFwdTmaWarpBudget = 14 * 1024;
constexpr int kBf16OddStripTiles = 24;   // BF16 strips at odd x-spacings on that path: 6 g dx % 16 == 0
BSI_HD int pad128(int b) { return (b + 127) & ~127; }
BSI_HD int fwd_tma_row_bytes(int gcells, int dx, bool bf16, int c = 3) { return gcells * dx * c * (bf16 ? 2 : 4); }
BSI_HD int fwd_tma_warp_smem(int blk_bytes) { return kStoreStages * blk_bytes + 128; }

// Rows per block of the tensor-store path, or 0 where it does not apply
// (rows or strips off 16-byte boundaries, boxes wider than 256 elements, no
// divisor of dy >= 2 whose blocks fit, or FP32 output at x-spacings >= 5).
// Measured on 512^3: FP32 at spacing 3 0.389 -> 0.352 ms and at 4 0.269 ->
// 0.250 ms (bound by per-row work); BF16 at 4, 6, 8 14-16% faster; FP32 at 6,
// already at the write roofline, 0.231 -> 0.246 ms (so not taken).
BSI_HD int fwd_tma_rows(int X, int dx, int dy, int gcells, bool bf16, int c = 3) {
    const int rowb = fwd_tma_row_bytes(gcells, dx, bf16, c);
    if (dx < 1 || dx > (bf16 ? kMaxSpecializedDx : 4) || (c * X * (bf16 ? 2 : 4)) % 16 != 0 || rowb % 16 != 0 ||
        rowb / 8 > 256)
        return 0;
    for (int rb = dy; rb >= 2; --rb)
        if (dy % rb == 0 && fwd_tma_warp_smem(pad128(rb * rowb)) <= kFwdTmaWarpBudget) return rb;
    return 0;
}

// ---------------------------------------------------------------- adjoint, tensor-copy path
//
// When the voxel gradient's rows are 16-byte multiples (X % 4 == 0) and
// dx <= 8, the adjoint fetches its input with TMA tensor copies from a 3-D
// view of the gradient as 8-byte elements (pairs of floats): (3X/2, Y, Z).
// One ring stage holds a BLOCK: rb consecutive rows of a voxel plane of the
// unit's tile-row, 32 tiles wide (rb divides dy, so a plane is dy / rb blocks).
// A box row is one contiguous run of a gradient row (<= 256 elements per box
// dimension): one box of 48 dx + 2 elements for dx <= 5, else two boxes of
// 24 dx + 2 elements, lanes 0..15 reading the first and 16..31 the second.
// The first box starts at the 16-byte group holding the unit's first float,
// which may lie before the array: elements outside it arrive as zeros.
BSI_HD int tma_boxes(int dx) { return dx <= 5 ? 1 : 2; }
BSI_HD int tma_box_width(int dx) { return tma_boxes(dx) == 1 ? 48 * dx + 2 : 24 * dx + 2; }
// Shared bytes of one box of rb rows, padded to the 128 bytes a tensor copy's
// destination is aligned to.
BSI_HD int tma_box_bytes(int dx, int rb) { return (8 * tma_box_width(dx) * rb + 127) & ~127; }
BSI_HD int tma_block_bytes(int dx, int rb) { return tma_boxes(dx) * tma_box_bytes(dx, rb); }

constexpr int kTmaMaxRows = 8;                   // rows per block
constexpr int kTmaBlockTarget = 14 * 1024;       // largest block that still leaves room for 2 stages x 8 warps
constexpr int kTmaMinStages = 2;
constexpr int kTmaMaxStages = 4;
constexpr int kTmaMaxWarps = 12;                 // register budget: 12 warps x 32 x 170 <= 65536
constexpr int kTmaMaxWarps2 = 11;                // two tile-rows per unit: 11 warps x 32 x 186
constexpr int kTmaSmemBudget = 227 * 1024;       // one CTA per SM takes all of its shared memory

// Rows per block for spacing (dx, dy): the largest divisor of dy up to
// kTmaMaxRows whose block fits kTmaBlockTarget (1 always does).
BSI_HD int tma_block_rows(int dx, int dy) {
    for (int rb = imin(dy, kTmaMaxRows); rb > 1; --rb)
        if (dy % rb == 0 && tma_block_bytes(dx, rb) <= kTmaBlockTarget) return rb;
    return 1;
}
// Shared memory of one warp: 128 bytes of mbarriers, then the ring of stages.
BSI_HD int tma_warp_smem(int stage_bytes, int stages) { return 128 + stages * stage_bytes; }
// Default ring depth for a stage size, 2 or 3: 3 where it still fits beside
// 12 warps (measured: a 4th stage slowed small blocks down; 3 beat 2 where
// both fit), and also where two stages fall short of 12 warps anyway while
// three keep at least 7.  Measured on the 512 x 512 x 300 volume at spacing 5
// (9.7 KB stages: 11 warps x 2 stages or 7 warps x 3): equal alone, 11 us
// faster right after a forward, whose field is still leaving L2 -- the deeper
// ring rides out the longer load latency.  Where two stages reach 12 warps
// (512^3 at spacing (4,5,6)) or three would leave 6 (spacing 8), fewer warps
// cost 12-25% and the ring stays at 2.
constexpr int kTmaMinDeepWarps = 7;
BSI_HD int tma_default_stages(int stage_bytes) {
    const int w2 = (kTmaSmemBudget - 128) / tma_warp_smem(stage_bytes, 2);
    const int w3 = (kTmaSmemBudget - 128) / tma_warp_smem(stage_bytes, 3);
    return (w3 >= kTmaMaxWarps || (w2 < kTmaMaxWarps && w3 >= kTmaMinDeepWarps)) ? 3 : 2;
}

// Float index (x * 3 + channel) of the unit's first float and its 16-byte group.
BSI_HD int tma_first_float(const AdjUnit& u, int dx) { return (u.col0 - kHalo) * 3 * dx; }
BSI_HD int tma_group_of(int f) { return f >= 0 ? f / 4 : -((-f + 3) / 4); }   // floor(f / 4)

// ---------------------------------------------------------------- non-integer spacing

// One volume with spacing num/den and lattice shift off/den per axis (x, y, z).
struct RatDesc {
    int X, Y, Z;
    int num[3], den[3], off[3];
    int nx, ny, nz;
    const float* phi;
    float* field;
};

// Stored grid points along one axis: floor(((N - 1) den + off) / num) + 4.
BSI_HD long long rational_dim(long long N, int num, int den, int off) {
    return N > 0 ? ((N - 1) * den + off) / num + 4 : 4;
}

// Cells of any width (bsi_cells_forward.cu, bsi_cells_adjoint.cu: non-integer spacing, integer x-spacings
// above kMaxSpecializedDx as den = 1, off = 0).  A cell of an axis holds the
// voxels x with floor((x den + off) / num) = its index; its width is the floor
// or the ceiling of num / den, less at the volume's ends.  A warp takes strips
// of sc x-cells.  A cell of up to 7 voxels belongs to one lane; a wider one is
// shared by `parts` neighbouring lanes, each taking an even run of it (floor or
// ceiling of width / parts, at most 7: odd runs keep the 12-byte voxel stride
// of the lanes off common shared-memory banks), so that a row's work is spread
// over the whole warp at every spacing.
constexpr int kCellRunMax = 7;      // cells of up to this many voxels belong to one lane
constexpr int kCellWideRun = 7;     // run bound for wider cells
constexpr int kCellRowsMax = 64;    // rows (planes) of a y-cell (z-cell): spacing <= 64

// First voxel of cell k of an axis: the least x with x den + off >= k num (k up
// to a strip past the last cell: k num stays below 2^30 + 2^22, see the limits of
// the API).
BSI_HD int cell_first(int k, int num, int den, int off) {
    const int t = k * num - off;
    return t <= 0 ? 0 : den == 1 ? t : (int)((unsigned)(t + den - 1) / (unsigned)den);
}

struct CellPlan {
    int ncx, ncy, ncz;   // cells per axis
    int parts, run;      // lanes per x-cell, and the longest run of one lane
    int vec;             // runs of 4 voxels on 16-byte boundaries (see cell_plan)
    int sc, nsx;         // x-cells per strip, strips
    int nc;              // columns a strip touches: sc + 3
    int zc, zsplit;      // z-cells per unit, or (zsplit > 1, zc = 1) units per z-cell
    int ysplit, nyu;     // units per y-cell (1 in the adjoint), y-units: ncy ysplit
    int nzu;             // z-units: ceil(ncz / zc) or ncz zsplit
    int ymax, zmax;      // most rows of a unit, most planes
    int slot;            // bytes of one staged row (16-byte multiple)
    int rb;              // rows per block
    int stage_bytes;     // rb slots
    int head_bytes;      // per warp, ahead of the ring: barriers, a spare row, the unit's y and z weights
    int warp_bytes;
    long long units;
    long long part_floats;   // adjoint: partial sums
};

constexpr int kCellSpareOff = 64;    // spare run (adjoint: zeros; forward: never stored) after the barriers
constexpr int kCellWeightOff = 192;  // y weights, then z weights (16 bytes each)
constexpr int kCellStages = 2;       // blocks in flight per warp

// One unit: planes [z0, z1) of the z-cells [kz0, kz1), rows [y0, y1) of y-cell
// jy, x-cells [c0, c0 + cells) with voxels [sx0, sx1).
struct CellUnit {
    int xs, jy, kz0, kz1, z0, z1, y0, y1;
};

template <bool YSPLIT>
BSI_HD CellUnit cell_unit(const RatDesc& d, const CellPlan& c, long long un) {
    CellUnit u;
    int zi;
    if (c.units <= 0x7fffffffLL) {   // 32-bit division (64-bit division is a long sequence)
        const unsigned t = (unsigned)un / (unsigned)c.nsx;
        u.xs = (int)((unsigned)un - t * (unsigned)c.nsx);
        zi = (int)(t / (unsigned)c.nyu);
        u.jy = (int)(t - (unsigned)zi * (unsigned)c.nyu);
    } else {
        u.xs = (int)(un % c.nsx);
        const long long t = un / c.nsx;
        u.jy = (int)(t % c.nyu);
        zi = (int)(t / c.nyu);
    }
    if (c.zsplit > 1) {
        u.kz0 = zi / c.zsplit;
        u.kz1 = u.kz0 + 1;
    } else {
        u.kz0 = zi * c.zc;
        u.kz1 = imin(u.kz0 + c.zc, c.ncz);
    }
    u.z0 = cell_first(u.kz0, d.num[2], d.den[2], d.off[2]);
    u.z1 = imin(d.Z, cell_first(u.kz1, d.num[2], d.den[2], d.off[2]));
    if (c.zsplit > 1) {
        const int n = u.z1 - u.z0, p = zi - u.kz0 * c.zsplit, a = u.z0;
        u.z0 = a + n * p / c.zsplit;
        u.z1 = a + n * (p + 1) / c.zsplit;
    }
    int p = 0;   // part of the y-cell
    if (YSPLIT && c.ysplit > 1) {
        p = u.jy % c.ysplit;
        u.jy /= c.ysplit;
    }
    u.y0 = cell_first(u.jy, d.num[1], d.den[1], d.off[1]);
    u.y1 = imin(d.Y, cell_first(u.jy + 1, d.num[1], d.den[1], d.off[1]));
    if (YSPLIT && c.ysplit > 1) {
        const int n = u.y1 - u.y0, a = u.y0;
        u.y0 = a + n * p / c.ysplit;
        u.y1 = a + n * (p + 1) / c.ysplit;
    }
    return u;
}

// The x side of strip xs and of one lane in it: its part lp of cell c0 + lc.
struct CellStrip {
    int c0, cells, sx0, sx1;
};
struct CellRun {
    int col, xa, cnt;   // the lane's cell, first voxel and voxels (0: none)
};

BSI_HD CellStrip cell_strip(const RatDesc& d, const CellPlan& c, int xs) {
    CellStrip s;
    s.c0 = xs * c.sc;
    s.cells = imin(c.sc, c.ncx - s.c0);
    s.sx0 = cell_first(s.c0, d.num[0], d.den[0], d.off[0]);
    s.sx1 = imin(d.X, cell_first(s.c0 + s.cells, d.num[0], d.den[0], d.off[0]));
    return s;
}

BSI_HD CellRun cell_run(const RatDesc& d, const CellPlan& c, const CellStrip& s, int lane) {
    CellRun r;
    const int lc = lane / c.parts, lp = lane - lc * c.parts;
    r.col = s.c0 + lc;
    r.xa = s.sx0;
    r.cnt = 0;
    if (lc < s.cells) {
        const int a = cell_first(r.col, d.num[0], d.den[0], d.off[0]);
        const int w = imin(d.X, cell_first(r.col + 1, d.num[0], d.den[0], d.off[0])) - a;
        const int i0 = c.vec ? imin(w, 4 * lp) : w * lp / c.parts;
        const int i1 = c.vec ? imin(w, 4 * lp + 4) : w * (lp + 1) / c.parts;
        r.xa = a + i0;
        r.cnt = i1 - i0;
    }
    return r;
}

// Float offset of a unit's partial sums: plane pz (0 .. zc + 2), grid row m (0 ..
// 3), column j (0 .. nc - 1).
BSI_HD long long cell_part(const CellPlan& c, long long un, int pz, int m, int j) {
    return ((un * (c.zc + kHalo) + pz) * 4 + m) * (3LL * c.nc) + 3LL * j;
}

// Shared memory of one warp: twelve warps (three CTAs) share an SM's 228 KB,
// 1 KB per CTA set aside.
constexpr int kCellWarpsPerSm = 12;
constexpr int kCellWarpBudget = (225 * 1024 / kCellWarpsPerSm) & ~127;

// Plan of a volume (a rule of its geometry only, so that a workspace query
// needs no device).  Adjoint: z-cells per unit, or units per z-cell (forward:
// one cell, or a part of it -- where parts of one plane still leave warps idle, of its
// rows too: forward of 64^3 at 24 12.1 -> 5.4 us, 128^3 at 32 10.3 -> 8.3), by a cost model of rounds over the warps of a
// 152-SM GPU x rows of a unit, in units of one staged row; a last, partial
// round costs 0.6 + 0.4 x its fill (a lone warp per scheduler runs faster); a unit costs about kUnitRows rows to start and half
// a row per plane of partial sums, and a partial sum is written and read once.  Only plans of
// at most max_floats partial sums (when >= 0); if none fits, the smallest.
// vec: rows on 16-byte boundaries (X % 4 == 0, aligned array) may take runs of
// exactly 4 voxels -- three 16-byte vectors at a lane stride of 48 bytes, which
// meets no bank conflict -- where the x-spacing is an integer multiple of 4 above
// kCellRunMax.
inline CellPlan cell_plan(const RatDesc& d, bool adjoint, bool vec, long long max_floats = -1) {
    constexpr double kUnitRows = 4.0;
    CellPlan c = {};
    auto cells = [&](int a, int N) { return (int)(((long long)(N - 1) * d.den[a] + d.off[a]) / d.num[a]) + 1; };
    auto widest = [&](int a, int N) { return imin(N, (d.num[a] + d.den[a] - 1) / d.den[a]); };
    c.ncx = cells(0, d.X);
    c.ncy = cells(1, d.Y);
    c.ncz = cells(2, d.Z);
    const int w = (d.num[0] + d.den[0] - 1) / d.den[0];
    c.vec = vec && d.X % 4 == 0 && d.den[0] == 1 && d.off[0] == 0 && w % 4 == 0 && w > kCellRunMax;
    c.parts = w <= kCellRunMax ? 1 : c.vec ? w / 4 : (w + kCellWideRun - 1) / kCellWideRun;
    c.run = (w + c.parts - 1) / c.parts;
    const int per = c.parts == 1 ? kGroupCells : kLanes / c.parts;
    c.nsx = (int)cdiv(c.ncx, per);
    c.sc = (int)cdiv(c.ncx, c.nsx);   // strips of even width
    c.nsx = (int)cdiv(c.ncx, c.sc);
    c.nc = c.sc + kHalo;
    const int vox = imin(d.X, (int)((long long)c.sc * d.num[0] / d.den[0]) + 1);
    c.slot = (12 * vox + 32 + 15) & ~15;
    const int yw = widest(1, d.Y);
    c.zmax = kCellRowsMax;
    const int zw = widest(2, d.Z);
    const double rows = (double)d.num[1] / d.den[1], planes = (double)d.num[2] / d.den[2];
    const double slots = 152.0 * kCellWarpsPerSm;
    c.zc = c.zsplit = c.ysplit = 1;
    auto size = [&](CellPlan& p) {
        p.nzu = p.zsplit > 1 ? p.ncz * p.zsplit : (int)cdiv(p.ncz, p.zc);
        p.nyu = p.ncy * p.ysplit;
        p.units = (long long)p.nzu * p.nyu * p.nsx;
        p.part_floats = adjoint ? p.units * (p.zc + kHalo) * 4 * 3 * p.nc : 0;
    };
    CellPlan best = c, p = c;
    double best_t = -1;
    bool fits = false;
    for (int k = adjoint ? 0 : 7; k < 14; ++k) {   // zc = 8 .. 1, then 2, 4 .. 64 units per z-cell
        p.zc = k < 8 ? 8 - k : 1;
        p.zsplit = k < 8 ? 1 : 1 << (k - 7);
        if (p.zc * zw > kCellRowsMax || p.zsplit > zw) continue;
        // parts of y-cells only beside the shortest parts of z-cells
        const int ymost = !adjoint && 2 * p.zsplit > zw ? yw : 1;
        for (p.ysplit = 1; p.ysplit <= ymost; p.ysplit *= 2) {
            size(p);
            const bool f = max_floats < 0 || p.part_floats <= max_floats;
            const double n = p.units / slots, full = (double)(long long)n, part = n - full;
            const double start = adjoint ? kUnitRows + 0.5 * (p.zc + kHalo) : kUnitRows;
            const double t = (full + (part > 1e-9 ? 0.6 + 0.4 * part : 0.0)) *
                                 (planes * p.zc / p.zsplit * rows / p.ysplit + start) +
                             p.part_floats * 4.0 / (12.0 * vox * slots);
            if (best_t < 0 || (f && !fits) || (f == fits && (f ? t < best_t : p.part_floats < best.part_floats))) {
                best = p;
                best_t = t;
                fits = f;
            }
        }
    }
    c = best;
    c.ymax = (int)cdiv(yw, c.ysplit);
    c.zmax = imin(kCellRowsMax, c.zc * zw);
    c.head_bytes = pad128(kCellWeightOff + 16 * (c.ymax + c.zmax));
    int rb = (kCellWarpBudget - c.head_bytes) / (kCellStages * c.slot);
    rb = imax(1, imin(imin(rb, c.ymax), kLanes));
    c.rb = (int)cdiv(c.ymax, cdiv(c.ymax, rb));   // even blocks
    c.stage_bytes = c.rb * c.slot;
    c.warp_bytes = pad128(c.head_bytes + kCellStages * c.stage_bytes);
    return c;
}

constexpr int kMaxWarpsPerCta = 8;
constexpr int kAdjWarpsMax = 4;   // adjoint partials kernel: 4-warp CTAs (register budget)
constexpr int kSmemBudget = 200 * 1024;   // dynamic shared memory per CTA we allow

// Warps per CTA such that the warps' shared memory fits the budget, at most
// `req` when a tile config asks for fewer (req = 0: no request).
BSI_HD int warps_per_cta(int warp_smem, int req = 0) {
    int w = kSmemBudget / warp_smem;
    if (req > 0 && req < w) w = req;
    return w < 1 ? 1 : (w > kMaxWarpsPerCta ? kMaxWarpsPerCta : w);
}

}  // namespace bsi
