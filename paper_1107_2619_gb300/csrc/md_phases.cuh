// Per-item device functions of the hot path, shared by the stand-alone kernels and the
// persistent step kernel.  Each function does the work of one item (an atom, a cell or a
// scan tile); the callers supply the loop.
//
// Systems: one or several independent replicas (batched systems).  Atoms of replica r
// occupy a contiguous range of the per-atom arrays; rep[i] (NULL for a single system) gives
// the replica of slot i, boxes[r] its box, rc[r] its link-cell grid, whose cells occupy the
// global cell range [rc[r].base, rc[r].base + ncell_r).
#pragma once

#include <cuda_runtime.h>

#include "md_bits.cuh"
#include "md_internal.cuh"
#include "md_pack2.cuh"

namespace mdk {
namespace ph {

__device__ __forceinline__ bool rebuild_requested(const Flags *f) {
    return *reinterpret_cast<const volatile int32_t *>(&f->need_rebuild) != 0;
}

__device__ __forceinline__ int replica_of(const Atoms &A, int i) { return A.rep ? A.rep[i] : 0; }

// Cell index along one edge from the wrapped fractional coordinate.
__device__ __forceinline__ int cell_coord(double x, double invL, int nc) {
    double s = x * invL;
    s = s - floor(s);
    int c = (int)(s * (double)nc);
    return min(max(c, 0), nc - 1);
}

// Positions in the image of the last build (ref: the position at that build), FP64 and FP32.
__device__ __forceinline__ double4_32a build_image64(const double4_32a &p, const double4_32a &ref, const Box &B) {
    return make_double4_32a(p.x - B.L[0] * floor(ref.x * B.invL[0]), p.y - B.L[1] * floor(ref.y * B.invL[1]),
                            p.z - B.L[2] * floor(ref.z * B.invL[2]), p.w);
}

// FP32 position in the periodic image its atom was wrapped into at the last list build (the
// image of ref, the position at that build): the wrapped position until the atom crosses a box
// face, continuous after it, so that it stays within skin/2 of its link cell (the group walks
// add each cell's image shift to these coordinates; the list passes take the minimum image).
__device__ __forceinline__ float4 build_image(const double4_32a &p, const double4_32a &ref, const Box &B,
                                              int species) {
    return make_float4((float)(p.x - B.L[0] * floor(ref.x * B.invL[0])),
                       (float)(p.y - B.L[1] * floor(ref.y * B.invL[1])),
                       (float)(p.z - B.L[2] * floor(ref.z * B.invL[2])), __int_as_float(species));
}

// Double-float copy of an FP64 image coordinate q (MD_PREC_DF): q + xoff split into an FP32 high
// part and the FP32 rounding of the remainder (conversions on the bit fields).
__device__ __forceinline__ void store_dfpos(const Atoms &A, int i, const double4_32a &q, const Box &B) {
    const double x = q.x + B.xoff[0], y = q.y + B.xoff[1], z = q.z + B.xoff[2];
    const float xh = eam::f32_rn(x), yh = eam::f32_rn(y), zh = eam::f32_rn(z);
    A.posx[2 * (size_t)i] = make_float4(xh, yh, zh, 0.f);
    A.posx[2 * (size_t)i + 1] = make_float4(eam::f32_rn(x - eam::f64_of_f32(xh)), eam::f32_rn(y - eam::f64_of_f32(yh)),
                                            eam::f32_rn(z - eam::f64_of_f32(zh)), 0.f);
}

// Fixed-point copy of an FP64 image coordinate q (Atoms::posq).  A coordinate that is not finite has
// none: it is reported here, as it would otherwise be by the forces it leads to.
__device__ __forceinline__ void store_fixed(const Atoms &A, int i, const double4_32a &q) {
    if (!(eam::finite64(q.x) && eam::finite64(q.y) && eam::finite64(q.z))) atomicOr(&A.flags->error, FLAG_NONFINITE);
    A.posq[i] = make_double4_32a(__longlong_as_double(eam::fix64(q.x, A.qfb)), __longlong_as_double(eam::fix64(q.y, A.qfb)),
                                 __longlong_as_double(eam::fix64(q.z, A.qfb)), 0.0);
}

// The whole box edges to take off per axis, floor(r / L), as three signed 10-bit fields (0: none, as
// for most atoms); kImageFar where one does not fit.
constexpr int kImageFar = (int)0x80000000;
__device__ __forceinline__ int pack_image(double fx, double fy, double fz) {
    const float x = eam::f32_rn(fx), y = eam::f32_rn(fy), z = eam::f32_rn(fz);   // whole numbers: exact where they fit
    if (!(fabsf(x) < 512.f && fabsf(y) < 512.f && fabsf(z) < 512.f)) return kImageFar;
    return (((int)x & 1023) << 20) | (((int)y & 1023) << 10) | ((int)z & 1023);
}

__device__ __forceinline__ int global_cell(const double4_32a &p, const Box &B, const RepCells &g) {
    const int cx = cell_coord(p.x, B.invL[0], g.nc[0]);
    const int cy = cell_coord(p.y, B.invL[1], g.nc[1]);
    const int cz = cell_coord(p.z, B.invL[2], g.nc[2]);
    return g.base + (cz * g.nc[1] + cy) * g.nc[0] + cx;
}

// Block-wide exclusive scan of one int per thread; returns the block total in `total`.
__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int &total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    int prefix = (w > 0 ? warp_sums[w - 1] : 0) + x - v;
    total = warp_sums[nw - 1];
    __syncthreads();
    return prefix;
}

// ---------------------------------------------------------------- integration (§2.3, §2.2)
// The exact displacement check: an atom more than skin/2 from its position at the last build (or
// not finite) asks for a rebuild.
__device__ __forceinline__ void check_exact(const Atoms &A, const double4_32a &p, const double4_32a &r, double lim2) {
    const double ex = __dsub_rn(p.x, r.x), ey = __dsub_rn(p.y, r.y), ez = __dsub_rn(p.z, r.z);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
    if (d2 > lim2 || !(d2 == d2)) {
        A.flags->need_rebuild = 1;
        A.flags->skin_exceeded = 1;
    }
}

// What follows a move of atom i to p: the skin check and the copies of the position that the
// passes read, in the periodic image of the last build.  The FP64 pipe bounds the per-atom work
// (see md_bits.cuh), so without a strain ramp (A.image_fixed) none of this runs on it for most
// atoms: the box edges to take off come from the build (reff.w, 0 for most), the FP32 copy is
// rounded on the bit fields, and the displacement is first formed from the FP32 positions, the
// exact check following only where that lies within its rounding of the limit (lim.d2f).  The
// copies, and the decision, are the same bits as with the exact operations throughout.
__device__ __forceinline__ void place(const Atoms &A, const Box *boxes, int i, const double4_32a &p, SkinLimit lim) {
    if (!A.image_fixed) {
        const double4_32a r = A.ref[i];
        check_exact(A, p, r, lim.d2);
        const Box &B = boxes[replica_of(A, i)];
        A.posf[i] = build_image(p, r, B, A.spec[i]);
        if (A.posd) {
            const double4_32a q = build_image64(p, r, B);
            A.posd[i] = q;
            if (A.posx) store_dfpos(A, i, q, B);
            if (A.posq) store_fixed(A, i, q);
        }
        return;
    }
    const float4 rf = A.reff[i];
    const int im = __float_as_int(rf.w);
    double4_32a q = p;
    if (im != 0) {
        const Box &B = boxes[replica_of(A, i)];
        if (im == kImageFar) {
            q = build_image64(p, A.ref[i], B);
        } else {   // small whole numbers, exact through FP32
            q.x = fma(-B.L[0], eam::f64_of_f32((float)((im << 2) >> 22)), p.x);
            q.y = fma(-B.L[1], eam::f64_of_f32((float)((im << 12) >> 22)), p.y);
            q.z = fma(-B.L[2], eam::f64_of_f32((float)((im << 22) >> 22)), p.z);
        }
    }
    const float fx = eam::f32_rn(q.x), fy = eam::f32_rn(q.y), fz = eam::f32_rn(q.z);
    const float ex = fx - rf.x, ey = fy - rf.y, ez = fz - rf.z;
    if (!(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= lim.d2f)) check_exact(A, p, A.ref[i], lim.d2);
    A.posf[i] = make_float4(fx, fy, fz, __int_as_float(A.spec[i]));
    if (A.posd) {
        A.posd[i] = q;
        if (A.posx) store_dfpos(A, i, q, boxes[replica_of(A, i)]);
        if (A.posq) store_fixed(A, i, q);
    }
}

// v += (dt/2) F/m;  r += dt v;  [z *= s];  then place().  Separately rounded FP64 operations, as in
// the definition.
__device__ __forceinline__ void kick_drift(const Atoms &A, const Box *boxes, int i, double half_dt, double dt,
                                           double s, bool strain, SkinLimit lim, const Thermo *th = nullptr) {
    double4_32a v = A.vel[i];
    if (th) {  // the thermostat half steps before this kick: v *= s_b, then v *= s_a
        const Thermo &t = th[replica_of(A, i)];
        v.x = __dmul_rn(__dmul_rn(v.x, t.s_b), t.s_a);
        v.y = __dmul_rn(__dmul_rn(v.y, t.s_b), t.s_a);
        v.z = __dmul_rn(__dmul_rn(v.z, t.s_b), t.s_a);
    }
    const double4_32a f = A.force[i];
    double4_32a p = A.pos[i];
    v.x = __dadd_rn(v.x, __dmul_rn(__dmul_rn(half_dt, f.x), v.w));
    v.y = __dadd_rn(v.y, __dmul_rn(__dmul_rn(half_dt, f.y), v.w));
    v.z = __dadd_rn(v.z, __dmul_rn(__dmul_rn(half_dt, f.z), v.w));
    p.x = __dadd_rn(p.x, __dmul_rn(dt, v.x));
    p.y = __dadd_rn(p.y, __dmul_rn(dt, v.y));
    p.z = __dadd_rn(p.z, __dmul_rn(dt, v.z));
    if (strain) p.z = __dmul_rn(p.z, s);
    A.vel[i] = v;
    A.pos[i] = p;
    place(A, boxes, i, p, lim);
}

// The predictor of the third-order predictor-corrector (md.h MD_INTEGRATOR_PC3): from the force f
// of the last evaluation (acceleration term q2 = (dt^2/2) f/m) and the third-derivative term q3,
//   r += dt v + q2 + q3,  v += (2 q2 + 3 q3) / dt,  g2 = q2 + 3 q3 (the predicted acceleration
// term, for the corrector), then the skin check and the pass copies, as after a drift.
__device__ __forceinline__ void predict_pc3(const Atoms &A, const Box *boxes, int i, double dt, SkinLimit lim) {
    double4_32a v = A.vel[i], p = A.pos[i];
    const double4_32a f = A.force[i], q3 = A.g3[i];
    const double h2 = 0.5 * dt * dt;
    const double ax = __dmul_rn(__dmul_rn(h2, f.x), v.w), ay = __dmul_rn(__dmul_rn(h2, f.y), v.w),
                 az = __dmul_rn(__dmul_rn(h2, f.z), v.w);
    p.x = __dadd_rn(p.x, __dadd_rn(__dadd_rn(__dmul_rn(dt, v.x), ax), q3.x));
    p.y = __dadd_rn(p.y, __dadd_rn(__dadd_rn(__dmul_rn(dt, v.y), ay), q3.y));
    p.z = __dadd_rn(p.z, __dadd_rn(__dadd_rn(__dmul_rn(dt, v.z), az), q3.z));
    const double bx = __dmul_rn(3.0, q3.x), by = __dmul_rn(3.0, q3.y), bz = __dmul_rn(3.0, q3.z);
    v.x = __dadd_rn(v.x, __ddiv_rn(__dadd_rn(__dmul_rn(2.0, ax), bx), dt));
    v.y = __dadd_rn(v.y, __ddiv_rn(__dadd_rn(__dmul_rn(2.0, ay), by), dt));
    v.z = __dadd_rn(v.z, __ddiv_rn(__dadd_rn(__dmul_rn(2.0, az), bz), dt));
    A.g2[i] = make_double4_32a(__dadd_rn(ax, bx), __dadd_rn(ay, by), __dadd_rn(az, bz), 0.0);
    A.vel[i] = v;
    A.pos[i] = p;
    place(A, boxes, i, p, lim);
}

// What opens a step: the half kick and drift of velocity Verlet, or the predictor.
__device__ __forceinline__ void open_step(const Atoms &A, const Box *boxes, int i, int motion, double half_dt,
                                          double dt, double s, bool strain, SkinLimit lim, const Thermo *th = nullptr) {
    if (motion == kMotionPC3) predict_pc3(A, boxes, i, dt, lim);
    else kick_drift(A, boxes, i, half_dt, dt, s, strain, lim, th);
}

// The displacement check of positions already placed (posf current: not after a corrector).
__device__ __forceinline__ void check_displacement(const Atoms &A, int i, SkinLimit lim) {
    if (A.image_fixed && !A.g3) {
        const float4 f = A.posf[i], rf = A.reff[i];
        const float ex = f.x - rf.x, ey = f.y - rf.y, ez = f.z - rf.z;
        if (fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= lim.d2f) return;
    }
    check_exact(A, A.pos[i], A.ref[i], lim.d2);
}

// ---------------------------------------------------------------- rebuild (§3.2.1, §3.2.2)
__device__ __forceinline__ void bin_atom(const Atoms &A, const Cells &C, const Box *boxes, int i) {
    const int r = replica_of(A, i);
    const int c = global_cell(A.pos[i], boxes[r], C.rc[r]);
    A.cell_of[i] = c;
    A.slot[i] = atomicAdd(&C.cell_count[c], 1);
}

// The scan works on tiles of blockDim.x * kScanItems cells.
constexpr int kScanItems = 4;

__device__ __forceinline__ int scan_tiles(const Cells &C) {
    const int tile = blockDim.x * kScanItems;
    return (C.ncell + tile - 1) / tile;
}

// Scan phase 1: tile sums.
__device__ __forceinline__ void scan_tile_sum(const Cells &C, int tile, int *ws) {
    const int base = tile * blockDim.x * kScanItems + threadIdx.x * kScanItems;
    int s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++)
        if (base + k < C.ncell) s += C.cell_count[base + k];
    int total;
    block_exclusive_scan(s, ws, total);
    if (threadIdx.x == 0) C.tile_sums[tile] = total;
}

// Scan phase 2 (one block): exclusive scan of the tile sums in place.
__device__ __forceinline__ void scan_top(const Cells &C, int *ws) {
    const int ntiles = scan_tiles(C);
    int carry = 0;
    for (int base = 0; base < ntiles; base += blockDim.x * kScanItems) {
        const int idx = base + threadIdx.x * kScanItems;
        int v[kScanItems], s = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            v[k] = (idx + k < ntiles) ? C.tile_sums[idx + k] : 0;
            s += v[k];
        }
        int total;
        int pre = block_exclusive_scan(s, ws, total) + carry;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            if (idx + k < ntiles) C.tile_sums[idx + k] = pre;
            pre += v[k];
        }
        carry += total;
    }
}

// Scan phase 3: cell_start of each cell of the tile (cell_start[ncell] = total by the last tile).
__device__ __forceinline__ void scan_apply(const Cells &C, int tile, int *ws) {
    const int idx = tile * blockDim.x * kScanItems + threadIdx.x * kScanItems;
    int v[kScanItems], s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        v[k] = (idx + k < C.ncell) ? C.cell_count[idx + k] : 0;
        s += v[k];
    }
    int total;
    int pre = block_exclusive_scan(s, ws, total) + C.tile_sums[tile];
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        if (idx + k < C.ncell) C.cell_start[idx + k] = pre;
        pre += v[k];
    }
    if (tile == scan_tiles(C) - 1 && threadIdx.x == blockDim.x - 1) C.cell_start[C.ncell] = pre;
}

__device__ __forceinline__ void scatter_atom(const Atoms &A, const Cells &C, int i) {
    A.order[C.cell_start[A.cell_of[i]] + A.slot[i]] = i;
}

// Inside each cell, order the atoms by caller id (deterministic renumbering), one warp per
// cell: the element with key rank q (the number of smaller keys in the cell) goes to slot
// s + q.  Keys are unique, so the ranks are a permutation.  The sorted slots are written to
// A.sorted (A.order is read while ranking); the cell count is reset for the next build.
__device__ __forceinline__ void sort_cell_warp(const Atoms &A, const Cells &C, int c, int lane) {
    const int s = C.cell_start[c], e = C.cell_start[c + 1];
    for (int a = s + lane; a < e; a += 32) {
        const int v = A.order[a];
        const int key = A.id[v];
        int rank = 0;
        for (int b = s; b < e; b++) rank += A.id[A.order[b]] < key ? 1 : 0;
        A.sorted[s + rank] = v;
    }
    if (lane == 0) C.cell_count[c] = 0;
}

// Stencil table of cell group g (one system): the staged slot of the first atom of each of its
// 9 (gx + 2) stencil cells and the total; a group whose neighbourhood exceeds the staging capacity
// sets tile_bad (the passes then take the list path until the next build).
__device__ __forceinline__ void group_table(const Cells &C, int g, Flags *f) {
    const RepCells rg = C.rc[0];
    const int nx = rg.nc[0], ny = rg.nc[1], nz = rg.nc[2];
    const int gxi = g % C.ngx, row = g / C.ngx, y = row % ny, z = row / ny;
    const int x0 = gxi * C.gx, len = min(C.gx, nx - x0);
    int32_t *loc = C.grp_loc + (size_t)g * (C.st_cells + 1);
    int acc = 0, q = 0;
    for (int dz = -1; dz <= 1; dz++) {
        const int zz = (z + dz + nz) % nz;
        for (int dy = -1; dy <= 1; dy++) {
            const int yy = (y + dy + ny) % ny;
            for (int dx = 0; dx < C.gx + 2; dx++, q++) {
                loc[q] = acc;
                if (dx > len + 1) continue;   // a shorter last group: empty slots
                const int xx = (x0 - 1 + dx + nx) % nx;
                const int c = rg.base + (zz * ny + yy) * nx + xx;
                acc += C.cell_start[c + 1] - C.cell_start[c];
            }
        }
    }
    loc[C.st_cells] = acc;
    atomicMax(&f->tile_max, acc);
    if (acc > C.cap) f->tile_bad = 1;
}

__device__ __forceinline__ void gather_atom(const Atoms &A, int k) {
    const int o = A.sorted[k];
    A.pos_tmp[k] = A.pos[o];
    A.vel_tmp[k] = A.vel[o];
    A.force_tmp[k] = A.force[o];
    A.id_tmp[k] = A.id[o];
    A.spec_tmp[k] = A.spec[o];
    if (A.g3) {
        A.g2_tmp[k] = A.g2[o];
        A.g3_tmp[k] = A.g3[o];
    }
}

__device__ __forceinline__ void copyback_atom(const Atoms &A, const Box *boxes, int k) {
    const double4_32a p = A.pos_tmp[k];
    A.pos[k] = p;
    A.ref[k] = p;
    A.vel[k] = A.vel_tmp[k];
    A.force[k] = A.force_tmp[k];
    const int id = A.id_tmp[k], sp = A.spec_tmp[k];
    A.id[k] = id;
    A.spec[k] = sp;
    A.rank[id] = k;
    if (A.g3) {
        A.g2[k] = A.g2_tmp[k];
        A.g3[k] = A.g3_tmp[k];
    }
    // wrapped into the box: p - L floor(p / L), its FP32 rounding, and the floors for place()
    const Box &B = boxes[replica_of(A, k)];
    const double fx = floor(p.x * B.invL[0]), fy = floor(p.y * B.invL[1]), fz = floor(p.z * B.invL[2]);
    const double4_32a q = make_double4_32a(fma(-B.L[0], fx, p.x), fma(-B.L[1], fy, p.y), fma(-B.L[2], fz, p.z), p.w);
    const float4 f = make_float4(eam::f32_rn(q.x), eam::f32_rn(q.y), eam::f32_rn(q.z), __int_as_float(sp));
    A.posf[k] = f;
    A.reff[k] = make_float4(f.x, f.y, f.z, __int_as_float(pack_image(fx, fy, fz)));
    if (A.posd) {
        A.posd[k] = q;
        if (A.posx) store_dfpos(A, k, q, B);
        if (A.posq) store_fixed(A, k, q);
    }
}

// The FP64 pair walk's row order (one warp per atom): the entries j > i first, those the build
// marked as inside r_cut at its FP32 positions (kInsideMark; cin[i] of them) ahead of the others,
// then the entries j < i, each group in its order; cup[i] = the number of entries j > i.  The marks
// are taken off.  The order only steers the walk (its flattened rows take the inside entries first,
// so that lanes rarely idle on a pair beyond r_cut); which entries count is still decided by every
// pass's own FP64 test.  The whole row (k_max <= kPairsKMax) is read into registers before any
// entry is written back.  (With the marks the row's neighbours need not be gathered again: 430 of
// the 1,480 us of a rebuild of fcc Cu 500,000 atoms before.)
constexpr int32_t kInsideMark = (int32_t)0x80000000;
__device__ __forceinline__ void partition_row_warp(const Atoms &A, int i, int lane) {
    const int cnt = min(A.count[i], A.k_max);
    const NbrRow row = nbr_row(A, i);
    int v[kPairsKMax / 32];
    unsigned in = 0;   // bit c: entry 32 c + lane is marked
#pragma unroll
    for (int c = 0; c < kPairsKMax / 32; c++) {
        const int k = 32 * c + lane;
        v[c] = -1;
        if (k < cnt) {
            const int e = *row.ptr(k);
            if (e & kInsideMark) in |= 1u << c;
            v[c] = e & ~kInsideMark;
        }
    }
    __syncwarp();
    const unsigned below = (1u << lane) - 1u;
    int nup = 0, nin = 0;
#pragma unroll
    for (int pass = 0; pass < 2; pass++) {
#pragma unroll
        for (int c = 0; c < kPairsKMax / 32; c++) {
            const bool up = v[c] > i && ((in >> c & 1u) != 0) == (pass == 0);
            const unsigned m = __ballot_sync(0xffffffffu, up);
            if (up) *row.ptr(nup + __popc(m & below)) = v[c];
            nup += __popc(m);
        }
        if (pass == 0) nin = nup;
    }
    int pos = nup;
#pragma unroll
    for (int c = 0; c < kPairsKMax / 32; c++) {
        const bool lo = v[c] >= 0 && v[c] < i;
        const unsigned m = __ballot_sync(0xffffffffu, lo);
        if (lo) *row.ptr(pos + __popc(m & below)) = v[c];
        pos += __popc(m);
    }
    if (lane == 0) {
        A.cup[i] = nup;
        A.cin[i] = nin;
    }
}

// The exact neighbour test: the IEEE operations, order and absence of contraction of the
// definition d = r_j - r_i; d -= L*rint(d*(1/L)); r2 = (dx dx + dy dy) + dz dz.
__device__ __forceinline__ double mi_exact(double d, double L, double invL) {
    return __dsub_rn(d, __dmul_rn(L, rint(__dmul_rn(d, invL))));
}

__device__ __forceinline__ bool within_exact(const double4_32a &pi, const double4_32a &pj, const Box &B,
                                             double rl2) {
    const double dx = mi_exact(__dsub_rn(pj.x, pi.x), B.L[0], B.invL[0]);
    const double dy = mi_exact(__dsub_rn(pj.y, pi.y), B.L[1], B.invL[1]);
    const double dz = mi_exact(__dsub_rn(pj.z, pi.z), B.L[2], B.invL[2]);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return r2 < rl2;
}

// The exact test of a candidate in the FP32 band, kept out of line: it is rare, and inlined it
// would be predicated into every iteration of the candidate loop.
static __device__ __noinline__ bool within_exact_band(const double4_32a *pos, int i, int j, const Box &B,
                                                      double rl2) {
    return within_exact(pos[i], pos[j], B, rl2);
}

// Candidates per iteration of the list build's inner loop (their loads are issued together):
// 4 or 2.  On GB300 4 built the fcc Cu list 10 % faster than 2, and 8 30 % slower than 4.
#ifndef MD_BUILD_UNROLL
#define MD_BUILD_UNROLL 4
#endif
// The cells of the stencil of link cell (cx, cy, cz) of a replica (+-R cells along each edge), in
// (dz, dy, dx) order: fn(js, je, sx, sy, sz, dz, dy, dx) with the cell's slot range and the shift
// by whole box edges that puts a cell across the periodic boundary next to the home cell.
template <typename Fn>
__device__ __forceinline__ void for_stencil(const Cells &C, const RepCells &g, int R, int cx, int cy, int cz,
                                            float Lx, float Ly, float Lz, Fn &&fn) {
    const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2];
    for (int dz = -R; dz <= R; dz++) {
        int z = cz + dz;
        float sz = 0.f;
        if (z < 0) { z += nz; sz = -Lz; }
        if (z >= nz) { z -= nz; sz = Lz; }
        for (int dy = -R; dy <= R; dy++) {
            int y = cy + dy;
            float sy = 0.f;
            if (y < 0) { y += ny; sy = -Ly; }
            if (y >= ny) { y -= ny; sy = Ly; }
            const int rowc = g.base + (z * ny + y) * nx;
            for (int dx = -R; dx <= R; dx++) {
                int x = cx + dx;
                float sx = 0.f;
                if (x < 0) { x += nx; sx = -Lx; }
                if (x >= nx) { x -= nx; sx = Lx; }
                const int cc = rowc + x;
                fn(C.cell_start[cc], C.cell_start[cc + 1], sx, sy, sz, dz, dy, dx);
            }
        }
    }
}

// Full list rows of the atoms of link cell c (§3.2.1: candidates from the cells around it, 27 for
// cells r_list wide, 125 for cells r_list / 2 wide) by a group of G lanes (G = 4, 8, 16 or 32;
// 32 / G cells per warp): lane a of the group takes atoms s + a, s + a + G, ... of the cell.  All
// lanes of the group walk the same neighbour cells and the same candidates in the same order,
// so a candidate is one broadcast load for the group and
// the control flow is uniform inside it.  Candidates are screened with FP32 wrapped coordinates,
// shifted by whole box edges for neighbour cells across the periodic boundary (no rounding to the
// nearest image per candidate).  Only a candidate whose FP32 r^2 lies in [band_lo, band_hi] (a band
// wider than the proven FP32 error) is decided by the exact FP64 test, so each row is the exact
// FP64 set, listed by cell in (dz, dy, dx) order and by ascending slot inside a cell.  Rows are cut
// at k_max (the count is kept).  Returns the longest row of this lane's atoms.  The stencil of
// +-reach cells along each edge needs >= 2 reach + 1 cells per edge (no cell visited twice).
// LOCAL (group walks, one system, reach 1): 1, every entry is also written to the 16-bit local
// list as the slot of the candidate in its cell group's stage (grp_loc of the stencil cell plus
// the candidate's rank inside its cell); 2, only the entries j > i are, as the half row of the
// half walk (lcount of them).  (Builds without local rows: build_slice.)  The global rows
// (A.nbr) are written only when `rows` is set (the counts always): the step kernel's group walks read the
// local rows alone while every group fits its stage.
template <int G, int LOCAL>
__device__ __forceinline__ int build_cell_group(const Atoms &A, const Cells &C, const Box *boxes, int c, int gl,
                                                double rl2, float band_lo, float band_hi, bool rows = true) {
    const int s = C.cell_start[c], e = C.cell_start[c + 1];
    if (s == e) return 0;
    const int r = replica_of(A, s);
    const Box &B = boxes[r];
    const RepCells g = C.rc[r];
    const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2];
    const int local = c - g.base;
    const int cx = local % nx, cy = (local / nx) % ny, cz = local / (nx * ny);
    const float Lx = B.Lf[0], Ly = B.Lf[1], Lz = B.Lf[2];
    const int R = C.reach;
    const int kmax = A.k_max;
    const long long plane = 4LL * A.n;
    const bool edge = cx < R || cx >= nx - R || cy < R || cy >= ny - R || cz < R || cz >= nz - R;
    int longest = 0;
    for (int a0 = s; a0 < e; a0 += G) {
        const int i = a0 + gl;
        const bool act = i < e;
        const int ii = act ? i : s;
        const float4 fi = A.posf[ii];
        int32_t *wp = A.nbr + 4 * (size_t)ii;   // entry cnt of the row (planes of 4 entries)
        uint16_t *lwp = A.lnbr + 4 * (size_t)ii;   // the same entry of the local list
        int cnt = 0, lcnt = 0;
        int lbase = 0;   // staged slot of the first atom of the current candidate cell (local list)
        // one candidate: append j to the row if it is a neighbour
        auto visit = [&](int j, int js, float r2) {
            if (r2 <= band_hi) {
                const bool in = r2 < band_lo || within_exact_band(A.pos, ii, j, B, rl2);
                if (in && act && j != i) {
                    if (cnt < kmax) {
                        if (rows) *wp = j;
                        if constexpr (LOCAL == 1) *lwp = (uint16_t)(lbase + (j - js));
                        if constexpr (LOCAL == 2) {
                            if (j > i) {
                                *lwp = (uint16_t)(lbase + (j - js));
                                lcnt++;
                                lwp += (lcnt & 3) ? 1 : plane - 3;
                            }
                        }
                    }
                    cnt++;
                    const long long adv = (cnt & 3) ? 1 : plane - 3;
                    wp += adv;
                    if constexpr (LOCAL == 1) lwp += adv;
                }
            }
        };
        // cell group of the home cell (group walks): stencil slots of this cell's neighbours
        const int32_t *gloc = nullptr;
        int gx0 = 0;
        if constexpr (LOCAL) {
            const int gxi = cx / C.gx;
            gx0 = gxi * C.gx;
            gloc = C.grp_loc + (size_t)((cz * ny + cy) * C.ngx + gxi) * (C.st_cells + 1);
        }
        for_stencil(C, g, R, cx, cy, cz, Lx, Ly, Lz,
                    [&](int js, int je, float sx, float sy, float sz, int dz, int dy, int dx) {
            if constexpr (LOCAL) lbase = gloc[((dz + 1) * 3 + (dy + 1)) * (C.gx + 2) + (cx - gx0 + dx + 1)];
            const float ox = sx - fi.x, oy = sy - fi.y, oz = sz - fi.z;
            int j = js;
#if MD_BUILD_UNROLL >= 4
            for (; j + 3 < je; j += 4) {
                const float4 f0 = A.posf[j], f1 = A.posf[j + 1], f2 = A.posf[j + 2], f3 = A.posf[j + 3];
                const float ax = f0.x + ox, ay = f0.y + oy, az = f0.z + oz;
                const float bx = f1.x + ox, by = f1.y + oy, bz = f1.z + oz;
                const float cx2 = f2.x + ox, cy2 = f2.y + oy, cz2 = f2.z + oz;
                const float dx2 = f3.x + ox, dy2 = f3.y + oy, dz2 = f3.z + oz;
                const float r0 = fmaf(ax, ax, fmaf(ay, ay, az * az));
                const float r1 = fmaf(bx, bx, fmaf(by, by, bz * bz));
                const float rr2 = fmaf(cx2, cx2, fmaf(cy2, cy2, cz2 * cz2));
                const float rr3 = fmaf(dx2, dx2, fmaf(dy2, dy2, dz2 * dz2));
                visit(j, js, r0);
                visit(j + 1, js, r1);
                visit(j + 2, js, rr2);
                visit(j + 3, js, rr3);
            }
#endif
            for (; j + 1 < je; j += 2) {
                const float4 f0 = A.posf[j], f1 = A.posf[j + 1];
                const float ax = f0.x + ox, ay = f0.y + oy, az = f0.z + oz;
                const float bx = f1.x + ox, by = f1.y + oy, bz = f1.z + oz;
                const float r0 = fmaf(ax, ax, fmaf(ay, ay, az * az));
                const float r1 = fmaf(bx, bx, fmaf(by, by, bz * bz));
                visit(j, js, r0);
                visit(j + 1, js, r1);
            }
            if (j < je) {
                const float4 f0 = A.posf[j];
                const float ax = f0.x + ox, ay = f0.y + oy, az = f0.z + oz;
                visit(j, js, fmaf(ax, ax, fmaf(ay, ay, az * az)));
            }
        });
        if (act) {
            A.count[i] = cnt;
            A.wrap[i] = edge ? 1 : 0;
            if constexpr (LOCAL == 2) A.lcount[i] = lcnt;
            if (cnt > kmax) atomicOr(&A.flags->error, FLAG_OVERFLOW);
            longest = max(longest, cnt);
        }
    }
    return longest;
}

// Full list rows of a slice of the atoms of link cell c by one warp: atoms s + slice, s + slice + S, ...
// of the cell's range (S slices per cell; list walks, no local rows).  The candidates, the atoms of
// the (2 reach + 1)^3 cells around c in (dz, dy, dx) order, are numbered through, and the lanes take 32
// consecutive ones at a time, empty cells and cell boundaries costing no lane; every home atom of
// the slice then tests the 32 at once, and a ballot places the accepted ones behind each other in
// candidate order, so that the rows are the exact FP64 set in the same order as build_cell_group's.
// A lane per home atom (build_cell_group) appended candidate by candidate with most lanes idle,
// and the appends' address chain bounded it.  Per rebuild, list phase, before -> after (us): 32 bcc
// Fe replicas of 623,572 atoms 473 -> 350, Fe-C 250,250 221 -> 129, bcc Fe 2,000 65 -> 29, fcc Cu
// 500,000 994 -> 984 (57 instructions per home atom and 32 candidates; issue slots 75 % busy).  With the
// candidates' shifted positions formed once, two homes at a time in packed FP32 arithmetic and the band
// looked at only where a candidate was accepted, the issue slots bound it less: a 20-step call of
// fcc Cu 500,000 mixed 12.55 -> 11.92 ms, its rebuilds 202 -> 169 us a step at FP64; the 32 replicas
// 3.39 -> 3.20 ms.  (Cells r_list / 2 wide, 42 % fewer candidates: 165 us a step, and slower passes.)
// MARK: entries inside r_cut (FP32) get kInsideMark, for partition_row_warp.
template <bool MARK>
__device__ __forceinline__ int build_slice(const Atoms &A, const Cells &C, const Box *boxes, int c, int slice, int S,
                                           int lane, double rl2, float band_lo, float band_hi) {
    const int s = C.cell_start[c] + slice, e = C.cell_start[c + 1];
    if (s >= e) return 0;
    const int r = replica_of(A, s);
    const Box &B = boxes[r];
    const RepCells g = C.rc[r];
    const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2];
    const int local = c - g.base;
    const int cx = local % nx, cy = (local / nx) % ny, cz = local / (nx * ny);
    const int R = C.reach, W = 2 * R + 1, nst = W * W * W;
    const int kmax = A.k_max;
    const bool edge = cx < R || cx >= nx - R || cy < R || cy >= ny - R || cz < R || cz >= nz - R;
    const unsigned full = 0xffffffffu, below = (1u << lane) - 1u;
    const int homes = (e - s + S - 1) / S;
    const unsigned row4 = 4u * (unsigned)A.n;
    constexpr float kFar = 1e18f;   // an x further from every atom than any list reaches
    int longest = 0;
    for (int h0 = 0; h0 < homes; h0 += 32) {
        const int nh = min(32, homes - h0);
        const int mine = s + S * (h0 + min(lane, nh - 1));   // this lane's home atom
        const float4 fp = A.posf[mine];
        const float hx = lane < nh ? -fp.x : kFar, hy = -fp.y, hz = -fp.z;
        int cnt = 0;
        for (int q0 = 0; q0 < nst; q0 += 32) {   // (one round for reach 1)
            // this lane's stencil cell: its first atom, length and shift by whole box edges
            const int q = q0 + lane;
            int first = 0, len = 0;
            float sx = 0.f, sy = 0.f, sz = 0.f;
            if (q < nst) {
                int x = cx + q % W - R, y = cy + (q / W) % W - R, z = cz + q / (W * W) - R;
                if (x < 0) { x += nx; sx = -B.Lf[0]; }
                if (x >= nx) { x -= nx; sx = B.Lf[0]; }
                if (y < 0) { y += ny; sy = -B.Lf[1]; }
                if (y >= ny) { y -= ny; sy = B.Lf[1]; }
                if (z < 0) { z += nz; sz = -B.Lf[2]; }
                if (z >= nz) { z -= nz; sz = B.Lf[2]; }
                const int cc = g.base + (z * ny + y) * nx + x;
                first = C.cell_start[cc];
                len = C.cell_start[cc + 1] - first;
            }
            // the non-empty cells moved to the first lanes (lane t: the t-th set bit of ne)
            const unsigned ne = __ballot_sync(full, len > 0);
            const int nne = __popc(ne);
            int src = 0;
#pragma unroll
            for (int b = 16; b > 0; b >>= 1)
                if (__popc(ne & ((1u << (src + b)) - 1u)) <= lane) src += b;
            first = __shfl_sync(full, first, src & 31);
            len = __shfl_sync(full, len, src & 31);
            sx = __shfl_sync(full, sx, src & 31);
            sy = __shfl_sync(full, sy, src & 31);
            sz = __shfl_sync(full, sz, src & 31);
            if (lane >= nne) len = 0;
            int off = len;   // candidates before this lane's cell
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(full, off, o);
                if (lane >= o) off += y;
            }
            const int total = __shfl_sync(full, off, 31);
            off -= len;
            for (int p0 = 0; p0 < total; p0 += 32) {
                // candidate p0 + lane: the cell it lies in, its slot and shifted position
                const bool cell = lane < nne;
                const int base = __popc(__ballot_sync(full, cell && off <= p0)) - 1;
                const unsigned starts =
                    __reduce_or_sync(full, cell && off > p0 && off < p0 + 32 ? 1u << (off - p0) : 0u);
                const int t = base + __popc(starts & (below | (1u << lane)));
                const int j = __shfl_sync(full, first, t) + p0 + lane - __shfl_sync(full, off, t);
                const float ox = __shfl_sync(full, sx, t), oy = __shfl_sync(full, sy, t), oz = __shfl_sync(full, sz, t);
                float x = kFar, y = 0.f, z = 0.f;
                if (p0 + lane < total) {
                    const float4 f = A.posf[j];
                    x = f.x + ox;
                    y = f.y + oy;
                    z = f.z + oz;
                }
                auto append = [&](float r2, int a) {
                    const int i = s + S * (h0 + a);
                    bool in = r2 <= band_hi && j != i;
                    unsigned m = __ballot_sync(full, in);
                    if (m == 0u) return;
                    if (__any_sync(full, in && r2 >= band_lo)) {   // the band: the exact test decides
                        if (in && r2 >= band_lo) in = within_exact_band(A.pos, i, j, B, rl2);
                        m = __ballot_sync(full, in);
                    }
                    const int k = __shfl_sync(full, cnt, a) + __popc(m & below);
                    if (in && k < kmax)
                        A.nbr[4 * (size_t)i + (unsigned long long)(unsigned)(k >> 2) * row4 + (k & 3)] =
                            MARK && r2 < A.pair_rc2f ? j | kInsideMark : j;
                    if (lane == a) cnt += __popc(m);
                };
                for (int a = 0; a < nh; a += 2) {   // two home atoms at a time (an odd last one: kFar)
                    auto less = [&](float c, float h) {   // c + the two homes' negated coordinates
                        return pk::add2(pk::pack(c, c),
                                        pk::pack(__shfl_sync(full, h, a), __shfl_sync(full, h, a + 1)));
                    };
                    const pk::F2 dx = less(x, hx), dy = less(y, hy), dz = less(z, hz);
                    float r0, r1;
                    pk::unpack(pk::fma2(dx, dx, pk::fma2(dy, dy, pk::mul2(dz, dz))), r0, r1);
                    append(r0, a);
                    append(r1, a + 1);
                }
            }
        }
        if (lane < nh) {
            A.count[mine] = cnt;
            A.wrap[mine] = edge ? 1 : 0;
            if (cnt > kmax) atomicOr(&A.flags->error, FLAG_OVERFLOW);
            longest = max(longest, cnt);
        }
    }
    return longest;
}

// Slices per link cell: enough that every warp of the launch has one, at most a home atom each.
__host__ __device__ inline int list_slices(long long ncell, long long nwarps) {
    const long long q = ncell > 0 ? nwarps / ncell : 1;
    return (int)(q < 1 ? 1 : (q > 32 ? 32 : q));
}

// The list phase over all cells and slices.
template <bool MARK>
__device__ __forceinline__ int build_slices(const Atoms &A, const Cells &C, const Box *boxes, long long warp,
                                            long long nwarps, int lane, double rl2, float band_lo, float band_hi) {
    const int S = list_slices(C.ncell, nwarps);
    int m = 0;
    for (long long q = warp; q < (long long)C.ncell * S; q += nwarps)
        m = max(m, build_slice<MARK>(A, C, boxes, (int)(q / S), (int)(q % S), S, lane, rl2, band_lo, band_hi));
    return m;
}

// The list phase over all cells: warp w of nwarps takes cell groups w, w + nwarps, ...; every
// lane returns the longest row it built (all 32 lanes of a warp take part in every iteration).
template <int G, int LOCAL>
__device__ __forceinline__ int build_cells(const Atoms &A, const Cells &C, const Box *boxes, long long warp,
                                           long long nwarps, int lane, double rl2, float band_lo, float band_hi,
                                           bool rows = true) {
    constexpr int CPW = 32 / G;   // cells per warp
    int m = 0;
    for (long long c0 = warp * CPW; c0 < C.ncell; c0 += nwarps * CPW) {
        const long long c = c0 + lane / G;
        if (c < C.ncell)
            m = max(m, build_cell_group<G, LOCAL>(A, C, boxes, (int)c, lane & (G - 1), rl2, band_lo, band_hi, rows));
    }
    return m;
}

template <int LOCAL>
__device__ __forceinline__ int build_cells_any(int G, const Atoms &A, const Cells &C, const Box *boxes, long long warp,
                                               long long nwarps, int lane, double rl2, float band_lo, float band_hi,
                                               bool rows = true) {
    if (G == 4) return build_cells<4, LOCAL>(A, C, boxes, warp, nwarps, lane, rl2, band_lo, band_hi, rows);
    if (G == 8) return build_cells<8, LOCAL>(A, C, boxes, warp, nwarps, lane, rl2, band_lo, band_hi, rows);
    if (G == 16) return build_cells<16, LOCAL>(A, C, boxes, warp, nwarps, lane, rl2, band_lo, band_hi, rows);
    return build_cells<32, LOCAL>(A, C, boxes, warp, nwarps, lane, rl2, band_lo, band_hi, rows);
}

}  // namespace ph
}  // namespace mdk
