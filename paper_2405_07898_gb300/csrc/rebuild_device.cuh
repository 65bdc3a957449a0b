// rebuild_device.cuh -- per-element device functions of the list rebuild,
// the opening kick and the energy reduction.  The kernels of rebuild.cu launch
// them one element per thread; the persistent step kernel (persistent.cu)
// runs them in grid-stride loops between grid barriers.  Every function takes
// the buffer set `s` and the record buffer `sp` explicitly.
#pragma once

#include "device_common.cuh"

namespace eammd {
namespace {

// Atom i of the caller's arrays (xyz interleaved; vel may be null) into buffer
// set s, in the caller's order.
template <class R>
__device__ __forceinline__ void load_atom(const Bufs<R> &B, int s, const double *pos, const double *vel, const int *types,
                                          int i)
{
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double x = pos[3 * (size_t)i + a];
        const double v = vel ? vel[3 * (size_t)i + a] : 0.0;
        finite = finite && isfinite(x) && isfinite(v);
        B.xr[s][a][i] = x;
        B.d[a][i] = 0.0;
        B.v[s][a][i] = v;
    }
    if (!finite) atomicOr(&B.st->error, ERR_NONFINITE);
    B.id[s][i] = i;
    B.type[s][i] = types[i];
}

// x as a float truncated toward zero, from its bits by integer operations
// (the FP64 pipe of this GPU is narrow): 0 below 2^-126, +-inf above the
// float range.
__device__ __forceinline__ float trunc_to_float(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (e < 897u) return 0.f;
    if (e > 1150u) return __uint_as_float((hi & 0x80000000u) | 0x7f800000u);
    return __uint_as_float((hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

// The rare FP64 paths of bin_atom, out of line: inlined, the compiler computes
// them for every atom and selects, and the FP64 pipe (72 % busy) bounds the
// pass.
__device__ __noinline__ double wrap_image(double x, double L)
{
    return __dsub_rn(x, __dmul_rn(L, floor(__ddiv_rn(x, L))));
}
__device__ __noinline__ int cell_index_exact(double x, double inv, int n)
{
    return (int)fmax(fmin(floor(__dmul_rn(x, inv)), (double)(n - 1)), 0.0);
}

// Cell index floor(RN(x inv)) clamped to [0, n - 1], for finite x.  The FP32
// product of the truncated x and the rounded inv is within 2^-21.8 |q| of the
// FP64 product (truncation 2^-23, two roundings 2^-24 each); where it lies
// farther than 2^-20 max(|q|, 1) from every integer both have the same floor,
// elsewhere the FP64 product decides.
__device__ __forceinline__ int cell_index(double x, double inv, float inv_f, int n)
{
    const float q32 = trunc_to_float(x) * inv_f;
    const float f = floorf(q32), frac = q32 - f;
    const float tol = 0x1p-20f * fmaxf(fabsf(q32), 1.0f);
    if (frac > tol && frac < 1.0f - tol) return min(max((int)f, 0), n - 1);
    return cell_index_exact(x, inv, n);
}

// Slot of an atom in its cell (arrival order): one atomic per distinct cell
// among the warp's active lanes (atoms in cell order mostly share cells); the
// lanes of a cell take consecutive slots from it in lane order.
__device__ __forceinline__ int cell_slot(int *count, int cell)
{
    const unsigned peers = __match_any_sync(__activemask(), cell);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(&count[cell], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + __popc(peers & ((1u << lane) - 1u));
}

// Periodic image of x = xr + d on periodic axes: kept when already in
// [0, L), else x - L floor(x / L); then bin: c_d = floor(x_d n_d/L_d) clamped
// to [0, n_d - 1].  The box test compares bit patterns (non-negative doubles
// order as their bits; -0 is inside).  The slot inside the cell is the
// arrival order (permute_atom puts the cell's atoms in the order of their ids).
template <class R>
__device__ __forceinline__ void bin_atom(const Bufs<R> &B, const Geom &G, int s, int i)
{
    int c[3];
    bool finite = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double L = G.box[a];
        double x = __dadd_rn(B.xr[s][a][i], B.d[a][i]);
        const long long xb = __double_as_longlong(x);
        const bool inside = (xb >= 0 && xb < __double_as_longlong(L)) || xb == (long long)0x8000000000000000ull;
        if (!((G.open_mask >> a) & 1) && !inside) {
            // (open axis: not wrapped; outside the box, the edge cell takes it)
            x = wrap_image(x, L);
        }
        finite = finite && ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff;
        B.xw[a][i] = x;
        c[a] = finite ? cell_index(x, G.inv_cell[a], G.inv_cell_f[a], G.ncell[a]) : 0;
    }
    if (!finite) atomicOr(&B.st->error, ERR_NONFINITE);
    int cell = (c[2] * G.ncell[1] + c[1]) * G.ncell[0] + c[0];
    B.cell_old[i] = cell;
    B.slot[i] = cell_slot(B.count, cell);
}

// Sum over the block of one int per thread; every thread returns it.  All
// threads must call (blockDim a multiple of 32).
__device__ __forceinline__ int block_sum_i(int v)
{
    __shared__ int sm[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    int t = (lane < nw) ? sm[lane] : 0;
    t = __reduce_add_sync(0xffffffffu, t);
    __syncthreads();
    return t;
}

// Cells [base, end) of the exclusive scan cell_start[c] = sum_{c' < c}
// count[c'], given prefix = cell_start[base], by one block in tiles of
// blockDim cells (at most 1024); the last part also writes
// cell_start[ncells].
__device__ __forceinline__ void scan_tiles(const int *count, int *cell_start, int base, int end, int ncells, int prefix)
{
    __shared__ int wt[33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    for (int t0 = base; t0 < end; t0 += blockDim.x) {
        const int c = t0 + threadIdx.x;
        const int v = (c < end) ? count[c] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wt[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int w = (lane < nw) ? wt[lane] : 0;
            int wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            wt[lane] = wi - w;  // exclusive prefix of the warp totals
            if (lane == 31) wt[32] = wi;
        }
        __syncthreads();
        if (c < end) {
            const int excl = prefix + wt[warp] + incl - v;
            cell_start[c] = excl;
            if (c == ncells - 1) cell_start[ncells] = excl + v;
        }
        prefix += wt[32];
        __syncthreads();
    }
}

// Part `part` of `nparts` of the scan, by one block on its own: it adds up the
// counts before its part and scans its part, so the parts need no second
// pass and no barrier between them.  The blocks together read the counts
// nparts/2 times, from L2.  The counts stay; the permutation zeroes them.
__device__ __forceinline__ void scan_part(const int *count, int *cell_start, int ncells, int part, int nparts)
{
    const int per = ((ncells + nparts - 1) / nparts + 31) & ~31;
    const int base = min(part * per, ncells), end = min(base + per, ncells);
    int v = 0;
    for (int c = threadIdx.x; c < base; c += blockDim.x) v += count[c];
    const int prefix = block_sum_i(v);
    if (base < end) scan_tiles(count, cell_start, base, end, ncells, prefix);
}

// Atom i to its arrival slot in its cell, with its original id.
template <class R>
__device__ __forceinline__ void scatter_atom(const Bufs<R> &B, int s, int i)
{
    const int q = B.cell_start[B.cell_old[i]] + B.slot[i];
    B.cell_atoms[q] = i;
    B.cell_ids[q] = B.id[s][i];
}

// The state of the atom in arrival slot q to its place in the other buffer
// set: atoms in cell order, ascending original id inside a cell.  The place
// is the number of smaller ids in the cell (a handful of consecutive words),
// so no pass sorts the cells first.  Positions become the wrapped positions,
// displacements restart at zero, and the cell-centred coordinates uref (and
// record buffer sp) are formed in FP64 and rounded.  s: the buffer set read.
template <class R>
__device__ __forceinline__ void permute_atom(const Bufs<R> &B, const Geom &G, int s, int sp, int q)
{
    const int t = 1 - s;
    const int i = B.cell_atoms[q];
    const int id = B.cell_ids[q];
    const int cell = B.cell_old[i];
    const int lo = B.cell_start[cell], hi = B.cell_start[cell + 1];
    int p = lo;
    for (int r = lo; r < hi; ++r) p += B.cell_ids[r] < id ? 1 : 0;
    const int cc[3] = {cell % G.ncell[0], (cell / G.ncell[0]) % G.ncell[1], cell / (G.ncell[0] * G.ncell[1])};
    R u[3];
    double X0 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double X = B.xw[a][i];
        if (a == 0) X0 = X;
        B.xr[t][a][p] = X;
        u[a] = (R)__dsub_rn(X, B.center[a][cc[a]]);
        B.uref[a][p] = u[a];
        B.v[t][a][p] = B.v[s][a][i];
        B.d[a][p] = 0.0;
    }
    B.shadow[sp][p] = mk4<R>(u[0], u[1], u[2], (R)0);
    B.screen[0][p] = (float)X0;
    if constexpr (sizeof(R) == 8) {
        B.rec32[sp][p] = make_float4((float)u[0], (float)u[1], (float)u[2], 0.f);
        B.screen[1][p] = (float)u[1];
        B.screen[2][p] = (float)u[2];
    }
    B.id[t][p] = id;
    const int ty = B.type[s][i];
    B.type[t][p] = ty;
    B.type8[p] = (uint8_t)ty;
    B.cell[p] = cell;
}

// Exact list test for a candidate near the list radius: the minimum-image
// squared distance with the operations and rounding order of the definition
// (d = x_j - x_i, +-L once on periodic axes, (dx^2 + dy^2) + dz^2, no fused
// operations).
__device__ __forceinline__ bool exact_in_list(const double *const xr[3], int p, int q, const Geom &G)
{
    double d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double x = __dsub_rn(xr[a][q], xr[a][p]);
        if (!((G.open_mask >> a) & 1)) {
            if (x > G.half_box[a]) x = __dsub_rn(x, G.box[a]);
            else if (x < -G.half_box[a]) x = __dadd_rn(x, G.box[a]);
        }
        d[a] = x;
    }
    double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
    return r2 < G.rl2;
}

// Whether the pair vector d = x_q - x_p (minimum image) lies in the upper
// half space: d_z > 0, or d_z = 0 and d_y > 0, or d_z = d_y = 0 and d_x > 0.
// dz is the FP32 component of the screen; where it is clearly
// away from zero (far beyond its rounding error) it decides, elsewhere the
// FP64 components of the definition do.  FP64 subtraction and the image
// shift are exactly antisymmetric, so the answers for (p, q) and (q, p) are
// complements: a pair is kept by exactly one of its atoms.
__device__ __forceinline__ bool upper_half(float dz, const double *const xr[3], int p, int q,
                                           const Geom &G)
{
    const float tol = 1e-4f;
    if (dz > tol) return true;
    if (dz < -tol) return false;
    double d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double x = __dsub_rn(xr[a][q], xr[a][p]);
        if (!((G.open_mask >> a) & 1)) {
            if (x > G.half_box[a]) x = __dsub_rn(x, G.box[a]);
            else if (x < -G.half_box[a]) x = __dadd_rn(x, G.box[a]);
        }
        d[a] = x;
    }
    if (d[2] != 0.0) return d[2] > 0.0;
    if (d[1] != 0.0) return d[1] > 0.0;
    return d[0] > 0.0;
}

// What the list build screens candidates with, in FP32: the coordinate x
// itself (the same origin for all cells of a row), and y and z relative to the
// cell's centre.  kScreenPad words after the arrays may be read and are ignored.
struct Screen {
    const float *x, *y, *z;
};
__device__ __forceinline__ Screen screen_of(const Bufs<float> &B) { return {B.screen[0], B.uref[1], B.uref[2]}; }
__device__ __forceinline__ Screen screen_of(const Bufs<double> &B) { return {B.screen[0], B.screen[1], B.screen[2]}; }

// Two FP32 operations in one instruction.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_get(F2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.v)); }
__device__ __forceinline__ F2 f2_add(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// Half-width of the band around r_list^2 inside which FP32 does not decide,
// for the atom at (x, y, z) of the screen.  With s the sum of the coordinates'
// sizes (a partner in the list is at most r_list farther out; an image shift
// adds the box edge), the pair vector is rounded by at most d = 3 s 2^-24, and
// r^2 by 2 r d + d^2; the band is 1.7 times that, and 16 r_list^2 2^-24 for the
// sum of squares.  An atom far beyond an open edge has a wide band, so its list
// stays exact (up to 1e24 Angstrom, where the band overflows).  x has one
// origin for the whole box, so the band also grows with the box's x edge (about
// 0.2 exact tests an atom at 10,000 Angstrom, 2 at 100,000): the price of a row
// of cells in one run.
__device__ __forceinline__ float screen_margin(const Geom &G, float x, float y, float z)
{
    const float rl = sqrtf(G.rl2_f);
    const float ex = fabsf(x) + G.box_f[0] + 2.f * rl;
    const float ey = fabsf(y) + 2.f * G.h_f[1] + 2.f * rl, ez = fabsf(z) + 2.f * G.h_f[2] + 2.f * rl;
    const float s = 0x1p-24f * (ex + ey + ez);
    return s * (10.f * rl + 16.f * s) + 0x1p-20f * G.rl2_f;
}

// Verlet list of atom p: the atoms of the 27 surrounding cells (in stencil
// order, ascending id inside a cell; cells beyond an open edge do not exist)
// closer than r_list.  The test runs in FP32, in the FP64 path too (FP64 tests
// of the ~173 candidates took 2,430 us of a 799,496-atom build); candidates
// within the rounding margin of r_list are decided by exact_in_list, so the
// list is bit-identical to the FP64 definition.
//
// The build is bound by instruction issue, so the candidates cost as few
// instructions as they can:
//   - the three cells of a stencil row are consecutive atoms, tested as one
//     run (two at a periodic edge) with one offset, since x has one origin;
//   - runs are read in aligned groups of four from arrays per coordinate, two
//     candidates an instruction (slots outside the run are masked away);
//   - a test is a subtraction whose sign bit is shifted into a mask, one for
//     either side of the margin, so no lane branches on a hit; the few hits
//     are appended afterwards, one an iteration.
// A branch per candidate is taken by some lane nearly every time, and cells
// on their own leave lanes waiting for the fullest cell in the warp.  A
// rebuild of 799,496 BCC atoms takes 228 us (331 before), of the 801,792-atom
// FCC slab 307 us (508), of the BCC atoms in the FP64 path 234 us (2,552).
// Also measured: a warp per cell with its stencil's candidates over the lanes
// and ballots as hit masks, 381 us (barriers and idle lanes in the appends).
// Returns the neighbour count (the list keeps at most cap of them; more
// raises ERR_LIST_OVERFLOW).  half: keep each pair once, in the same order:
// only the neighbours q whose pair vector x_q - x_p lies in the upper half
// space (upper_half).  Every atom's neighbourhood is close to centrally
// symmetric, so each lists about half its neighbours.
//
// `xr`: exact positions, `cell_of`: the atoms' cells, lp: column 0 of atom p.
__device__ __forceinline__ int list_walk(const Geom &G, const Screen &sc, const double *const (&xr)[3],
                                         const int *cell_of, const int *cell_start, int p, uint32_t *lp, int ld, int cap,
                                         bool half)
{
    int cnt = 0;
    const int nx = G.ncell[0], ny = G.ncell[1], nz = G.ncell[2];
    const int cell = cell_of[p];
    const int cx = cell % nx, cy = (cell / nx) % ny, cz = cell / (nx * ny);
    const float px = sc.x[p], py = sc.y[p], pz = sc.z[p];
    const float margin = screen_margin(G, px, py, pz);
    const F2 hi = f2(-(G.rl2_f + margin), -(G.rl2_f + margin)), band = f2(2.f * margin, 2.f * margin);
    const bool open_x = G.open_mask & 1, open_y = (G.open_mask >> 1) & 1, open_z = (G.open_mask >> 2) & 1;
#pragma unroll 1
    for (int row = 0; row < 9; ++row) {
        const int dz = row / 3 - 1, dy = row % 3 - 1;
        int ez = cz + dz, ey = cy + dy;
        if (ez < 0 || ez >= nz) {
            if (open_z) continue;  // no cell beyond an open edge
            ez += (ez < 0) ? nz : -nz;
        }
        if (ey < 0 || ey >= ny) {
            if (open_y) continue;
            ey += (ey < 0) ? ny : -ny;
        }
        const int *cs = cell_start + (ez * ny + ey) * nx;
        const float oy = (float)dy * G.h_f[1] - py, oz = (float)dz * G.h_f[2] - pz;
        const F2 oy2 = f2(oy, oy), oz2 = f2(oz, oz);
        // cells cx - 1, cx, cx + 1: one run of atoms, with the parts beyond an
        // edge apart (-1: the last cell, first; 1: the first cell, last)
        const int c1 = cs[cx], c2 = cs[cx + 1];
        const uint32_t code = list_entry(0u, -1, dy, dz);
#pragma unroll 1
        for (int part = (cx == 0 ? -1 : 0); part <= (cx == nx - 1 ? 1 : 0); ++part) {
            int r0, r1;          // the run
            float image = 0.f;
            if (part == 0) {
                r0 = cx == 0 ? c1 : cs[cx - 1];
                r1 = cx == nx - 1 ? c2 : cs[cx + 2];
            } else {
                if (open_x) continue;
                r0 = cs[part < 0 ? nx - 1 : 0];
                r1 = cs[part < 0 ? nx : 1];
                image = part < 0 ? -G.box_f[0] : G.box_f[0];
            }
            // dx + 1 of atom q of the run is (q >= b1) + (q >= b2)
            const int b1 = part == 0 ? c1 : (part < 0 ? 0x7fffffff : 0), b2 = part == 0 ? c2 : b1;
            const float ox = image - px;
            const F2 ox2 = f2(ox, ox);
            for (int a = r0 & ~3; a < r1; a += 32) {  // a multiple of four, as the arrays are aligned
                unsigned in = 0u, near = 0u;  // sign bits of r2 - hi, r2 - lo; the first slot ends highest
                const int m = min((r1 - a + 3) & ~3, 32);
                for (int k = 0; k < m; k += 4) {
                    const float4 X = *reinterpret_cast<const float4 *>(sc.x + a + k);
                    const float4 Y = *reinterpret_cast<const float4 *>(sc.y + a + k);
                    const float4 Z = *reinterpret_cast<const float4 *>(sc.z + a + k);
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        const F2 ax = f2_add(g ? f2(X.z, X.w) : f2(X.x, X.y), ox2);
                        const F2 ay = f2_add(g ? f2(Y.z, Y.w) : f2(Y.x, Y.y), oy2);
                        const F2 az = f2_add(g ? f2(Z.z, Z.w) : f2(Z.x, Z.y), oz2);
                        const F2 u = f2_fma(az, az, f2_fma(ay, ay, f2_fma(ax, ax, hi)));  // r2 - hi
                        float u0, u1, v0, v1;
                        f2_get(u, u0, u1);
                        f2_get(f2_add(u, band), v0, v1);  // r2 - lo
                        in = __funnelshift_l(__float_as_uint(u0), in, 1);
                        in = __funnelshift_l(__float_as_uint(u1), in, 1);
                        near = __funnelshift_l(__float_as_uint(v0), near, 1);
                        near = __funnelshift_l(__float_as_uint(v1), near, 1);
                    }
                }
                in <<= 32 - m;
                near <<= 32 - m;
                // slots before and after the run, and the atom itself
                if (a < r0) in &= 0xffffffffu >> (r0 - a);
                if (r1 - a < 32) in &= ~(0xffffffffu >> (r1 - a));
                if ((unsigned)(p - a) < 32u) in &= ~(0x80000000u >> (p - a));
                for (unsigned unsure = in & ~near; unsure;) {  // rare
                    const int k = __clz((int)unsure);
                    const unsigned bit = 0x80000000u >> k;
                    unsure &= ~bit;
                    if (!exact_in_list(xr, p, a + k, G)) in &= ~bit;
                }
                if (half) {
                    for (unsigned m2 = in; m2;) {
                        const int k = __clz((int)m2);
                        const unsigned bit = 0x80000000u >> k;
                        m2 &= ~bit;
                        if (!upper_half(sc.z[a + k] + oz, xr, p, a + k, G)) in &= ~bit;
                    }
                }
                while (in) {
                    const int k = __clz((int)in);
                    const int q = a + k;
                    in &= 0x7fffffffu >> k;
                    const uint32_t e = code + (uint32_t)q + ((q >= b1 ? 1u : 0u) + (q >= b2 ? 1u : 0u) << kCodeShift);
                    if (cnt < cap) *lp = e;
                    lp += ld;
                    ++cnt;
                }
            }
        }
    }
    return cnt;
}

template <class R>
__device__ __forceinline__ int list_atom(const Bufs<R> &B, const Geom &G, int s, int p, int ld, int cap,
                                         bool half = false)
{
    const double *const xr[3] = {B.xr[s][0], B.xr[s][1], B.xr[s][2]};
    const int cnt = list_walk(G, screen_of(B), xr, B.cell, B.cell_start, p, B.list + p, ld, cap, half);
    B.nnb[p] = min(cnt, cap);
    if (cnt > cap) atomicOr(&B.st->error, ERR_LIST_OVERFLOW);
    return cnt;
}

// Stencil cell of lane c < 27 around cell (cx, cy, cz): c = 9 (dz + 1) +
// 3 (dy + 1) + (dx + 1), the stencil order.  Its atoms are [q0, q1), empty for
// the other lanes and beyond an open edge.
__device__ __forceinline__ void stencil_cell(const Geom &G, const int *cell_start, int lane, int cx, int cy, int cz,
                                             int &dx, int &dy, int &dz, int &q0, int &q1)
{
    const int nx = G.ncell[0], ny = G.ncell[1], nz = G.ncell[2];
    dz = lane / 9 - 1;
    dy = (lane / 3) % 3 - 1;
    dx = lane % 3 - 1;
    int ex = cx + dx, ey = cy + dy, ez = cz + dz;
    bool valid = lane < 27;
    if (ex < 0 || ex >= nx) {
        if (G.open_mask & 1) valid = false;
        else ex += (ex < 0) ? nx : -nx;
    }
    if (ey < 0 || ey >= ny) {
        if ((G.open_mask >> 1) & 1) valid = false;
        else ey += (ey < 0) ? ny : -ny;
    }
    if (ez < 0 || ez >= nz) {
        if ((G.open_mask >> 2) & 1) valid = false;
        else ez += (ez < 0) ? nz : -nz;
    }
    q0 = q1 = 0;
    if (valid) {
        const int e = (ez * ny + ey) * nx + ex;
        q0 = cell_start[e];
        q1 = cell_start[e + 1];
    }
}

// list_atom with the 32 lanes of a warp on atom p: lane c < 27 walks
// stencil cell c = 9 (dz + 1) + 3 (dy + 1) + (dx + 1) -- the stencil order --
// issuing its candidates' record loads four at a time, and an exclusive warp
// prefix sum of the cells' hit counts gives each cell its place in the list,
// so the list is the one list_atom writes, entry for entry.  The walk per
// atom is a few rounds of independent loads (the cells in parallel) instead
// of a chain of ~27: for systems of a few thousand atoms, whose records were
// just written by other SMs, the chain's L2 round trips are the cost of the
// build.  A cell's decisions are kept as a bit mask for its first 64
// candidates and recomputed beyond them.  All 32 lanes must call; every lane
// returns the count.
template <class R>
__device__ __forceinline__ int list_atom_warp(const Bufs<R> &B, const Geom &G, int s, int p, int ld,
                                              int cap)
{
    constexpr int UQ = 4;  // candidate loads in flight per lane
    const int lane = (int)(threadIdx.x & 31u);
    const double *const xr[3] = {B.xr[s][0], B.xr[s][1], B.xr[s][2]};
    const Screen sc = screen_of(B);
    const int nx = G.ncell[0], ny = G.ncell[1];
    const int cell = B.cell[p];
    const int cx = cell % nx, cy = (cell / nx) % ny, cz = cell / (nx * ny);
    const float px = sc.x[p], py = sc.y[p], pz = sc.z[p];
    const float margin = screen_margin(G, px, py, pz);
    const float lo = G.rl2_f - margin, hi = G.rl2_f + margin;
    int dx, dy, dz, q0, q1;
    stencil_cell(G, B.cell_start, lane, cx, cy, cz, dx, dy, dz, q0, q1);
    // x has one origin for all cells: only an image needs a shift
    const float ox = (cx + dx < 0 ? -G.box_f[0] : (cx + dx >= G.ncell[0] ? G.box_f[0] : 0.f)) - px;
    const float oy = (float)dy * G.h_f[1] - py, oz = (float)dz * G.h_f[2] - pz;
    auto in_list = [&](float x, float y, float z, int q) -> bool {
        const float ddx = x + ox, ddy = y + oy, ddz = z + oz;
        const float r2 = fmaf(ddz, ddz, fmaf(ddy, ddy, ddx * ddx));
        return !(r2 > hi || q == p) && (r2 < lo || exact_in_list(xr, p, q, G));
    };
    unsigned long long bits = 0ull;
    int hits = 0;
    for (int q = q0; q < q1; q += UQ) {
        float x[UQ], y[UQ], z[UQ];
#pragma unroll
        for (int k = 0; k < UQ; ++k) {
            x[k] = sc.x[min(q + k, q1 - 1)];
            y[k] = sc.y[min(q + k, q1 - 1)];
            z[k] = sc.z[min(q + k, q1 - 1)];
        }
#pragma unroll
        for (int k = 0; k < UQ; ++k) {
            if (q + k < q1 && in_list(x[k], y[k], z[k], q + k)) {
                if (q + k - q0 < 64) bits |= 1ull << (q + k - q0);
                ++hits;
            }
        }
    }
    int incl = hits;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    int pos = incl - hits;
    uint32_t *lp = B.list + p;
    const uint32_t code = list_entry(0u, dx, dy, dz);
    while (bits) {
        const int k = __ffsll((long long)bits) - 1;
        bits &= bits - 1ull;
        if (pos < cap) lp[(size_t)pos * ld] = (uint32_t)(q0 + k) | code;
        ++pos;
    }
    for (int q = q0 + 64; q < q1; ++q)
        if (in_list(sc.x[q], sc.y[q], sc.z[q], q)) {
            if (pos < cap) lp[(size_t)pos * ld] = (uint32_t)q | code;
            ++pos;
        }
    if (lane == 0) {
        B.nnb[p] = min(total, cap);
        if (total > cap) atomicOr(&B.st->error, ERR_LIST_OVERFLOW);
    }
    return total;
}

// Largest neighbour count into st->max_nnb: a warp that exceeds it adds its
// own (no block barrier, which made warps wait for the block's slowest; the
// word is read first, so only a few warps write).  All lanes must call.
__device__ __forceinline__ void warp_max_nnb(int cnt, int *dst)
{
    const int m = __reduce_max_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0 && m > *(volatile int *)dst) atomicMax(dst, m);
}

// Opening kick and drift of atom i from the forces cached at the last closed
// step: v += F dt/(2m), x += v dt; record buffer sp ^ 1 gets the new
// coordinates.  Returns the squared displacement since the last build (FP32).
template <class R>
__device__ __forceinline__ float open_atom(const Bufs<R> &B, const Launch &L, int s, int sp, int i)
{
    int ti = L.ntypes > 1 ? B.type[s][i] : 0;
    double kq = L.half_kick[ti];
    double dn[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double v = B.v[s][a][i];
        v = fma((double)B.fcache[a][i], kq, v);
        B.v[s][a][i] = v;
        dn[a] = fma(v, L.dt, B.d[a][i]);
        B.d[a][i] = dn[a];
    }
    R u0 = B.uref[0][i] + (R)dn[0], u1 = B.uref[1][i] + (R)dn[1], u2 = B.uref[2][i] + (R)dn[2];
    B.shadow[sp ^ 1][i] = mk4<R>(u0, u1, u2, (R)0);
    if constexpr (sizeof(R) == 8) B.rec32[sp ^ 1][i] = make_float4((float)u0, (float)u1, (float)u2, 0.f);
    float fx = (float)dn[0], fy = (float)dn[1], fz = (float)dn[2];
    return fx * fx + fy * fy + fz * fz;
}

// Sum of partials[slot * stride + b], b < nb, by one block (any size) in a
// fixed order; the result goes to the DevState field of the slot (0: embedding
// energy, 1: pair energy, 2: kinetic energy, 3..8: virial).
__device__ __forceinline__ void reduce_slot(const double *partials, DevState *st, int slot, int nb, int stride)
{
    __shared__ double sm[32];
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) s += partials[(size_t)slot * stride + b];
    s = warp_sum_d(s);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sm[w];
        if (slot == 0) st->e_embed = t;
        else if (slot == 1) st->e_pair = t;
        else if (slot == 2) st->ke = t;
        else st->virial[slot - 3] = t;
    }
    __syncthreads();
}

}  // namespace
}  // namespace eammd
