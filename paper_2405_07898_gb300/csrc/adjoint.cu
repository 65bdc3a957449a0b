// adjoint.cu -- gradient of the force-matching loss with respect to the
// spline coefficients of phi, f and F (single atom type, FP64 path).
//
// For one configuration with energy E (Eq. 3) and forces F (Eq. 4):
//   L = (E - E_ref)^2 / N + w sum_i |F_i - F_ref,i|^2.
// With A = 2 (E - E_ref)/N and g = F - F_ref, and since F = -dE/dx,
//   dL/dtheta = A dE/dtheta - 2 w D_g[dE/dtheta],
// D_g the derivative along the position perturbation dx = g:
//   dr_ij = (x_j - x_i)/r . (g_j - g_i),   drho_i = sum_j f'(r_ij) dr_ij.
// Per interval row (a, b, c, d) of the spline that holds x, with
// B = (1, t, t^2, t^3) and B' = (0, 1, 2t, 3t^2):
//   phi row of r_ij (each ordered pair):  1/2 A B - w B' dr_ij
//   f   row of r_ij (each ordered pair):  A F'_i B - 2w (F''_i drho_i B + F'_i B' dr_ij)
//   F   row of rho_i (each atom):         A B - 2w B' drho_i
// rho is recomputed here from the neighbour list (no per-pair term is
// stored).  Each warp owns shared-memory bins for all rows; its lanes add in
// lane order, warps and blocks are summed in a fixed order: the gradient is
// bitwise reproducible.
#include "device_common.cuh"

#include <cuda_runtime.h>

namespace eammd {
namespace {

struct AdjDesc {
    // spline grids (FP64) of phi, f, F
    double x0[3], h[3], inv_h[3];
    int nint[3];       // intervals
    int row0[3];       // first bin row of each function in the bin array
    int nrows;         // total rows (sum of nint)
    double e_ref, w;
};

__device__ __forceinline__ int adj_seg(const AdjDesc &D, int q, double x, double &t)
{
    int k;
    if (x < D.x0[q]) k = 0;
    else k = min((int)((x - D.x0[q]) * D.inv_h[q]), D.nint[q] - 1);
    t = x - (D.x0[q] + (double)k * D.h[q]);
    return k;
}

// value and slope rows of the coefficient derivative at x (inside: the
// cubic; beyond an end: the tangent line used by the spline evaluation)
__device__ __forceinline__ int adj_rows(const AdjDesc &D, int q, double x, double bv[4], double bd[4])
{
    double t;
    int k = adj_seg(D, q, x, t);
    double x_end = D.x0[q] + (double)D.nint[q] * D.h[q];
    if (x < D.x0[q]) {
        bv[0] = 1.0; bv[1] = x - D.x0[q]; bv[2] = 0.0; bv[3] = 0.0;
        bd[0] = 0.0; bd[1] = 1.0; bd[2] = 0.0; bd[3] = 0.0;
    } else if (x > x_end) {
        double hh = D.h[q], e = x - x_end;
        bv[0] = 1.0; bv[1] = hh + e; bv[2] = hh * hh + 2.0 * hh * e; bv[3] = hh * hh * hh + 3.0 * hh * hh * e;
        bd[0] = 0.0; bd[1] = 1.0; bd[2] = 2.0 * hh; bd[3] = 3.0 * hh * hh;
    } else {
        bv[0] = 1.0; bv[1] = t; bv[2] = t * t; bv[3] = t * t * t;
        bd[0] = 0.0; bd[1] = 1.0; bd[2] = 2.0 * t; bd[3] = 3.0 * t * t;
    }
    return D.row0[q] + k;
}

// spline value, first and second derivative from a coefficient row
__device__ __forceinline__ double adj_eval(const double4_32a *coef, int offset, const AdjDesc &D, int q, double x,
                                           double &d1, double &d2)
{
    double t;
    int k = adj_seg(D, q, x, t);
    double x_end = D.x0[q] + (double)D.nint[q] * D.h[q];
    if (x < D.x0[q]) {
        double4_32a c = coef[offset];
        d1 = c.y; d2 = 0.0;
        return c.x + c.y * (x - D.x0[q]);
    }
    if (x > x_end) {
        double4_32a c = coef[offset + D.nint[q] - 1];
        double hh = D.h[q];
        double ye = c.x + hh * (c.y + hh * (c.z + hh * c.w));
        double se = c.y + hh * (2.0 * c.z + 3.0 * hh * c.w);
        d1 = se; d2 = 0.0;
        return ye + se * (x - x_end);
    }
    double4_32a c = coef[offset + k];
    d1 = c.y + t * (2.0 * c.z + 3.0 * t * c.w);
    d2 = 2.0 * c.z + 6.0 * t * c.w;
    return c.x + t * (c.y + t * (c.z + t * c.w));
}

// g = F - F_ref in sorted order; block partial sums of |g|^2
__global__ void k_adj_g(Bufs<double> B, const double *f_ref, double *g, int n, double *partials)
{
    const int s = B.st->set;
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    double sq = 0.0;
    if (p < n) {
        size_t o = 3 * (size_t)B.id[s][p];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double v = B.fcache[c][p] - f_ref[o + c];
            g[(size_t)c * n + p] = v;
            sq += v * v;
        }
    }
    double v1[1] = {sq};
    block_sums_t<1, double>(v1, partials, gridDim.x, 0);
}

// rho_i recomputed from the list, and drho_i.  kAdjLanes lanes share an atom
// (columns l, l + kAdjLanes, ...; their sums meet by shuffles), so that the few
// atoms of a configuration reach every SM: the pass is one chain of L2 trips
// and FP64 latencies per listed pair (2,000 atoms under ncu: 82 us with a lane per atom
// and its 26 pairs in sequence, 15 us with 8 lanes).
constexpr int kAdjLanes = 8;
constexpr int kAdjRhoBlock = 64;

__global__ void k_adj_rho(Bufs<double> B, Geom G, int n, int ld, AdjDesc D, int off_f, const double *g,
                          double *rho_out, double *drho_out)
{
    double h[3];
    load_h<double>(G, h);
    const double4_32a *sw = B.shadow[B.st->sp];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int p = t / kAdjLanes, l = t % kAdjLanes;
    double rho = 0.0, drho = 0.0;
    if (p < n) {
        const double4_32a ui = sw[p];
        const int nn = B.nnb[p];
        const double gx = g[p], gy = g[(size_t)n + p], gz = g[2 * (size_t)n + p];
        for (int k = l; k < nn; k += kAdjLanes) {
            const uint32_t e = B.list[(size_t)k * ld + p];
            const int j = (int)(e & kIndexMask);
            const double4_32a uj = sw[j];
            const double hx = g[j], hy = g[(size_t)n + j], hz = g[2 * (size_t)n + j];
            const Shift<double> s = entry_shift<double>(e, h);
            const double dx = (uj.x - ui.x) + s.x, dy = (uj.y - ui.y) + s.y, dz = (uj.z - ui.z) + s.z;
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (!(r2 < G.rc2)) continue;
            double rinv, r, d1, d2;
            inv_r(r2, rinv, r);
            rho += adj_eval(B.coef, off_f, D, 1, r, d1, d2);
            drho += d1 * ((dx * (hx - gx) + dy * (hy - gy) + dz * (hz - gz)) * rinv);
        }
    }
#pragma unroll
    for (int o = kAdjLanes / 2; o > 0; o >>= 1) {
        rho += __shfl_xor_sync(0xffffffffu, rho, o);
        drho += __shfl_xor_sync(0xffffffffu, drho, o);
    }
    if (p < n && l == 0) {
        rho_out[p] = rho;
        drho_out[p] = drho;
    }
}

// Adds each lane's four values to its row of the warp's bins (row < 0: none).
// Lanes with the same row take turns in lane order, lanes with different rows
// go together, so every bin sees its additions in lane order whatever the
// other rows: a warp needs as many turns as its fullest row has lanes (about
// 4 to 10 of 32).  All 32 lanes must call.
__device__ __forceinline__ void add_rows(double *bins, int row, const double *c)
{
    const unsigned peers = __match_any_sync(0xffffffffu, row);
    const int turn = row < 0 ? -1 : __popc(peers & ((1u << (threadIdx.x & 31u)) - 1u));
    const int turns = __reduce_max_sync(0xffffffffu, turn) + 1;
    for (int k = 0; k < turns; ++k) {
        if (turn == k) {
#pragma unroll
            for (int q = 0; q < 4; ++q) bins[4 * row + q] += c[q];
        }
        __syncwarp();
    }
}

// Contributions of kAdjAtoms atoms to the coefficient bins.  The block's
// warps share the atoms; a warp holds them twice, lane l atom l % kAdjAtoms,
// and takes list columns 2w + (l / kAdjAtoms), stepping by 2 x warps (warp 0
// also the F rows).  Each warp adds into bins of its own in dynamic shared
// memory (4 * nrows doubles); the block adds its warps' bins in warp order
// and writes the sum.  2,000 atoms, 64 knots: 105 us with the 32 lanes adding
// one after another (4 warps, 63 blocks), 27 us with add_rows, 8 warps and
// 125 blocks.
constexpr int kAdjAtoms = 16;

__global__ void k_adj_accum(Bufs<double> B, Geom G, int n, int ld, AdjDesc D, int off_f, int off_F, const double *g,
                            const double *rho_in, const double *drho_in, double *block_bins)
{
    extern __shared__ double bins_all[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    for (int r = threadIdx.x; r < warps * 4 * D.nrows; r += blockDim.x) bins_all[r] = 0.0;
    double *bins = bins_all + (size_t)warp * 4 * D.nrows;
    double h[3];
    load_h<double>(G, h);
    const DevState *st = B.st;
    const double A = 2.0 * ((st->e_embed + st->e_pair) - D.e_ref) / (double)n;
    const double4_32a *sw = B.shadow[st->sp];
    const int half = lane / kAdjAtoms;
    const int p = blockIdx.x * kAdjAtoms + lane % kAdjAtoms;
    const bool active = p < n;
    double4_32a ui = make_double4_32a(0, 0, 0, 0);
    double gx = 0, gy = 0, gz = 0, dF = 0, d2F = 0, drho = 0, rho = 0;
    int nn = 0;
    if (active) {
        ui = sw[p];
        nn = B.nnb[p];
        gx = g[p]; gy = g[(size_t)n + p]; gz = g[2 * (size_t)n + p];
        drho = drho_in[p];
        rho = rho_in[p];
        adj_eval(B.coef, off_F, D, 2, rho, dF, d2F);
    }
    __syncthreads();
    double ca[4], cb[4], bv[4], bd[4];
    if (warp == 0) {  // F row of rho_p
        int row = -1;
        if (active && half == 0) {
            row = adj_rows(D, 2, rho, bv, bd);
#pragma unroll
            for (int c = 0; c < 4; ++c) ca[c] = A * bv[c] - 2.0 * D.w * bd[c] * drho;
        }
        add_rows(bins, row, ca);
    }
    int kmax = nn;
    for (int o = 16; o > 0; o >>= 1) kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    for (int k0 = 2 * warp; k0 < kmax; k0 += 2 * warps) {
        const int k = k0 + half;
        int row_a = -1, row_b = -1;
        if (k < nn) {
            const uint32_t e = B.list[(size_t)k * ld + p];
            const int j = (int)(e & kIndexMask);
            const double4_32a uj = sw[j];
            const double hx = g[j], hy = g[(size_t)n + j], hz = g[2 * (size_t)n + j];
            const Shift<double> s = entry_shift<double>(e, h);
            const double dx = (uj.x - ui.x) + s.x, dy = (uj.y - ui.y) + s.y, dz = (uj.z - ui.z) + s.z;
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (r2 < G.rc2) {
                double rinv, r;
                inv_r(r2, rinv, r);
                const double dr = (dx * (hx - gx) + dy * (hy - gy) + dz * (hz - gz)) * rinv;
                row_a = adj_rows(D, 0, r, bv, bd);  // phi
#pragma unroll
                for (int c = 0; c < 4; ++c) ca[c] = 0.5 * A * bv[c] - D.w * bd[c] * dr;
                row_b = adj_rows(D, 1, r, bv, bd);  // f
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    cb[c] = A * dF * bv[c] - 2.0 * D.w * (d2F * drho * bv[c] + dF * bd[c] * dr);
            }
        }
        add_rows(bins, row_a, ca);
        add_rows(bins, row_b, cb);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < 4 * D.nrows; r += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < warps; ++w) s += bins_all[(size_t)w * 4 * D.nrows + r];
        block_bins[(size_t)blockIdx.x * 4 * D.nrows + r] = s;
    }
}

// Sum of the blocks' bins, in a fixed order: 32 coefficients per block of
// 32 x kFinishParts threads, part y taking block bins y, y + kFinishParts, ...
// (four loads in flight), the parts added in order.  Also the |g|^2 block
// partials (block 0).  One thread per coefficient walked all the bins in
// sequence: 42 us at 2,000 atoms, against 5 us.
constexpr int kFinishParts = 16;

__global__ void k_adj_finish(const double *block_bins, int nblocks, int nrows, const double *partials_g, int nb_g,
                             double *coef_grad, double *sq_out)
{
    __shared__ double sm[kFinishParts][33];
    const int x = threadIdx.x, y = threadIdx.y, r = blockIdx.x * 32 + x;
    double s = 0.0;
    if (r < 4 * nrows) {
        const double *b = block_bins + r;
        const size_t step = 4 * (size_t)nrows;
#pragma unroll 4
        for (int k = y; k < nblocks; k += kFinishParts) s += b[(size_t)k * step];
    }
    sm[y][x] = s;
    __syncthreads();
    if (y == 0 && r < 4 * nrows) {
        double t = 0.0;
        for (int k = 0; k < kFinishParts; ++k) t += sm[k][x];
        coef_grad[r] = t;
    }
    if (blockIdx.x == 0 && y == 1) {
        double q = 0.0;
        for (int b = x; b < nb_g; b += 32) q += partials_g[b];
        q = warp_sum_d(q);
        if (x == 0) *sq_out = q;
    }
}

// knot gradient: for knot q of function fn, sum over that function's
// coefficient rows of M[row][q] * coef_grad[row] (M stored transposed:
// Mt[q][row] over the function's 4*nint coefficients), a warp per knot: lane l
// rows l, l + 32, ..., the lanes' sums meeting by shuffles (47 us with a
// thread per knot at 3 x 64 knots, 7 us so).
__global__ void k_adj_knots(const double *coef_grad, const double *Mt, int nknots_total, const int *knot_func,
                            const int *func_coef0, const int *func_ncoef, const long long *knot_mt0,
                            double *knot_grad)
{
    const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (q >= nknots_total) return;  // the same for a warp's lanes
    const int fn = knot_func[q];
    const double *m = Mt + knot_mt0[q];
    const double *cg = coef_grad + func_coef0[fn];
    double s = 0.0;
    for (int r = lane; r < func_ncoef[fn]; r += 32) s += m[r] * cg[r];
    s = warp_sum_d(s);
    if (lane == 0) knot_grad[q] = s;
}

// Warps of a block of the accumulation: as many as share 16 atoms' columns
// usefully (8) while their bins fit 96 KB, which lets two blocks share an SM;
// 4 for larger tables (up to the limit the host checks).
int adjoint_warps(int nrows) { return 8 * sizeof(double) * 4 * (size_t)nrows <= 96 * 1024 ? 8 : kAdjWarps; }

}  // namespace

int launch_adjoint(const Bufs<double> &B, const Geom &G, const Launch &L, const AdjointArgs &a)
{
    AdjDesc D;
    int row = 0;
    for (int q = 0; q < 3; ++q) {
        D.x0[q] = a.x0[q];
        D.h[q] = a.h[q];
        D.inv_h[q] = 1.0 / a.h[q];
        D.nint[q] = a.nint[q];
        D.row0[q] = row;
        row += a.nint[q];
    }
    D.nrows = row;
    D.e_ref = a.e_ref;
    D.w = a.w;
    const int n = L.n;
    const int nb = blocks_for(n, 256);
    k_adj_g<<<nb, 256, 0, L.stream>>>(B, a.f_ref, a.g, n, a.partials_g);
    k_adj_rho<<<blocks_for((long long)n * kAdjLanes, kAdjRhoBlock), kAdjRhoBlock, 0, L.stream>>>(
        B, G, n, L.ld, D, a.off_f, a.g, a.rho, a.drho);
    const int nw = adjoint_blocks(n), warps = adjoint_warps(D.nrows);
    const size_t smem = adjoint_smem_bytes(D.nrows);
    k_adj_accum<<<nw, 32 * warps, smem, L.stream>>>(B, G, n, L.ld, D, a.off_f, a.off_F, a.g, a.rho, a.drho,
                                                    a.block_bins);
    k_adj_finish<<<blocks_for(4 * D.nrows, 32), dim3(32, kFinishParts), 0, L.stream>>>(
        a.block_bins, nw, D.nrows, a.partials_g, nb, a.coef_grad, a.sq);
    int launched = 4;
    if (a.knot_grad) {
        k_adj_knots<<<blocks_for((long long)a.nknots_total * 32, 256), 256, 0, L.stream>>>(
            a.coef_grad, a.Mt, a.nknots_total, a.knot_func, a.func_coef0, a.func_ncoef, a.knot_mt0, a.knot_grad);
        ++launched;
    }
    return launched;
}

size_t adjoint_smem_bytes(int nrows) { return sizeof(double) * 4 * (size_t)nrows * adjoint_warps(nrows); }

int adjoint_blocks(int n) { return blocks_for(n, kAdjAtoms); }

// The limit belongs to the kernel, not to a context: always the largest that
// the host admits, so that contexts of different tables do not lower it for
// each other.
cudaError_t allow_adjoint_smem()
{
    return cudaFuncSetAttribute(k_adj_accum, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kAdjMaxSmem);
}

}  // namespace eammd
