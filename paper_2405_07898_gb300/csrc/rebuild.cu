// rebuild.cu -- sm_103a kernels of the EAM timestep other than the pair
// passes (those are in pair_kernels.cuh):
//   candidate exchange + neighbour list  -> k_bin .. k_build_list (every
//                                           rebuild, Section "Neighbor list")
//   atom swap                            -> the spatial re-sort inside the
//                                           rebuild (k_bin .. k_permute)
//   per-step control                     -> k_decide (rebuild condition),
//                                           k_open (first kick and drift of
//                                           an md_step call), k_reduce
//   state in and out                     -> k_load_state, k_store_state
// R is the pair-arithmetic type: float in the mixed-precision path, double in
// the FP64 path.  Positions, velocities, the drift and all sums over atoms are
// FP64 in both paths.
#include "rebuild_device.cuh"

#include <cuda_runtime.h>

namespace eammd {
namespace {

// Largest system whose list the graph path builds with a warp per atom.
// Measured with graphs (BCC, 1,000 K): +26 % timesteps/s at 1,024 atoms,
// +14 % at 18,522, +2 % at 43,904, and a loss from 118,638 atoms up.
constexpr int64_t kListWarpMaxAtoms = 32768;

// Largest cell grid whose scan is one launch: its blocks read the counts
// nblocks/2 times over, which costs more than the second launch above that.
constexpr int kScanOneLaunch = 65536;

// --------------------------------------------------------------------------
// list build (every rebuild): wrap and bin, scan, scatter, permute, list

template <class R>
__global__ void k_bin(Bufs<R> B, Geom G, int n)
{
    const DevState *st = B.st;
    if (!st->need_rebuild) return;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) bin_atom<R>(B, G, st->set, i);
}

// Per block of kScanBlock cells: total count.
template <class R>
__global__ void k_scan_blocks(Bufs<R> B, int ncells)
{
    if (!B.st->need_rebuild) return;
    const int base = blockIdx.x * kScanBlock;
    int v = 0;
    for (int c = base + threadIdx.x; c < min(base + kScanBlock, ncells); c += blockDim.x) v += B.count[c];
    v = block_sum_i(v);
    if (threadIdx.x == 0) B.block_sums[blockIdx.x] = v;
}

// Accounts of the build, by one thread of the scan: no other thread of that
// launch reads these words.  k_bin reads the old buffer set; the kernels
// after the scan write the new one (and copy from the other).
__device__ __forceinline__ void count_build(DevState *st, int in_graph)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->set = 1 - st->set;
        st->since_build = 0;
        st->rebuilds += 1;
        st->graph_rebuilds += in_graph;
        st->max_nnb = 0;
    }
}

// Exclusive scan of the cell counts: cell_start[c] = sum_{c' < c} count[c'].
// Block b adds the totals of blocks < b (k_scan_blocks), then scans its own
// kScanBlock cells (blockDim.x == kScanBlock).
template <class R>
__global__ void __launch_bounds__(kScanBlock) k_scan_apply(Bufs<R> B, int ncells, int in_graph)
{
    if (!B.st->need_rebuild) return;
    count_build(B.st, in_graph);
    const int b = blockIdx.x, base = b * kScanBlock;
    int v = 0;
    for (int k = threadIdx.x; k < b; k += blockDim.x) v += B.block_sums[k];
    scan_tiles(B.count, B.cell_start, base, min(base + kScanBlock, ncells), ncells, block_sum_i(v));
}

// The same in one launch, for grids of at most kScanOneLaunch cells: every
// block adds up all the counts before its part itself.
template <class R>
__global__ void __launch_bounds__(kScanBlock) k_scan(Bufs<R> B, int ncells, int in_graph)
{
    if (!B.st->need_rebuild) return;
    count_build(B.st, in_graph);
    scan_part(B.count, B.cell_start, ncells, blockIdx.x, gridDim.x);
}

template <class R>
__global__ void k_scatter(Bufs<R> B, int n)
{
    const DevState *st = B.st;
    if (!st->need_rebuild) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) scatter_atom<R>(B, 1 - st->set, i);
}

template <class R>
__global__ void k_permute(Bufs<R> B, Geom G, int n)
{
    const DevState *st = B.st;
    if (!st->need_rebuild) return;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n) permute_atom<R>(B, G, 1 - st->set, st->sp, q);
    for (int c = q; c < G.ncells; c += gridDim.x * blockDim.x) B.count[c] = 0;  // for the next build
}

// A warp per atom (list_atom_warp), for systems of up to kListWarpMaxAtoms:
// there the thread-per-atom walk waits on load latency.  Above that it is
// bound by instruction issue, which the warp form multiplies (a 799,496-atom
// rebuild took about 780 us with it).
template <class R>
__global__ void __launch_bounds__(256) k_build_list_warp(Bufs<R> B, Geom G, int n, int ld, int cap)
{
    DevState *st = B.st;
    if (!st->need_rebuild) return;
    const int p = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);  // the same for a warp's lanes
    const int cnt = (p < n) ? list_atom_warp<R>(B, G, st->set, p, ld, cap) : 0;
    warp_max_nnb(cnt, &st->max_nnb);
}

template <class R>
__global__ void __launch_bounds__(256, 6) k_build_list(Bufs<R> B, Geom G, int n, int ld, int cap, int half)
{
    DevState *st = B.st;
    if (!st->need_rebuild) return;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int cnt = (p < n) ? list_atom<R>(B, G, st->set, p, ld, cap, half != 0) : 0;
    warp_max_nnb(cnt, &st->max_nnb);
}

// --------------------------------------------------------------------------
// per-step kernels

// Start of a step: account for the drift just taken, flip the shadow buffer
// and decide whether the list must be rebuilt before the force evaluation
// (10 steps since the last build, or an atom moved more than skin/2).
__global__ void k_decide(DevState *st, int rebuild_every, double disp2_thr, cudaGraphConditionalHandle h_if,
                         int use_cond)
{
    st->sp ^= 1;
    st->step += 1;
    st->since_build += 1;
    float md = __uint_as_float(st->maxdisp2);
    st->maxdisp2 = 0u;
    int need = (st->since_build >= rebuild_every) || ((double)md > disp2_thr);
    st->need_rebuild = need;
    if (use_cond) cudaGraphSetConditional(h_if, need ? 1u : 0u);
}

// Opening kick and drift of a step from the forces cached at the last
// closed step: v += F dt/(2m), x += v dt.
template <class R>
__global__ void k_open(Bufs<R> B, Launch L)
{
    const DevState *st = B.st;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const float d2 = (i < L.n) ? open_atom<R>(B, L, st->set, st->sp, i) : 0.f;
    block_max_disp(d2, &B.st->maxdisp2);
}

// Fixed-order sum of the per-block partials: block `slot` sums slot 0
// (embedding energy) over the density pass's blocks, or slots 1..8 (pair
// energy, kinetic energy, virial) over the force pass's blocks.
template <class R>
__global__ void __launch_bounds__(1024) k_reduce(Bufs<R> B, int nb_d, int nb_f, int stride)
{
    const int slot = blockIdx.x;
    reduce_slot(B.partials, B.st, slot, slot == 0 ? nb_d : nb_f, stride);
}

// Host arrays in, device SoA out: state of md_create / md_set_state in the
// caller's atom order (the next list build sorts it).  The cell counts start
// from zero: a single launch that timed out inside a build leaves its own.
template <class R>
__global__ void k_load_state(Bufs<R> B, const double *pos, const double *vel, const int *types, int n, int ncells)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) load_atom<R>(B, B.st->set, pos, vel, types, i);
    for (int c = i; c < ncells; c += gridDim.x * blockDim.x) B.count[c] = 0;
}

// Device SoA (sorted) out to interleaved arrays in the caller's order.
template <class R>
__global__ void k_store_state(Bufs<R> B, double *pos, double *vel, double *force, int n)
{
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int s = B.st->set;
    size_t o = 3 * (size_t)B.id[s][p];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (pos) pos[o + a] = __dadd_rn(B.xr[s][a][p], B.d[a][p]);
        if (vel) vel[o + a] = B.v[s][a][p];
        if (force) force[o + a] = (double)B.fcache[a][p];
    }
}

}  // namespace

// --------------------------------------------------------------------------
// launchers

template <class R>
int launch_rebuild(const Bufs<R> &B, const Geom &G, const Launch &L)
{
    const int b = L.block, nb = blocks_for(L.n, b);
    const int nsb = blocks_for(G.ncells, kScanBlock);
    k_bin<R><<<nb, b, 0, L.stream>>>(B, G, L.n);
    if (G.ncells <= kScanOneLaunch) {
        k_scan<R><<<nsb, kScanBlock, 0, L.stream>>>(B, G.ncells, L.use_cond);
    } else {
        k_scan_blocks<R><<<nsb, 256, 0, L.stream>>>(B, G.ncells);
        k_scan_apply<R><<<nsb, kScanBlock, 0, L.stream>>>(B, G.ncells, L.use_cond);
    }
    k_scatter<R><<<nb, b, 0, L.stream>>>(B, L.n);
    k_permute<R><<<nb, b, 0, L.stream>>>(B, G, L.n);
    if (!L.half && (int64_t)L.n <= kListWarpMaxAtoms)
        k_build_list_warp<R><<<blocks_for((int64_t)L.n * 32, 256), 256, 0, L.stream>>>(B, G, L.n, L.ld, L.cap);
    else
        k_build_list<R><<<blocks_for(L.n, L.list_block), L.list_block, 0, L.stream>>>(B, G, L.n, L.ld, L.cap, L.half);
    return rebuild_kernels(G);
}

int rebuild_kernels(const Geom &G) { return G.ncells <= kScanOneLaunch ? 5 : 6; }

template <class R>
int launch_decide(const Bufs<R> &B, const Launch &L)
{
    k_decide<<<1, 1, 0, L.stream>>>(B.st, L.rebuild_every, L.disp2_thr, L.cond, L.use_cond);
    return 1;
}

template <class R>
int launch_open(const Bufs<R> &B, const Geom &G, const Launch &L)
{
    (void)G;
    k_open<R><<<L.nblocks, L.block, 0, L.stream>>>(B, L);
    return 1;
}

template <class R>
int launch_reduce(const Bufs<R> &B, const Launch &L)
{
    k_reduce<R><<<9, 1024, 0, L.stream>>>(B, L.nb_d, L.nb_f, L.pstride);
    return 1;
}

template <class R>
int launch_load_state(const Bufs<R> &B, const Geom &G, const Launch &L, const double *pos, const double *vel,
                      const int *types)
{
    k_load_state<R><<<L.nblocks, L.block, 0, L.stream>>>(B, pos, vel, types, L.n, G.ncells);
    return 1;
}

template <class R>
int launch_store_state(const Bufs<R> &B, const Launch &L, double *pos, double *vel, double *force)
{
    k_store_state<R><<<L.nblocks, L.block, 0, L.stream>>>(B, pos, vel, force, L.n);
    return 1;
}

#define EAMMD_INSTANTIATE(R)                                                                   \
    template int launch_rebuild<R>(const Bufs<R> &, const Geom &, const Launch &);              \
    template int launch_decide<R>(const Bufs<R> &, const Launch &);                             \
    template int launch_open<R>(const Bufs<R> &, const Geom &, const Launch &);                 \
    template int launch_reduce<R>(const Bufs<R> &, const Launch &);                             \
    template int launch_load_state<R>(const Bufs<R> &, const Geom &, const Launch &, const double *,   \
                                      const double *, const int *);                             \
    template int launch_store_state<R>(const Bufs<R> &, const Launch &, double *, double *, double *);

EAMMD_INSTANTIATE(float)
EAMMD_INSTANTIATE(double)

}  // namespace eammd
