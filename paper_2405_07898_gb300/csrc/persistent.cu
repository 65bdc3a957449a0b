// persistent.cu -- md_step as one launch: every phase of every step (opening
// kick, rebuild decision, list rebuild, density, force with the kicks and the
// drift, energy sums) runs in one cooperative-grid kernel whose blocks meet at
// grid barriers (k_steps).  For small systems, where a step is a few
// microseconds of work, this removes the per-kernel launch and scheduling
// gaps of the graph path.  The per-atom arithmetic is that of the graph path (same device
// functions, same lanes per atom), so positions, velocities and forces are
// bitwise equal; energy sums differ in rounding only (other block partition).
//
// Grid barriers: all blocks are resident (cooperative launch); a barrier is
// an arrival counter in device memory.  A wait gives up after the wait limit
// (md_options.wait_limit_us, 1 s by default) of %globaltimer and raises
// ERR_TIMEOUT; the block leaves the kernel, and the others see the error word
// or run into the limit themselves, so the kernel ends within about the limit
// of a stuck block and the host reports MD_ERR_TIMEOUT.
#include "pair_kernels.cuh"
#include "rebuild_device.cuh"

#include <algorithm>

namespace eammd {
namespace {

__device__ __forceinline__ void prefetch_l1(const void *p)
{
    asm volatile("prefetch.global.L1 [%0];" ::"l"(__cvta_generic_to_global(p)));
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(__cvta_generic_to_global(p)) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(__cvta_generic_to_global(p)) : "memory");
    return v;
}

// Grid barrier on a counter that only grows during a launch (zeroed by the
// host before it): barrier b of the launch (b = 1, 2, ...) is passed once the
// counter reaches b x gridDim.x.  Arrival is a release add whose result
// nobody waits for (every block counts the barriers itself); the wait polls
// with acquire loads, so every block sees the writes all blocks made before
// the barrier.  A trip to L2 is about 0.4 us and a barrier is a chain of them:
// the fence of the release, the add, the polls.  (1,024 atoms, 2.6 barriers a
// step: 11.35 us a step with the add's result waited for, the error word read
// first and relaxed polls before one acquire load, 11.26 with relaxed polls
// and a fence, 10.45 so.)
// Returns false once a wait of the launch has timed out (a block that waits
// reads the clock every 4th poll and the error word every 64th; one that gave
// up arrives no more, so nobody passes a later barrier).
__device__ __forceinline__ bool grid_barrier(PersistScratch *ps, unsigned *err, uint64_t wait_ns,
                                             unsigned long long &target)
{
    __shared__ int ok;
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int good = 1;
        asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(__cvta_generic_to_global(&ps->arrive)) : "memory");
        if (ld_acquire(&ps->arrive) < target) {
            const uint64_t t0 = global_ns();
            unsigned spins = 0;
            while (ld_acquire(&ps->arrive) < target) {
                ++spins;
                if (((spins & 3u) == 0 && global_ns() - t0 > wait_ns) ||
                    ((spins & 63u) == 0 && (ld_acquire(err) & ERR_TIMEOUT))) {
                    atomicOr(err, ERR_TIMEOUT);
                    good = 0;
                    break;
                }
            }
        }
        ok = good;
    }
    __syncthreads();
    return ok;
}

// The list build of the single launch: a warp per atom (list_atom_warp)
// while the grid's warps cover the atoms in at most this many passes, else
// one thread per atom (list_atom).  Measured on the BCC sweep: 8 passes
// gains 5-14 % per step up to 18,522 atoms; 16 and 64 lose at 43,904 and
// 118,638 atoms.
constexpr int kListWarpPasses = 8;

// One step loop of nsteps steps (nsteps >= 1).  The counters of DevState
// (set, record buffer, steps since the build) advance identically in every
// block; block 0 writes them back at the end.  The largest squared
// displacement alternates between two words: the force pass of step k writes
// word k & 1, the decision of step k + 1 reads it (the opening drift writes
// word 1 for the decision of step 0).
template <class R, int KIND, int TPA>
__global__ void __launch_bounds__(256) k_steps(Bufs<R> B, Geom G, Launch L, long long nsteps, PersistScratch *ps,
                                               MeasureArgs M)
{
    using R4 = typename V4<R>::T;
    constexpr int kEnergyKind = KIND == KIND_TYPES ? KIND_ANY : KIND;  // as the graph path's last step
    constexpr int UD = PairsInFlight<R, KIND>::density, UF = PairsInFlight<R, KIND>::force;
    DevState *st = B.st;
    unsigned *err = &st->error;
    unsigned long long target = 0;  // of the grid barriers
    // a launch that timed out left its phase half done, and a build that it
    // had begun left its cell counts: nothing runs on it until the state is
    // set anew (the error word is cleared then, the counts as it is loaded)
    if (__syncthreads_or((int)(ld_acquire(err) & ERR_TIMEOUT))) return;
    int s = st->set, sp = st->sp, since = st->since_build;
    long long step = st->step, rebuilds = 0;
    int need = 0;
    const int n = L.n, nthreads = gridDim.x * blockDim.x, gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const int width = blockDim.x / TPA, l = threadIdx.x % TPA;
    const int ntiles = (n + width - 1) / width;
    R h[3];
    load_h<R>(G, h);
    const R rc2 = g_rc2<R>(G);

    if (M.on) {
        // a state to evaluate: one round below
        if (M.pos) {
            for (int i = gtid; i < n; i += nthreads) load_atom<R>(B, s, M.pos, M.vel, M.types, i);
            for (int c = gtid; c < G.ncells; c += nthreads) B.count[c] = 0;  // a launch that timed out leaves its counts
        }
    } else {
        // opening kick and drift from the cached forces
        float d2 = 0.f;
        for (int i = gtid; i < n; i += nthreads) d2 = fmaxf(d2, open_atom<R>(B, L, s, sp, i));
        block_max_disp(d2, &ps->maxdisp[1]);
    }
    if (!grid_barrier(ps, err, L.wait_ns, target)) return;

    for (long long k = 0; k < nsteps; ++k) {
        const bool last = k == nsteps - 1;
        // decision (as k_decide)
        if (!M.on) {
            sp ^= 1;
            step += 1;
            since += 1;
        }
        const float md = __uint_as_float(ld_acquire(&ps->maxdisp[(k + 1) & 1]));
        // (as a condition: with M.on selecting between the two, 2,000 atoms in
        // FP64 took 1,855 us per 100 steps instead of 1,845)
        need = M.on == MEASURE_REBUILD ||
               (M.on == 0 && ((since >= L.rebuild_every) || ((double)md > L.disp2_thr)));
        // word k & 1 was last read by the decision of step k - 1
        if (gtid == 0) ps->maxdisp[k & 1] = 0u;

        if (need) {
            for (int i = gtid; i < n; i += nthreads) bin_atom<R>(B, G, s, i);
            if (!grid_barrier(ps, err, L.wait_ns, target)) return;
            scan_part(B.count, B.cell_start, G.ncells, blockIdx.x, gridDim.x);
            if (!grid_barrier(ps, err, L.wait_ns, target)) return;
            for (int i = gtid; i < n; i += nthreads) scatter_atom<R>(B, s, i);
            if (!grid_barrier(ps, err, L.wait_ns, target)) return;
            for (int q = gtid; q < n; q += nthreads) permute_atom<R>(B, G, s, sp, q);
            for (int c = gtid; c < G.ncells; c += nthreads) B.count[c] = 0;  // for the next build
            if (gtid == 0) st->max_nnb = 0;
            s = 1 - s;
            since = 0;
            rebuilds += 1;
            if (!grid_barrier(ps, err, L.wait_ns, target)) return;
            if ((long long)n * 32 <= (long long)nthreads * kListWarpPasses) {
                // a warp per atom, one lane per stencil cell; the grid's warps
                // take the atoms in at most kListWarpPasses passes
                const int nwarps = nthreads >> 5;
                const int w0 = gtid >> 5;
                int cmax = 0;
                for (int base = 0; base < n; base += nwarps) {
                    const int p = base + w0;
                    // the warp's lanes share p, so the whole warp takes this branch
                    if (p < n) cmax = max(cmax, list_atom_warp<R>(B, G, s, p, L.ld, L.cap));
                }
                warp_max_nnb(cmax, &st->max_nnb);
            } else {
                int cmax = 0;
                for (int p = gtid; p < n; p += nthreads) cmax = max(cmax, list_atom<R>(B, G, s, p, L.ld, L.cap));
                warp_max_nnb(cmax, &st->max_nnb);
            }
            if (!grid_barrier(ps, err, L.wait_ns, target)) return;
        }

        // density pass
        {
            R4 *sw = B.shadow[sp];
            R e_embed = (R)0;
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
                const int i = tile * width + threadIdx.x / TPA;
                const bool active = i < n;
                const int ti = (KIND != KIND_ONE && active) ? B.type[s][i] : 0;
                R rho = density_atom<R, KIND, TPA, UD>(B, G, L, h, rc2, s, sp, i, l, active, GlobalFetch<R>{sw},
                                                        TabGlobal<R>(B));
                rho = lane_sum<TPA>(rho);
                if (active && l == 0) e_embed += embed<R>(B, sw, i, ti, rho);
            }
            if (last) {
                const R v[1] = {e_embed};
                block_sums_t<1, R>(v, B.partials, L.pstride, 0);
            }
        }
        if (!grid_barrier(ps, err, L.wait_ns, target)) return;

        // force pass with the closing kick (and, but for the last step, the
        // next opening kick and the drift)
        {
            const R4 *sw = B.shadow[sp];
            R e7[7] = {0, 0, 0, 0, 0, 0, 0};
            double ke = 0.0;
            float d2max = 0.f;
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
                const int i = tile * width + threadIdx.x / TPA;
                const bool active = i < n;
                const int ti = (KIND != KIND_ONE && active) ? B.type[s][i] : 0;
                R f[3] = {0, 0, 0};
                float d2 = 0.f;
                // the integration's inputs into L1 while the pair loop runs
                if (active && l == 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        prefetch_l1(B.v[s][c] + i);
                        prefetch_l1(B.d[c] + i);
                        prefetch_l1(B.uref[c] + i);
                    }
                }
                if (last) {
                    force_atom<R, kEnergyKind, true, TPA, UF>(B, G, L, h, rc2, s, sp, i, l, ti, active, GlobalFetch<R>{sw}, f,
                                                        e7, TabGlobal<R>(B));
#pragma unroll
                    for (int c = 0; c < 3; ++c) f[c] = lane_sum<TPA>(f[c]);
                    if (active && M.on) integrate<R, MODE_MEASURE, true, TPA>(B, L, s, sp, i, l, ti, f, ke, d2);
                    else if (active) integrate<R, MODE_CLOSE, true, TPA>(B, L, s, sp, i, l, ti, f, ke, d2);
                } else {
                    force_atom<R, KIND, false, TPA, UF>(B, G, L, h, rc2, s, sp, i, l, ti, active, GlobalFetch<R>{sw}, f,
                                                         e7, TabGlobal<R>(B));
#pragma unroll
                    for (int c = 0; c < 3; ++c) f[c] = lane_sum<TPA>(f[c]);
                    if (active) integrate<R, MODE_CLOSE_OPEN, false, TPA>(B, L, s, sp, i, l, ti, f, ke, d2);
                }
                d2max = fmaxf(d2max, lane_sum<TPA>(d2));
            }
            if (last) {
                const R ke_hi = (R)ke;
                const R ke_lo = (R)(ke - (double)ke_hi);
                const R v8[8] = {e7[0], ke_hi, e7[1], e7[2], e7[3], e7[4], e7[5], e7[6]};
                const R lo8[8] = {0, ke_lo, 0, 0, 0, 0, 0, 0};
                block_sums_t<8, R>(v8, B.partials, L.pstride, 1, lo8);
            } else {
                block_max_disp(d2max, &ps->maxdisp[k & 1]);
            }
        }
        if (!grid_barrier(ps, err, L.wait_ns, target)) return;
    }

    // energies of the last step, counters back to DevState
    for (int slot = blockIdx.x; slot < 9; slot += gridDim.x) reduce_slot(B.partials, st, slot, gridDim.x, L.pstride);
    if (gtid == 0) {
        st->set = s;
        st->sp = sp;
        st->since_build = since;
        st->step = step;
        st->rebuilds += rebuilds;
        st->need_rebuild = need;
        st->maxdisp2 = 0u;
        ps->maxdisp[0] = 0u;
        ps->maxdisp[1] = 0u;
    }
}

template <class R, int KIND>
const void *steps_kernel(int tpa)
{
    switch (tpa) {
    case 1: return (const void *)k_steps<R, KIND, 1>;
    case 2: return (const void *)k_steps<R, KIND, 2>;
    case 4: return (const void *)k_steps<R, KIND, 4>;
    default: return (const void *)k_steps<R, KIND, 8>;
    }
}

template <class R>
const void *steps_kernel_of(int multi, int tpa)
{
    if (multi == KIND_TYPES) return steps_kernel<R, KIND_TYPES>(tpa);
    return multi ? steps_kernel<R, KIND_ANY>(tpa) : steps_kernel<R, KIND_ONE>(tpa);
}

}  // namespace

template <class R>
int persistent_grid(const Launch &L, int tpa, int block)
{
    const void *fn = steps_kernel_of<R>(L.multi, tpa);
    int per_sm = 0, dev = 0, nsm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, compact_bytes<R>(block, tpa)) != cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || per_sm <= 0)
        return 0;
    const int width = block / tpa;
    const int ntiles = (L.n + width - 1) / width;
    return std::max(1, std::min(ntiles, per_sm * nsm));
}

template <class R>
cudaError_t launch_steps(const Bufs<R> &B, const Geom &G, const Launch &L, long long nsteps, const PersistSched &sched,
                         PersistScratch *ps, const MeasureArgs &measure)
{
    const void *fn = steps_kernel_of<R>(L.multi, sched.tpa);
    Bufs<R> b = B;
    Geom g = G;
    Launch l = L;
    long long ns = nsteps;
    PersistScratch *p = ps;
    MeasureArgs m = measure;
    // a state is evaluated whatever the wait limit of the steps is
    if (m.on) l.wait_ns = std::max(l.wait_ns, kLeastWaitNs);
    void *args[] = {&b, &g, &l, &ns, &p, &m};
    cudaError_t e = cudaMemsetAsync(ps, 0, sizeof(PersistScratch), L.stream);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(fn, dim3(sched.grid), dim3(sched.block), args,
                                       compact_bytes<R>(sched.block, sched.tpa), L.stream);
}

template int persistent_grid<float>(const Launch &, int, int);
template int persistent_grid<double>(const Launch &, int, int);
template cudaError_t launch_steps<float>(const Bufs<float> &, const Geom &, const Launch &, long long,
                                         const PersistSched &, PersistScratch *,
                                         const MeasureArgs &);
template cudaError_t launch_steps<double>(const Bufs<double> &, const Geom &, const Launch &, long long,
                                          const PersistSched &, PersistScratch *,
                                         const MeasureArgs &);

}  // namespace eammd
