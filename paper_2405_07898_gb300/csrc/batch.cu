// batch.cu -- many independent periodic systems ("replicas") advanced in one
// persistent launch.
//
// Each team takes a replica from a queue ordered costliest first and runs
// every phase of every step of that replica itself -- list rebuild (wrap,
// bin, scan, scatter, permute, list), density (Eq. 2), force (Eq. 4) fused
// with the velocity-Verlet kicks and drift (Eq. 5) -- with barriers inside the
// team only, so replicas never wait on each other and small systems pay no
// launch per step.  A team is one thread block, or a cluster of blocks where
// replicas are fewer than SMs (or one replica would outlast the rest).  The
// phases are the per-atom functions of the single-system mixed-precision path
// (rebuild_device.cuh, pair_kernels.cuh, one lane per atom), run on a view of
// the replica's part of the batch's arrays, so every replica's list equals
// the FP64 definition and its arithmetic is that of a single context.
//
// What bounds it is what bounds the single system's pair passes (gathers
// through L1, their latency), and the balance of the SMs.  50 steps: 512
// replicas of 3.0 M atoms 56.5 ms (74.8 with this file's earlier own phases,
// which built lists by warps and ballots and loaded a table row in two
// halves); 24 replicas of 1,500-9,000 atoms 3.8 ms in teams of blocks, 23.5
// with a block each; 100 replicas 7.1 against 15.3; 200 replicas 21.9 against
// 37.3.
#include "eammd.h"
#include "pair_kernels.cuh"
#include "rebuild_device.cuh"
#include "spline_host.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

namespace eammd {
namespace {

constexpr int kMaxTeam = 8;  // blocks of a team
// Largest replica whose state is read through pinned memory (4.7 MB); larger
// ones are copied straight into the caller's arrays.
constexpr int kBatchStageAtoms = 65536;
constexpr int kBatchDensityPairs = 4, kBatchForcePairs = 2;  // pairs in flight per lane

// A replica: its view of the arrays, geometry and constants (B.st is its
// DevState; L.n, L.ld, L.cap, L.rebuild_every, L.disp2_thr, L.ke_factor).
struct Replica {
    Bufs<float> B;
    Geom G;
    Launch L;
    double mass;
};

struct BatchArgs {
    const Replica *rep;
    const int *order;  // replicas, costliest first
    int *queue;
    unsigned *maxdisp;  // two words per replica: the largest squared displacement, alternating
    double *part;       // [replica][block of the team][3]: energy sums of the last step
    int nrep;
};

enum { BATCH_INIT = 0, BATCH_RUN = 1 };

struct BatchSmem {
    Replica R;
    int next;
    double red[32];
};

__device__ __forceinline__ int cluster_rank()
{
    int r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ int cluster_size()
{
    int r;
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
    return r;
}

// Barrier of the team; every thread of it sees the writes all made before.
template <bool TEAM>
__device__ __forceinline__ void team_sync()
{
    if (TEAM) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}

// The team's next replica (index into the order), from its first block.
template <bool TEAM>
__device__ __forceinline__ int next_replica(const BatchArgs &A, BatchSmem &S, int rank, int size)
{
    if (rank == 0 && threadIdx.x == 0) {
        const int k = atomicAdd(A.queue, 1);
        S.next = k;
        if (TEAM) {
            const unsigned mine = (unsigned)__cvta_generic_to_shared(&S.next);
            for (int r = 1; r < size; ++r) {
                unsigned there;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(mine), "r"(r));
                asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(there), "r"(k) : "memory");
            }
        }
    }
    team_sync<TEAM>();
    return S.next;
}

// FP64 sum over the block of per-thread float pairs (thread 0 returns it):
// warps in float pairs, then FP64 over the warps in warp order.
__device__ __forceinline__ double block_sum_ff(float hi, float lo, BatchSmem &S)
{
    const double s = warp_sum_ff(hi, lo);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) S.red[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += S.red[w];
    return t;
}

// Largest squared displacement of the warp into a word of non-negative float bits.
__device__ __forceinline__ void warp_max_disp(float d2, unsigned *dst)
{
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(d2));
    if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned *)dst) atomicMax(dst, m);
}

// The replica's spline rows, for tables of any size (segment_fused takes up to
// kMaxFusedIntervals intervals).
struct TabBatch : TabGlobal<float> {
    __device__ __forceinline__ explicit TabBatch(const Bufs<float> &B) : TabGlobal<float>(B) {}
    __device__ __forceinline__ int interval(const SplineDesc<float> &g, float r, float &t) const
    {
        return g.nint > kMaxFusedIntervals ? segment(g, r, t) : segment_fused(g, r, t);
    }
};

// Force phase of atoms [i0, i1): MODE and ENERGY as in the single-system pass.
template <int MODE, bool ENERGY>
__device__ __forceinline__ void force_phase(const Replica &R, const float (&h)[3], float rc2, int s, int sp, int i0, int i1,
                                            float &e_pair, double &ke, float &d2max)
{
    const Bufs<float> &B = R.B;
    const float4 *sw = B.shadow[sp];
    for (int i = i0 + (int)threadIdx.x; i < i1; i += blockDim.x) {
        float f[3] = {0.f, 0.f, 0.f}, e7[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, d2 = 0.f;
        force_lane<float, KIND_ONE, ENERGY, 1, kBatchForcePairs>(B, R.L, h, rc2, s, B.nnb + i, R.L.cap, 0, 0, sw[i],
                                                              ListGlobal{B.list + i, R.L.ld}, GlobalFetch<float>{sw}, f,
                                                              e7, TabBatch(B));
        integrate<float, MODE, ENERGY, 1>(B, R.L, s, sp, i, 0, 0, f, ke, d2);
        if (ENERGY) e_pair += e7[0];
        d2max = fmaxf(d2max, d2);
    }
}

// All steps of one replica by one team.
template <bool TEAM>
__device__ void run_replica(const BatchArgs &A, BatchSmem &S, int r, int rank, int size, int mode, int nsteps)
{
    const Replica &R = S.R;
    const Bufs<float> &B = R.B;
    const Geom &G = R.G;
    DevState *st = B.st;
    unsigned *maxdisp = A.maxdisp + 2 * r;
    const int n = R.L.n, tid = (int)threadIdx.x, nt = (int)blockDim.x;
    // this block's atoms (consecutive: neighbours share its L1) and cells
    const int per = ((n + size - 1) / size + 31) & ~31, i0 = min(rank * per, n), i1 = min(i0 + per, n);
    int s = st->set, sp = st->sp, since = st->since_build;
    long long rebuilds = 0;
    float h[3];
    load_h<float>(G, h);
    const float rc2 = G.rc2_f;
    const int steps = (mode == BATCH_INIT) ? 1 : nsteps;
    if (mode == BATCH_RUN) {
        // opening kick and drift from the cached forces
        float d2 = 0.f;
        for (int i = i0 + tid; i < i1; i += nt) d2 = fmaxf(d2, open_atom<float>(B, R.L, s, sp, i));
        warp_max_disp(d2, &maxdisp[1]);
        team_sync<TEAM>();
    }
    for (int it = 0; it < steps; ++it) {
        const bool last = it == steps - 1;
        bool need = true;
        if (mode == BATCH_RUN) {
            sp ^= 1;
            ++since;
            const float md = __uint_as_float(*(volatile unsigned *)&maxdisp[(it + 1) & 1]);
            need = since >= R.L.rebuild_every || (double)md > R.L.disp2_thr;
            // word it & 1 was last read by the decision of step it - 1
            if (rank == 0 && tid == 0) *(volatile unsigned *)&maxdisp[it & 1] = 0u;
        }
        if (need) {
            for (int i = i0 + tid; i < i1; i += nt) bin_atom<float>(B, G, s, i);
            team_sync<TEAM>();
            scan_part(B.count, B.cell_start, G.ncells, rank, size);
            team_sync<TEAM>();
            for (int i = i0 + tid; i < i1; i += nt) scatter_atom<float>(B, s, i);
            team_sync<TEAM>();
            for (int q = i0 + tid; q < i1; q += nt) permute_atom<float>(B, G, s, sp, q);
            for (int c = rank * nt + tid; c < G.ncells; c += size * nt) B.count[c] = 0;  // for the next build
            s = 1 - s;
            since = 0;
            rebuilds += 1;
            team_sync<TEAM>();
            int cmax = 0;
            for (int p = i0 + tid; p < i1; p += nt) cmax = max(cmax, list_atom<float>(B, G, s, p, R.L.ld, R.L.cap));
            warp_max_nnb(cmax, &st->max_nnb);
            team_sync<TEAM>();
        }
        // density pass: rho, F'(rho) into the record's w; F(rho) for the energy
        float4 *sw = B.shadow[sp];
        float e_emb = 0.f;
        for (int i = i0 + tid; i < i1; i += nt) {
            const float rho = density_lane<float, KIND_ONE, 1, kBatchDensityPairs>(
                B, h, rc2, s, B.nnb + i, R.L.cap, 0, sw[i], ListGlobal{B.list + i, R.L.ld}, GlobalFetch<float>{sw},
                TabBatch(B));
            e_emb += embed<float>(B, sw, i, 0, rho);
        }
        team_sync<TEAM>();
        // force pass fused with the kicks and the drift
        float e_pair = 0.f, d2max = 0.f;
        double ke = 0.0;
        if (mode == BATCH_INIT) force_phase<MODE_MEASURE, true>(R, h, rc2, s, sp, i0, i1, e_pair, ke, d2max);
        else if (last) force_phase<MODE_CLOSE, true>(R, h, rc2, s, sp, i0, i1, e_pair, ke, d2max);
        else force_phase<MODE_CLOSE_OPEN, false>(R, h, rc2, s, sp, i0, i1, e_pair, ke, d2max);
        if (last) {
            const float kh = (float)ke;
            const double eb = block_sum_ff(e_emb, 0.f, S), ep = block_sum_ff(e_pair, 0.f, S);
            const double kt = block_sum_ff(kh, (float)(ke - (double)kh), S);
            if (tid == 0) {
                double *part = A.part + 3 * ((size_t)r * kMaxTeam + rank);
                part[0] = eb;
                part[1] = ep;
                part[2] = kt;
            }
        } else {
            warp_max_disp(d2max, &maxdisp[it & 1]);
        }
        team_sync<TEAM>();
    }
    if (rank == 0 && tid == 0) {
        double sum[3] = {0.0, 0.0, 0.0};
        for (int b = 0; b < size; ++b)
            for (int k = 0; k < 3; ++k) sum[k] += ((volatile double *)A.part)[3 * ((size_t)r * kMaxTeam + b) + k];
        st->e_embed = sum[0];
        st->e_pair = sum[1];
        st->ke = sum[2];
        st->set = s;
        st->sp = sp;
        st->since_build = since;
        st->rebuilds += rebuilds;
        if (mode == BATCH_RUN) st->step += nsteps;
        maxdisp[0] = 0u;
        maxdisp[1] = 0u;
    }
}

template <int BS, int MINB, bool TEAM>
__global__ void __launch_bounds__(BS, MINB) k_batch(BatchArgs A, int mode, int nsteps, double dt)
{
    __shared__ BatchSmem S;
    const int rank = TEAM ? cluster_rank() : 0, size = TEAM ? cluster_size() : 1;
    if (TEAM) team_sync<TEAM>();  // the team's blocks run before one writes to another
    for (;;) {
        const int k = next_replica<TEAM>(A, S, rank, size);
        if (k >= A.nrep) return;  // the same for the team
        const int r = A.order[k];
        // the replica's description to shared memory, word by word
        const unsigned *src = reinterpret_cast<const unsigned *>(A.rep + r);
        unsigned *dst = reinterpret_cast<unsigned *>(&S.R);
        for (int w = threadIdx.x; w < (int)(sizeof(Replica) / sizeof(unsigned)); w += blockDim.x) dst[w] = src[w];
        __syncthreads();
        if (threadIdx.x == 0) {
            S.R.L.dt = dt;
            S.R.L.half_kick[0] = 0.5 * dt * kAccel / S.R.mass;
        }
        __syncthreads();
        run_replica<TEAM>(A, S, r, rank, size, mode, nsteps);
        team_sync<TEAM>();  // nobody writes the next number into a block that still works
    }
}

// replica state to the caller's order (AoS): positions, velocities, forces
__global__ void k_batch_store(const Replica *rep, int r, double *pos, double *vel, double *force)
{
    const Bufs<float> &B = rep[r].B;
    const int s = B.st->set;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= rep[r].L.n) return;
    const size_t o = 3 * (size_t)B.id[s][p];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (pos) pos[o + a] = __dadd_rn(B.xr[s][a][p], B.d[a][p]);
        if (vel) vel[o + a] = B.v[s][a][p];
        if (force) force[o + a] = (double)B.fcache[a][p];
    }
}


// ==========================================================================
// host side

SplineDesc<float> batch_desc(const md_spline &s, int offset, const double *row_last, const double *row0)
{
    SplineDesc<float> d;
    d.offset = offset;
    d.nint = s.n - 1;
    d.x0 = (float)s.x0;
    d.inv_h = (float)(1.0 / s.dx);
    d.h_hi = (float)s.dx;
    d.h_lo = (float)(s.dx - (double)d.h_hi);
    const double x_end = s.x0 + (double)(s.n - 1) * s.dx;
    d.x_end = (float)x_end;
    d.y_lo = (float)row0[0];
    d.s_lo = (float)row0[1];
    const double t = s.dx;
    d.y_end = (float)(row_last[0] + t * (row_last[1] + t * (row_last[2] + t * row_last[3])));
    d.s_end = (float)(row_last[1] + t * (2.0 * row_last[2] + 3.0 * t * row_last[3]));
    return d;
}

thread_local std::string g_batch_create_error;

}  // namespace
}  // namespace eammd

using namespace eammd;

struct md_batch {
    int nrep = 0;
    int64_t total = 0;
    std::vector<Replica> rep;       // as on the device
    int cap = 0;
    BatchArgs A{};
    Replica *rep_dev = nullptr;
    DevState *st = nullptr;         // one per replica
    DevState *st_host = nullptr;    // pinned
    bool st_current = false;        // st_host holds the device's states, st_status what they say
    bool replayable = false;        // steps were captured by the caller: the states are read at every call
    md_status st_status = MD_OK;
    std::string st_message;
    double *host_stage = nullptr;   // pinned: positions, velocities, forces of one replica (kBatchStageAtoms)
    std::vector<void *> allocs;
    md_options opt{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int grid = 0;
    int schedule = 0;               // index into kSchedules
    int chosen = 0;                 // that of md_batch_create
    double *stage = nullptr;
    int max_n = 0;
    long long launches = 0;
    struct G { int nsteps; double dt; cudaGraph_t g; cudaGraphExec_t e; };
    std::vector<G> graphs;
    std::string err;
    md_status fail(md_status s, const std::string &m)
    {
        err = m;
        return s;
    }
};

namespace {

void *balloc(md_batch *b, size_t bytes)
{
    bytes = ((bytes ? bytes : 256) + 255) & ~size_t(255);
    void *p = nullptr;
    if (b->opt.alloc) {
        p = b->opt.alloc(bytes, b->opt.alloc_ctx);
    } else if (cudaMalloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        p = nullptr;
    }
    if (p) b->allocs.push_back(p);
    return p;
}

template <class T>
bool balloc_n(md_batch *b, T *&p, size_t count)
{
    p = (T *)balloc(b, count * sizeof(T));
    return p != nullptr;
}

#define BCK(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return b->fail(e_ == cudaErrorMemoryAllocation ? MD_ERR_OOM : MD_ERR_CUDA,             \
                           std::string(#call) + ": " + cudaGetErrorString(e_));                    \
    } while (0)

// Shapes of the launch: threads per block, blocks per SM, blocks of a team.
// The first five are those of md_options.batch_schedule (1..5).  Teams of
// several blocks serve batches with fewer replicas than SMs, and keep one
// large replica from outlasting the rest.
struct BatchSchedule {
    int block, min_blocks, team;
};
constexpr BatchSchedule kSchedules[] = {{512, 1, 1}, {256, 2, 1}, {256, 3, 1}, {1024, 1, 1},
                                        {512, 2, 1}, {1024, 1, 2}, {1024, 1, 4}, {1024, 1, 8}};
constexpr int kPublicSchedules = 5, kNumSchedules = 8;

const void *batch_kernel(int sched)
{
    switch (sched) {
    case 0: return (const void *)k_batch<512, 1, false>;
    case 1: return (const void *)k_batch<256, 2, false>;
    case 2: return (const void *)k_batch<256, 3, false>;
    case 3: return (const void *)k_batch<1024, 1, false>;
    case 4: return (const void *)k_batch<512, 2, false>;
    default: return (const void *)k_batch<1024, 1, true>;
    }
}

// Shapes that were timed, per device and batch (replicas, atoms, largest
// replica, cells, list capacity, steps between builds), kept for the life of
// the process like the single system's schedules: the shape partitions the
// energy sums, so batches of the same systems give the same bits, and only the
// first of them pays for the trials.
struct BatchKey {
    int dev, nrep, max_n, cap, rebuild_every;
    long long atoms, cells;
    bool operator==(const BatchKey &o) const
    {
        return dev == o.dev && nrep == o.nrep && max_n == o.max_n && cap == o.cap && rebuild_every == o.rebuild_every &&
               atoms == o.atoms && cells == o.cells;
    }
};
std::mutex g_batch_mu;
std::vector<std::pair<BatchKey, int>> g_batch_cache;
constexpr size_t kBatchCacheMax = 256;

void batch_config(int sched, int grid, cudaStream_t stream, cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr)
{
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSchedules[sched].block);
    cfg.stream = stream;
    attr = cudaLaunchAttribute{};
    if (kSchedules[sched].team > 1) {
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = kSchedules[sched].team;
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
}

void batch_drop_graphs(md_batch *b)
{
    for (auto &g : b->graphs) {
        cudaGraphExecDestroy(g.e);
        cudaGraphDestroy(g.g);
    }
    b->graphs.clear();
}

// Blocks of the launch: as many teams as can be resident, at most one per
// replica; 0 if the shape cannot run.
int batch_grid(int sched, int nrep)
{
    const BatchSchedule &k = kSchedules[sched];
    int teams = 0;
    if (k.team > 1) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        batch_config(sched, k.team, nullptr, cfg, attr);
        if (cudaOccupancyMaxActiveClusters(&teams, batch_kernel(sched), &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
    } else {
        int per_sm = 0, sms = 1, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel(sched), k.block, 0);
        teams = std::max(per_sm, 1) * sms;
    }
    return std::min(nrep, teams) * k.team;
}

md_status batch_launch(md_batch *b, int mode, int nsteps, double dt)
{
    b->st_current = false;
    BCK(cudaMemsetAsync(b->A.queue, 0, sizeof(int), b->stream));
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    batch_config(b->schedule, b->grid, b->stream, cfg, attr);
    BatchArgs A = b->A;
    void *args[] = {&A, &mode, &nsteps, &dt};
    BCK(cudaLaunchKernelExC(&cfg, batch_kernel(b->schedule), args));
    b->launches += 1;
    return MD_OK;
}

// Waits for the stream; after new work also reads every replica's state and
// finds the first error.  With nothing queued since, the states and the
// answer read last still stand.
md_status batch_sync(md_batch *b)
{
    if (!b->st_current)
        BCK(cudaMemcpyAsync(b->st_host, b->st, sizeof(DevState) * b->nrep, cudaMemcpyDeviceToHost, b->stream));
    BCK(cudaStreamSynchronize(b->stream));
    if (!b->st_current) {
        b->st_current = !b->replayable;
        b->st_status = MD_OK;
        b->st_message.clear();
        for (int r = 0; r < b->nrep; ++r) {
            const unsigned e = b->st_host[r].error;
            if (e & ERR_LIST_OVERFLOW) {
                b->st_status = MD_ERR_LIST_OVERFLOW;
                b->st_message = "replica " + std::to_string(r) + ": list capacity exceeded (" +
                                std::to_string(b->st_host[r].max_nnb) + " > " + std::to_string(b->cap) + ")";
                break;
            }
            if (e & ERR_NONFINITE) {
                b->st_status = MD_ERR_NONFINITE;
                b->st_message = "replica " + std::to_string(r) + ": non-finite force";
                break;
            }
        }
    }
    return b->st_status == MD_OK ? MD_OK : b->fail(b->st_status, b->st_message);
}

}  // namespace

extern "C" {

md_status md_batch_create(int32_t nrep, const md_replica *reps, int32_t npot, const md_potential *pots,
                          const md_options *opt, md_batch **out)
{
    g_batch_create_error.clear();
    auto bad = [](md_status s, const std::string &m) {
        g_batch_create_error = m;
        return s;
    };
    if (!out) return bad(MD_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (nrep < 1 || !reps || npot < 1 || !pots) return bad(MD_ERR_ARG, "need at least one replica and potential");
    md_options o;
    md_options_default(&o);
    if (opt) o = *opt;
    if (o.precision != MD_PRECISION_MIXED) return bad(MD_ERR_ARG, "batches run the mixed-precision path");
    if (o.open_axes != 0) return bad(MD_ERR_ARG, "batch replicas are periodic (open_axes must be 0)");
    if ((o.alloc == nullptr) != (o.free == nullptr)) return bad(MD_ERR_ARG, "alloc and free go together");
    if (o.rebuild_every < 1) o.rebuild_every = 10;
    if (o.batch_schedule < 0 || o.batch_schedule > kPublicSchedules)
        return bad(MD_ERR_ARG, "batch_schedule must be 0 (tuned) or 1..5");
    // potentials: one type each, f and phi on one grid (fused rows); per
    // potential the fused rows, the derivative rows and the f rows (as in a
    // single context)
    std::vector<double> rowsF, rows2;
    std::vector<size_t> off2(npot);
    std::vector<Tables<float>> tabs(npot);
    for (int q = 0; q < npot; ++q) {
        const md_potential &pt = pots[q];
        if (pt.ntypes != 1 || !pt.mass || !pt.F || !pt.f || !pt.phi || !(pt.mass[0] > 0.0) || !(pt.r_cut > 0.0) ||
            !(pt.skin >= 0.0))
            return bad(MD_ERR_ARG, "batch potentials have one atom type, mass > 0, r_cut > 0, skin >= 0");
        const md_spline &F = pt.F[0], &f = pt.f[0], &ph = pt.phi[0];
        for (const md_spline *sp : {&F, &f, &ph}) {
            if (sp->n < 2 || !(sp->dx > 0.0) || !sp->y) return bad(MD_ERR_ARG, "bad spline");
            for (int k = 0; k < sp->n; ++k)
                if (!std::isfinite(sp->y[k])) return bad(MD_ERR_ARG, "non-finite knot value");
        }
        if (f.n != ph.n || f.x0 != ph.x0 || f.dx != ph.dx || f.x0 > 0.0 || f.x0 + (f.n - 1) * f.dx < pt.r_cut)
            return bad(MD_ERR_ARG, "batch potentials need f and phi on one grid covering [0, r_cut]");
        std::vector<double> rf, rp;
        Tables<float> &t = tabs[q];
        memset(&t, 0, sizeof(t));
        t.ntypes = 1;
        t.fused = 1;
        int offF = (int)(rowsF.size() / 4);
        if (!hermite_coefficients(F, rowsF)) return bad(MD_ERR_ARG, "singular spline");
        t.F[0] = batch_desc(F, offF, &rowsF[rowsF.size() - 4], &rowsF[4 * (size_t)offF]);
        if (!hermite_coefficients(f, rf) || !hermite_coefficients(ph, rp)) return bad(MD_ERR_ARG, "singular spline");
        t.fphi = batch_desc(f, 0, &rf[rf.size() - 4], &rf[0]);
        off2[q] = rows2.size() / 4;
        for (int k = 0; k < f.n - 1; ++k) {
            for (int c = 0; c < 4; ++c) rows2.push_back(rf[4 * (size_t)k + c]);
            for (int c = 0; c < 4; ++c) rows2.push_back(rp[4 * (size_t)k + c]);
        }
        for (int k = 0; k < f.n - 1; ++k) {
            for (const double *c : {&rf[4 * (size_t)k], &rp[4 * (size_t)k]}) {
                rows2.push_back(c[1]);
                rows2.push_back(2.0 * c[2]);
                rows2.push_back((double)(3.f * (float)c[3]));
            }
            rows2.push_back(0.0);
            rows2.push_back(0.0);
        }
        for (int k = 0; k < f.n - 1; ++k)
            for (int c = 0; c < 4; ++c) rows2.push_back(rf[4 * (size_t)k + c]);
        if (rows2.size() % 8) rows2.resize(rows2.size() + 4, 0.0);  // the next potential's rows stay 32-byte aligned
    }
    md_batch *b = new (std::nothrow) md_batch();
    if (!b) return bad(MD_ERR_OOM, "host allocation failed");
    b->opt = o;
    b->nrep = nrep;
    b->rep.resize(nrep);
    struct Place {
        size_t atom, cell, cs;
    };
    std::vector<Place> place(nrep);
    int64_t atom_off = 0, cell_off = 0, cs_off = 0, natoms = 0;
    double max_expect = 0.0;
    std::vector<double> cost(nrep);
    for (int r = 0; r < nrep; ++r) {
        const md_replica &R = reps[r];
        if (R.potential < 0 || R.potential >= npot || R.n < 1 || !R.pos) {
            delete b;
            return bad(MD_ERR_ARG, "replica " + std::to_string(r) + ": bad potential index, n or pos");
        }
        const md_potential &pt = pots[R.potential];
        const double r_list = pt.r_cut + pt.skin;
        Replica &P = b->rep[r];
        memset(&P, 0, sizeof(P));
        Geom &G = P.G;
        for (int a = 0; a < 3; ++a) {
            const double L = R.box[a];
            if (!(L > 0.0) || std::floor(L / r_list) < 3.0) {
                delete b;
                return bad(MD_ERR_BOX, "replica " + std::to_string(r) + ": box edge shorter than 3 (r_cut + skin)");
            }
            G.box[a] = L;
            G.half_box[a] = 0.5 * L;
            G.ncell[a] = (int)std::floor(L / r_list);
            G.inv_cell[a] = (double)G.ncell[a] / L;
            G.h[a] = L / (double)G.ncell[a];
            G.h_f[a] = (float)G.h[a];
            G.inv_cell_f[a] = (float)G.inv_cell[a];
            G.box_f[a] = (float)L;
        }
        G.ncells = G.ncell[0] * G.ncell[1] * G.ncell[2];
        G.rl2 = r_list * r_list;
        G.rl2_f = (float)G.rl2;
        G.rc2 = pt.r_cut * pt.r_cut;
        G.rc2_f = (float)G.rc2;
        P.L.n = (int)R.n;
        P.L.ld = (int)((R.n + 31) / 32 * 32);
        P.L.ntypes = 1;
        P.L.rebuild_every = o.rebuild_every;
        P.L.disp2_thr = 0.25 * pt.skin * pt.skin;
        P.L.ke_factor[0] = 0.5 * pt.mass[0] / kAccel;
        P.mass = pt.mass[0];
        const double vol = R.box[0] * R.box[1] * R.box[2];
        const double expect = (double)R.n / vol * 4.0 / 3.0 * M_PI * r_list * r_list * r_list;
        max_expect = std::max(max_expect, expect);
        cost[r] = (double)R.n * (expect + 8.0);  // listed pairs and a fixed part per atom
        for (int64_t i = 0; i < 3 * R.n; ++i)
            if (!std::isfinite(R.pos[i]) || (R.vel && !std::isfinite(R.vel[i]))) {
                delete b;
                return bad(MD_ERR_NONFINITE, "replica " + std::to_string(r) + ": non-finite input");
            }
        place[r] = {(size_t)atom_off, (size_t)cell_off, (size_t)cs_off};
        atom_off += (R.n + 31) / 32 * 32;  // the list build reads aligned groups of four
        natoms += R.n;
        cell_off += G.ncells;
        cs_off += G.ncells + 1;
        b->max_n = std::max(b->max_n, (int)R.n);
    }
    if (natoms >= (int64_t)kIndexMask) {
        delete b;
        return bad(MD_ERR_CAPACITY, "more than 2^26 atoms in all");
    }
    b->total = natoms;
    const int cap = o.list_capacity > 0 ? o.list_capacity : std::max(16, ((int)std::ceil(1.25 * max_expect) + 8 + 3) & ~3);
    b->cap = cap;
    // order: costliest first
    std::vector<int> order_h(nrep);
    for (int r = 0; r < nrep; ++r) order_h[r] = r;
    std::stable_sort(order_h.begin(), order_h.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    if (o.cuda_stream) {
        b->stream = (cudaStream_t)o.cuda_stream;
    } else if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) == cudaSuccess) {
        b->own_stream = true;
    } else {
        delete b;
        return bad(MD_ERR_CUDA, "cannot create a stream");
    }
    Bufs<float> B{};
    const size_t N = (size_t)atom_off + kScreenPad;
    bool ok = true;
    for (int s = 0; s < 2; ++s)
        for (int a = 0; a < 3; ++a) ok = ok && balloc_n(b, B.xr[s][a], N) && balloc_n(b, B.v[s][a], N);
    for (int a = 0; a < 3; ++a)
        ok = ok && balloc_n(b, B.d[a], N) && balloc_n(b, B.xw[a], N) && balloc_n(b, B.uref[a], N) &&
             balloc_n(b, B.fcache[a], N);
    for (int s = 0; s < 2; ++s) ok = ok && balloc_n(b, B.id[s], N) && balloc_n(b, B.type[s], N) && balloc_n(b, B.shadow[s], N);
    ok = ok && balloc_n(b, B.cell, N) && balloc_n(b, B.cell_old, N) && balloc_n(b, B.slot, N) &&
         balloc_n(b, B.cell_atoms, N) && balloc_n(b, B.cell_ids, N) && balloc_n(b, B.screen[0], N) && balloc_n(b, B.type8, N) && balloc_n(b, B.nnb, N);
    ok = ok && balloc_n(b, B.count, (size_t)cell_off) && balloc_n(b, B.cell_start, (size_t)cs_off);
    ok = ok && balloc_n(b, B.list, (size_t)cap * (size_t)atom_off);
    size_t ncenter = 0;
    for (auto &R : b->rep) ncenter += (size_t)(R.G.ncell[0] + R.G.ncell[1] + R.G.ncell[2]);
    float4 *coef = nullptr, *coef2 = nullptr;
    Tables<float> *tab = nullptr;
    double *center = nullptr;
    int *order = nullptr;
    ok = ok && balloc_n(b, coef, rowsF.size() / 4) && balloc_n(b, coef2, rows2.size() / 4) &&
         balloc_n(b, tab, (size_t)npot) && balloc_n(b, center, ncenter) && balloc_n(b, b->rep_dev, (size_t)nrep) &&
         balloc_n(b, b->st, (size_t)nrep) && balloc_n(b, order, (size_t)nrep) && balloc_n(b, b->A.queue, 1) &&
         balloc_n(b, b->A.maxdisp, 2 * (size_t)nrep) && balloc_n(b, b->A.part, 3 * (size_t)kMaxTeam * nrep) &&
         balloc_n(b, b->stage, 9 * (size_t)b->max_n);
    if (!ok) {
        md_batch_destroy(b);
        return bad(MD_ERR_OOM, "device allocation failed");
    }
    // the replicas' views
    std::vector<double> centers(ncenter);
    size_t cen = 0;
    for (int r = 0; r < nrep; ++r) {
        Replica &R = b->rep[r];
        const Place &at = place[r];
        const int q = reps[r].potential;
        R.L.cap = cap;
        R.B = B;
        Bufs<float> &V = R.B;
        for (int a = 0; a < 3; ++a) {
            for (int s = 0; s < 2; ++s) {
                V.xr[s][a] += at.atom;
                V.v[s][a] += at.atom;
            }
            V.d[a] += at.atom;
            V.xw[a] += at.atom;
            V.uref[a] += at.atom;
            V.fcache[a] += at.atom;
            V.center[a] = center + cen;
            for (int k = 0; k < R.G.ncell[a]; ++k) centers[cen++] = ((double)k + 0.5) * R.G.h[a];
        }
        for (int s = 0; s < 2; ++s) {
            V.id[s] += at.atom;
            V.type[s] += at.atom;
            V.shadow[s] += at.atom;
        }
        V.cell += at.atom;
        V.cell_old += at.atom;
        V.slot += at.atom;
        V.cell_atoms += at.atom;
        V.cell_ids += at.atom;
        V.screen[0] += at.atom;
        V.type8 += at.atom;
        V.nnb += at.atom;
        V.count += at.cell;
        V.cell_start += at.cs;
        V.list += (size_t)cap * at.atom;
        const size_t nint = (size_t)tabs[q].fphi.nint;
        V.coef = coef;
        V.coef2 = coef2 + off2[q];
        V.coef_d = V.coef2 + 2 * nint;
        V.coef_f = V.coef2 + 4 * nint;
        V.tables = tab + q;
        V.st = b->st + r;
    }
    auto up4 = [](float4 *dst, const std::vector<double> &src) {
        std::vector<float4> t(src.size() / 4);
        for (size_t k = 0; k < t.size(); ++k)
            t[k] = make_float4((float)src[4 * k], (float)src[4 * k + 1], (float)src[4 * k + 2], (float)src[4 * k + 3]);
        return cudaMemcpy(dst, t.data(), t.size() * sizeof(float4), cudaMemcpyHostToDevice);
    };
    auto up = [](void *dst, const void *src, size_t bytes) { return cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice); };
    cudaError_t ce = up4(coef, rowsF);
    if (ce == cudaSuccess) ce = up4(coef2, rows2);
    if (ce == cudaSuccess) ce = up(tab, tabs.data(), sizeof(Tables<float>) * npot);
    if (ce == cudaSuccess) ce = up(center, centers.data(), sizeof(double) * ncenter);
    if (ce == cudaSuccess) ce = up(b->rep_dev, b->rep.data(), sizeof(Replica) * nrep);
    if (ce == cudaSuccess) ce = up(order, order_h.data(), sizeof(int) * nrep);
    if (ce == cudaSuccess) ce = cudaMemset(B.count, 0, sizeof(int) * (size_t)cell_off);
    if (ce == cudaSuccess) ce = cudaMemset(b->st, 0, sizeof(DevState) * (size_t)nrep);
    if (ce == cudaSuccess) ce = cudaMemset(b->A.maxdisp, 0, sizeof(unsigned) * 2 * (size_t)nrep);
    // the list build reads (and ignores) words between and after the replicas
    for (int a = 0; a < 3 && ce == cudaSuccess; ++a) ce = cudaMemset(B.uref[a], 0, sizeof(float) * N);
    if (ce == cudaSuccess) ce = cudaMemset(B.screen[0], 0, sizeof(float) * N);
    for (int s = 0; s < 2 && ce == cudaSuccess; ++s) ce = cudaMemset(B.type[s], 0, sizeof(int) * N);
    for (int a = 0; a < 3 && ce == cudaSuccess; ++a) ce = cudaMemset(B.d[a], 0, sizeof(double) * N);
    if (ce == cudaSuccess) ce = cudaMallocHost((void **)&b->st_host, sizeof(DevState) * nrep);
    if (ce == cudaSuccess)
        ce = cudaMallocHost((void **)&b->host_stage, sizeof(double) * 9 * (size_t)std::min(b->max_n, kBatchStageAtoms));
    // the replicas' states, caller order within each replica
    {
        std::vector<double> x(N, 0.0);
        for (int k = 0; k < 6 && ce == cudaSuccess; ++k) {
            const int a = k % 3;
            for (int r = 0; r < nrep; ++r) {
                const double *src = k < 3 ? reps[r].pos : reps[r].vel;
                double *dst = x.data() + place[r].atom;
                for (int64_t i = 0; i < reps[r].n; ++i) dst[i] = src ? src[3 * i + a] : 0.0;
            }
            ce = up(k < 3 ? B.xr[0][a] : B.v[0][a], x.data(), sizeof(double) * N);
        }
        std::vector<int> id(N, 0);
        for (int r = 0; r < nrep; ++r)
            for (int64_t i = 0; i < reps[r].n; ++i) id[place[r].atom + i] = (int)i;
        if (ce == cudaSuccess) ce = up(B.id[0], id.data(), sizeof(int) * N);
    }
    if (ce != cudaSuccess) {
        md_batch_destroy(b);
        return bad(MD_ERR_CUDA, std::string("upload: ") + cudaGetErrorString(ce));
    }
    b->A.rep = b->rep_dev;
    b->A.order = order;
    b->A.nrep = nrep;
    b->schedule = 0;
    b->grid = batch_grid(0, nrep);
    md_status rc = batch_launch(b, BATCH_INIT, 1, 0.0);
    if (rc == MD_OK) rc = batch_sync(b);
    // schedule autotuner: right after the initial build every replica is
    // rebuild_every steps from its next build, so rebuild_every - 1 steps of
    // dt = 0 change nothing but the counters, which are restored afterwards
    if (rc == MD_OK && o.batch_schedule > 0) {
        b->schedule = o.batch_schedule - 1;
        b->grid = batch_grid(b->schedule, nrep);
    } else if (rc == MD_OK && o.rebuild_every > 1 && o.lanes_per_atom == 0) {
        const int trial = std::min(o.rebuild_every - 1, 8);
        int sms = 152, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const BatchKey key{dev, nrep, b->max_n, cap, o.rebuild_every, natoms, cell_off};
        int best_s = -1;
        {
            std::lock_guard<std::mutex> lock(g_batch_mu);
            for (auto &e : g_batch_cache)
                if (e.first == key && batch_grid(e.second, nrep) > 0) best_s = e.second;
        }
        const bool known = best_s >= 0;
        if (!known) best_s = 0;
        float best = 1e30f;
        cudaEvent_t t0, t1;
        cudaEventCreate(&t0);
        cudaEventCreate(&t1);
        const std::vector<DevState> saved(b->st_host, b->st_host + nrep);
        for (int round = known ? 2 : 0; round < 2 && rc == MD_OK; ++round)
            for (int sc = 0; sc < kNumSchedules && rc == MD_OK; ++sc) {
                // teams where they can fill SMs that single blocks leave idle
                // or late: up to 4 replicas per SM for pairs, 1 for more
                const int team = kSchedules[sc].team;
                if (team > 1 && nrep > (team == 2 ? 4 * sms : sms)) continue;
                const int grid = batch_grid(sc, nrep);
                if (grid <= 0) continue;
                b->schedule = sc;
                b->grid = grid;
                cudaEventRecord(t0, b->stream);
                rc = batch_launch(b, BATCH_RUN, trial, 0.0);
                cudaEventRecord(t1, b->stream);
                if (rc == MD_OK) rc = batch_sync(b);
                float ms = 0;
                cudaEventElapsedTime(&ms, t0, t1);
                // a later shape must win by 3 %
                if (round == 1 && ms < 0.97f * best) {
                    best = ms;
                    best_s = sc;
                }
                // back to the state after the initial build
                b->st_current = false;
                if (rc == MD_OK && cudaMemcpy(b->st, saved.data(), sizeof(DevState) * nrep, cudaMemcpyHostToDevice) != cudaSuccess)
                    rc = MD_ERR_CUDA;
            }
        cudaEventDestroy(t0);
        cudaEventDestroy(t1);
        b->schedule = best_s;
        b->grid = batch_grid(best_s, nrep);
        b->launches = 1;
        if (!known && rc == MD_OK) {
            std::lock_guard<std::mutex> lock(g_batch_mu);
            if (g_batch_cache.size() < kBatchCacheMax) g_batch_cache.push_back({key, best_s});
        }
    }
    if (rc == MD_OK) rc = batch_sync(b);
    if (rc != MD_OK) {
        g_batch_create_error = b->err;
        md_batch_destroy(b);
        return rc;
    }
    b->chosen = b->schedule;
    // rebuild counters start after the initial build
    for (int r = 0; r < nrep; ++r) b->st_host[r].rebuilds = 0;
    b->st_current = false;
    if (cudaMemcpy(b->st, b->st_host, sizeof(DevState) * nrep, cudaMemcpyHostToDevice) != cudaSuccess) {
        md_batch_destroy(b);
        return bad(MD_ERR_CUDA, "state upload failed");
    }
    *out = b;
    return MD_OK;
}

md_status md_batch_step(md_batch *b, int64_t nsteps, double dt)
{
    if (!b) return MD_ERR_ARG;
    if (nsteps < 0 || nsteps > (int64_t)1 << 30 || !std::isfinite(dt)) return b->fail(MD_ERR_ARG, "bad nsteps or dt");
    if (nsteps == 0) return MD_OK;
    b->replayable = b->replayable || is_capturing(b->stream);
    if (!b->opt.use_graphs) return batch_launch(b, BATCH_RUN, (int)nsteps, dt);
    for (auto &g : b->graphs)
        if (g.nsteps == (int)nsteps && g.dt == dt) {
            b->st_current = false;
            BCK(cudaGraphLaunch(g.e, b->stream));
            b->launches += 1;
            return MD_OK;
        }
    cudaStream_t cs;
    BCK(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaStream_t keep = b->stream;
    b->stream = cs;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    md_status rc = (e == cudaSuccess) ? batch_launch(b, BATCH_RUN, (int)nsteps, dt) : MD_ERR_CUDA;
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(cs, &g);
    b->stream = keep;
    b->launches -= 1;
    cudaStreamDestroy(cs);
    if (e != cudaSuccess || e2 != cudaSuccess || rc != MD_OK) return b->fail(MD_ERR_CUDA, "graph capture failed");
    cudaGraphExec_t ex;
    BCK(cudaGraphInstantiate(&ex, g, 0));
    b->graphs.push_back({(int)nsteps, dt, g, ex});
    b->st_current = false;
    BCK(cudaGraphLaunch(ex, b->stream));
    b->launches += 1;
    return MD_OK;
}

md_status md_batch_energy(md_batch *b, double *pe, double *ke)
{
    if (!b) return MD_ERR_ARG;
    md_status rc = batch_sync(b);
    if (rc != MD_OK) return rc;
    for (int r = 0; r < b->nrep; ++r) {
        if (pe) pe[r] = b->st_host[r].e_embed + b->st_host[r].e_pair;
        if (ke) ke[r] = b->st_host[r].ke;
    }
    return MD_OK;
}

md_status md_batch_get_state(md_batch *b, int32_t r, double *pos, double *vel, double *force)
{
    if (!b) return MD_ERR_ARG;
    if (r < 0 || r >= b->nrep) return b->fail(MD_ERR_ARG, "replica index out of range");
    md_status rc = batch_sync(b);
    if (rc != MD_OK) return rc;
    const size_t n = (size_t)b->rep[r].L.n;
    // gathered on the device, one copy to pinned memory, then into the
    // caller's arrays (a copy per array into pageable memory took 230 us a
    // replica of 5,900 atoms)
    double *out[3] = {pos, vel, force}, *at[3] = {nullptr, nullptr, nullptr};
    size_t len = 0;
    for (int k = 0; k < 3; ++k)
        if (out[k]) {
            at[k] = b->stage + len;
            len += 3 * n;
        }
    if (len == 0) return MD_OK;
    k_batch_store<<<(int)((n + 255) / 256), 256, 0, b->stream>>>(b->rep_dev, r, at[0], at[1], at[2]);
    b->launches += 1;
    BCK(cudaGetLastError());
    if (n > (size_t)kBatchStageAtoms) {
        for (int k = 0; k < 3; ++k)
            if (out[k])
                BCK(cudaMemcpyAsync(out[k], at[k], sizeof(double) * 3 * n, cudaMemcpyDeviceToHost, b->stream));
        BCK(cudaStreamSynchronize(b->stream));
        return MD_OK;
    }
    BCK(cudaMemcpyAsync(b->host_stage, b->stage, sizeof(double) * len, cudaMemcpyDeviceToHost, b->stream));
    BCK(cudaStreamSynchronize(b->stream));
    for (int k = 0; k < 3; ++k)
        if (out[k]) memcpy(out[k], b->host_stage + (at[k] - b->stage), sizeof(double) * 3 * n);
    return MD_OK;
}

md_status md_batch_info(md_batch *b, md_batch_info_t *out)
{
    if (!b || !out) return b ? b->fail(MD_ERR_ARG, "out is NULL") : MD_ERR_ARG;
    md_status rc = batch_sync(b);
    if (rc != MD_OK) return rc;
    memset(out, 0, sizeof(*out));
    out->replicas = b->nrep;
    out->atoms = b->total;
    out->blocks = b->grid;
    out->threads_per_block = kSchedules[b->schedule].block;
    out->list_capacity = b->cap;
    out->kernel_launches = b->launches;
    out->blocks_per_replica = kSchedules[b->schedule].team;
    for (int r = 0; r < b->nrep; ++r) {
        out->rebuilds += b->st_host[r].rebuilds;
        out->max_neighbors = std::max(out->max_neighbors, b->st_host[r].max_nnb);
        out->steps = std::max<int64_t>(out->steps, b->st_host[r].step);
    }
    return MD_OK;
}

md_status md_batch_set_schedule(md_batch *b, int32_t schedule)
{
    if (!b) return MD_ERR_ARG;
    if (schedule < 0 || schedule > kNumSchedules) return b->fail(MD_ERR_ARG, "schedule must be 0..8");
    const int sched = schedule == 0 ? b->chosen : schedule - 1;
    const int grid = batch_grid(sched, b->nrep);
    if (grid <= 0) return b->fail(MD_ERR_CUDA, "the launch shape cannot be resident");
    if (sched == b->schedule) return MD_OK;
    BCK(cudaStreamSynchronize(b->stream));
    batch_drop_graphs(b);  // captured with the other shape
    b->schedule = sched;
    b->grid = grid;
    return MD_OK;
}

const char *md_batch_last_error(const md_batch *b) { return b ? b->err.c_str() : g_batch_create_error.c_str(); }

void md_batch_destroy(md_batch *b)
{
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    batch_drop_graphs(b);
    for (void *p : b->allocs) {
        if (b->opt.free) b->opt.free(p, b->opt.alloc_ctx);
        else cudaFree(p);
    }
    if (b->st_host) cudaFreeHost(b->st_host);
    if (b->host_stage) cudaFreeHost(b->host_stage);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
}

}  // extern "C"
