// pair_kernels.cuh -- the density and force passes of the EAM timestep.
//
// Atom-parallel schedule (k_density, k_force): TPA lanes cooperate on one
// atom; lane l walks list columns l, l+TPA, ... a few at a time (every
// gather of a round issued before any is used: three pairs a round in the
// density pass, two in the force pass with the next round in flight), and
// the lanes' sums meet by warp shuffles.  Neighbour records and spline rows
// are gathered from global memory through L1.
// The neighbour record is the 16-byte shadow (u_x, u_y, u_z, F'_j): one
// gather gives the force pass both the position and the embedding derivative
// the density pass stored.  With one atom type whose f and phi share a knot
// grid, both splines of an interval sit in one 32-byte row (coef2), read with
// one 256-bit load.
#pragma once

#include "device_common.cuh"

#include <type_traits>

namespace eammd {
namespace {

// Kinds of spline tables: one type whose f and phi share a knot grid; any
// tables; several types whose f and phi all share one grid.
enum TableKind { KIND_ONE = 0, KIND_ANY = 1, KIND_TYPES = 2 };

template <class R> struct PairIn {
    R dx, dy, dz, r2;
};

template <class R>
__device__ __forceinline__ PairIn<R> pair_vector(const typename V4<R>::T &ui, const typename V4<R>::T &uj,
                                                 const Shift<R> &shf)
{
    PairIn<R> p;
    p.dx = (uj.x - ui.x) + shf.x;
    p.dy = (uj.y - ui.y) + shf.y;
    p.dz = (uj.z - ui.z) + shf.z;
    p.r2 = fma(p.dz, p.dz, fma(p.dy, p.dy, p.dx * p.dx));
    return p;
}

// Pair vector and squared distance in FP64 from the atom's own coordinates
// shifted into the neighbour's cell (one addition per component less than
// u_j - u_i + shift; the three candidates per axis are formed once per atom).
template <class R> struct Own {
    typename V4<R>::T u;
    R h[3];
    __device__ __forceinline__ Own(const typename V4<R>::T &ui, const R (&hh)[3]) : u(ui), h{hh[0], hh[1], hh[2]} {}
    __device__ __forceinline__ PairIn<R> to(const typename V4<R>::T &uj, uint32_t e) const
    {
        return pair_vector<R>(u, uj, entry_shift<R>(e, h));
    }
};
template <> struct Own<double> {
    double x[3], y[3], z[3];
    __device__ __forceinline__ Own(const double4_32a &u, const double (&h)[3])
        : x{u.x + h[0], u.x, u.x - h[0]}, y{u.y + h[1], u.y, u.y - h[1]}, z{u.z + h[2], u.z, u.z - h[2]}
    {
    }
    static __device__ __forceinline__ double pick(const double (&v)[3], uint32_t t)
    {
        return t == 1u ? v[1] : (t == 0u ? v[0] : v[2]);
    }
    __device__ __forceinline__ PairIn<double> to(const double4_32a &uj, uint32_t e) const
    {
        const uint32_t c = e >> kCodeShift;
        PairIn<double> p;
        p.dx = uj.x - pick(x, c & 3u);
        p.dy = uj.y - pick(y, (c >> 2) & 3u);
        p.dz = uj.z - pick(z, c >> 4);
        p.r2 = fma(p.dz, p.dz, fma(p.dy, p.dy, p.dx * p.dx));
        return p;
    }
};

// r2 < rc2 for a non-negative r2 (or NaN: false).  Non-negative doubles order
// as their bits, which keeps the comparison off the FP64 pipe.
__device__ __forceinline__ bool within(float r2, float rc2) { return r2 < rc2; }
__device__ __forceinline__ bool within(double r2, double rc2)
{
    return (unsigned long long)__double_as_longlong(r2) < (unsigned long long)__double_as_longlong(rc2);
}

// Both 16-byte halves of a 32-byte fused row with one 256-bit load.
template <class R>
__device__ __forceinline__ void load_row2(const typename V4<R>::T *row, typename V4<R>::T &a, typename V4<R>::T &b);
template <>
__device__ __forceinline__ void load_row2<float>(const float4 *row, float4 &a, float4 &b)
{
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(row));
}
template <>
__device__ __forceinline__ void load_row2<double>(const double4_32a *row, double4_32a &a, double4_32a &b)
{
    a = row[0];
    b = row[1];
}

template <int TPA, class T>
__device__ __forceinline__ T lane_sum(T v)
{
#pragma unroll
    for (int o = TPA / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Where a list entry's neighbour record is read from.
template <class R>
struct GlobalFetch {
    const typename V4<R>::T *sw;
    __device__ __forceinline__ typename V4<R>::T operator()(uint32_t e) const { return sw[e & kIndexMask]; }
};

// The same, through the texture path (FP32 records, density pass).
struct TexFetch {
    cudaTextureObject_t t;
    __device__ __forceinline__ float4 operator()(uint32_t e) const
    {
        return tex1Dfetch<float4>(t, (int)(e & kIndexMask));
    }
};

// Where the spline rows of the one-type path are read from: coef2 in device
// memory (row 2k: f, row 2k+1: phi, both in one 32-byte load); the density
// pass reads the f rows alone from coef_f, where a 128-byte line holds eight
// intervals instead of four; the force pass without energies reads coef_d,
// the rows of f' and phi' (b, 2c, 3d of each, six of a row's eight words).
template <class R>
struct TabGlobal {
    const typename V4<R>::T *coef2;
    const typename V4<R>::T *coef_f;  // f rows alone: more intervals per cache line
    const typename V4<R>::T *coef_d;  // f' and phi' rows (of a type pair: slopes_types)
    const uint8_t *type8;             // types of the atoms, where there are several
    __device__ __forceinline__ explicit TabGlobal(const Bufs<R> &B)
        : coef2(B.coef2), coef_f(B.coef_f), coef_d(B.coef_d), type8(B.type8)
    {
    }
    // interval of r (tables of up to kMaxFusedIntervals intervals)
    __device__ __forceinline__ int interval(const SplineDesc<R> &g, R r, R &t) const { return segment_fused(g, r, t); }
    __device__ __forceinline__ typename V4<R>::T f(int kk) const { return coef_f[kk]; }
    __device__ __forceinline__ void fphi(int kk, typename V4<R>::T &cf, typename V4<R>::T &cp) const
    {
        load_row2<R>(coef2 + 2 * kk, cf, cp);
    }
    // f' of types ti and tj and phi' of the pair at t, row kk of the nint of
    // each type pair: 16 words, nine in use (b, 2c, 3d of f_a, f_b and phi,
    // a <= b), by one 256-bit load and one word
    __device__ __forceinline__ void slopes_types(int ntypes, int nint, int ti, int tj, int kk, R t, R &fi, R &fj,
                                                 R &pd) const
    {
        typename V4<R>::T a, b;
        const typename V4<R>::T *row = coef_d + 4 * ((size_t)pair_index(ntypes, ti, tj) * nint + kk);
        load_row2<R>(row, a, b);
        const R p3 = reinterpret_cast<const R *>(row)[8];
        const R fa = fma(t, fma(t, a.z, a.y), a.x), fb = fma(t, fma(t, b.y, b.x), a.w);
        fi = ti <= tj ? fa : fb;
        fj = ti <= tj ? fb : fa;
        pd = fma(t, fma(t, p3, b.w), b.z);
    }
    // f' and phi' at t
    __device__ __forceinline__ void slopes(int kk, R t, R &fd, R &pd) const
    {
        typename V4<R>::T a, b;
        load_row2<R>(coef_d + 2 * kk, a, b);
        fd = fma(t, fma(t, a.z, a.y), a.x);
        pd = fma(t, fma(t, b.y, b.x), a.w);
    }
};
// Where list column k of the lane's atom is read from.
struct ListGlobal {
    const uint32_t *lp;  // list + i
    int ld;
    __device__ __forceinline__ uint32_t operator()(int k) const { return lp[(size_t)k * ld]; }
};
__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---- FP64: the listed pairs that are in range, compacted before the FP64 work
//
// An FP64 instruction takes its 16 cycles of the SM's pipe whether one lane of
// the warp needs it or all: with 14 of 26 listed pairs in range (BCC), nearly
// every column had some lane in range and cost every FP64 operation of a pair.
// So the columns are first tested in FP32 (records rounded to FP32, a margin
// for their rounding), the entries that may be in range go to shared memory
// one behind the other, and the FP64 passes walk those, exact test included.
// With several lanes per atom the entries found are dealt out anew over the
// lanes.  The order of an atom's entries is that of its list.
// 799,496 BCC atoms: density 760 -> 484 us, force 1,267 -> 681 us; the FP64
// operations alone take about 440 and 580 us of the pipe.
constexpr int kCompactColumns = 32;  // list columns taken at a time

// Bytes of shared memory a block of the pair passes needs.
template <class R>
constexpr size_t compact_bytes(int block, int tpa)
{
    return sizeof(R) == 8 ? sizeof(uint32_t) * kCompactColumns * (size_t)(block / tpa) : 0;
}

extern __shared__ uint32_t compact_smem[];

// Entry k of the compacted columns of the lane's atom.
struct ListCompact {
    const uint32_t *p;  // compact_smem + atom of the block
    int width;          // atoms of the block
    __device__ __forceinline__ uint32_t operator()(int k) const { return p[k * width]; }
};

// Upper bound of r_cut^2 in FP32 for the atom at u: with m the sum of the
// records' sizes (a partner in range is at most a shift and r_cut farther from
// its cell's centre), the pair vector is rounded by at most d = 2 m 2^-24 and
// r^2 by 2 r d + d^2; the margin is 2.5 times that and more, so that no pair in
// range is missed however far outside an open box.
__device__ __forceinline__ float compact_bound(const Geom &G, const float4 &u)
{
    const float rc = sqrtf(G.rc2_f);
    const float m = fabsf(u.x) + fabsf(u.y) + fabsf(u.z) + 2.f * (G.h_f[0] + G.h_f[1] + G.h_f[2]) + 6.f * rc;
    const float s = 0x1p-24f * m;
    return G.rc2_f + (s * (10.f * rc + 16.f * s) + 0x1p-20f * G.rc2_f);
}

// Entries of columns [k0, min(k0 + kCompactColumns, nn)) of the lane's atom
// that may be in range, to shared memory; returns their number.  All lanes of
// the warp must call (nn = 0 without an atom).
template <int TPA, class List>
__device__ __forceinline__ int compact_columns(const Geom &G, const float4 *rec, const float4 &ui, float bound, int k0,
                                               int nn, int l, const List &list, uint32_t *buf, int width)
{
    constexpr int U = 4;  // columns in flight per lane
    const float h[3] = {G.h_f[0], G.h_f[1], G.h_f[2]};
    const int k1 = min(k0 + kCompactColumns, nn);
    const unsigned lane = threadIdx.x & 31u;
    const unsigned group = TPA == 1 ? 0u : ((TPA == 32 ? 0u : (1u << (TPA & 31))) - 1u) << (lane & ~(unsigned)(TPA - 1));
    const unsigned before = (1u << lane) - 1u;
    // the warp's lanes go round together where they exchange their finds
    const int kend = TPA == 1 ? k1 : (int)__reduce_max_sync(0xffffffffu, (unsigned)max(k1, 0));
    int cnt = 0;
    for (int k = k0; k < kend; k += U * TPA) {
        uint32_t e[U];
        float4 u[U];
#pragma unroll
        for (int q = 0; q < U; ++q) e[q] = (k + l + q * TPA < k1) ? list(k + l + q * TPA) : 0u;
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = (k + l + q * TPA < k1) ? rec[e[q] & kIndexMask] : ui;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const PairIn<float> p = pair_vector<float>(ui, u[q], entry_shift<float>(e[q], h));
            const bool in = (k + l + q * TPA < k1) && !(p.r2 > bound);  // (an overflow too)
            if (TPA == 1) {
                if (in) buf[cnt * width] = e[q];
                cnt += in ? 1 : 0;
            } else {
                const unsigned m = __ballot_sync(0xffffffffu, in) & group;
                if (in) buf[(cnt + __popc(m & before)) * width] = e[q];
                cnt += __popc(m);
            }
        }
    }
    __syncwarp();
    return cnt;
}

// This lane's part of rho_i = sum over listed j with r < r_cut of f_{t_j}(r_ij)
// (Eq. 2).
// In the force pass the list columns of the first round are read before the
// neighbour count is known (every column below cap lies inside the list);
// while a round is computed, the next round's records and the columns of the
// round after are in flight.  Columns at or beyond nn never address a record.
template <class R, int KIND, int TPA, int U, class List, class Fetch, class Tab>
__device__ __forceinline__ R density_lane(const Bufs<R> &B, const R (&h)[3], R rc2, int s, const int *nnb_i,
                                          int cap, int l, const typename V4<R>::T &ui, const List &list,
                                          const Fetch &fetch, const Tab &tab, R rho = (R)0)
{
    using R4 = typename V4<R>::T;
    const Tables<R> &T = *B.tables;
    const SplineDesc<R> g = T.fphi;
    const Own<R> own(ui, h);
    // Many lanes per atom (small systems, bound by latency): the columns of
    // the first round are read before the neighbour count is known, as in the
    // force pass.  With few lanes the registers cost more than the wait.
    constexpr bool kEarly = TPA >= 4;
    uint32_t e[U];
    if (kEarly) {
#pragma unroll
        for (int q = 0; q < U; ++q) e[q] = (l + q * TPA < cap) ? list(l + q * TPA) : 0u;
    }
    const int nn = *nnb_i;
    // U pairs per round (columns k, k + TPA, ...), all gathers issued before
    // any is used; the sum runs in column order
    for (int k = l; k < nn; k += U * TPA) {
        if (!kEarly || k != l) {
#pragma unroll
            for (int q = 0; q < U; ++q) e[q] = (k + q * TPA < nn) ? list(k + q * TPA) : 0u;
        }
        R4 u[U];
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = fetch(q == 0 || k + q * TPA < nn ? e[q] : e[0]);
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const PairIn<R> p = own.to(u[q], e[q]);
            if ((q == 0 || k + q * TPA < nn) && within(p.r2, rc2)) {
                R rinv, r;
                inv_r(p.r2, rinv, r);
                if (KIND == KIND_ANY) {
                    R val, der;
                    const int j = (int)(e[q] & kIndexMask);
                    spline_r(T.f[B.type[s][j]], B.coef, r, val, der);
                    rho += val;
                } else {
                    R t;
                    int kk = tab.interval(g, r, t);
                    if (KIND == KIND_TYPES) kk += (int)tab.type8[e[q] & kIndexMask] * g.nint;
                    const R4 c = tab.f(kk);
                    rho += fma(t, fma(t, fma(t, c.w, c.z), c.y), c.x);
                }
            }
        }
    }
    return rho;
}

// F'(rho_i) into the atom's record (w word) and F(rho_i) for the energy.
template <class R>
__device__ __forceinline__ R embed(const Bufs<R> &B, typename V4<R>::T *sw, int i, int ti, R rho)
{
    const Tables<R> &T = *B.tables;
    R Fv, Fd;
    if (spline_any(T.F[ti], B.coef, rho, Fv, Fd)) atomicAdd(&B.st->table_oor, 1ull);
    // the force pass reads w with the coordinates; the density pass never does
    reinterpret_cast<R *>(sw + i)[3] = Fd;
    return Fv;
}

// This lane's part of the force of Eq. 4,
//   s_ij = phi'_{t_i t_j}(r) + F'_i f'_{t_j}(r) + F'_j f'_{t_i}(r),
//   F_i  = sum_j s_ij (x_j - x_i) / r,
// and, when ENERGY, of the pair energy and the virial (e7: pair energy, then
// W xx yy zz xy xz yz).
template <class R, int KIND, bool ENERGY, int TPA, int U, class List, class Fetch, class Tab>
__device__ __forceinline__ void force_lane(const Bufs<R> &B, const Launch &L, const R (&h)[3], R rc2,
                                           int s, const int *nnb_i, int cap, int l, int ti,
                                           const typename V4<R>::T &ui, const List &list, const Fetch &fetch, R (&f)[3], R (&e7)[7],
                                           const Tab &tab)
{
    using R4 = typename V4<R>::T;
    const Tables<R> &T = *B.tables;
    const SplineDesc<R> g = T.fphi;
    const R Fpi = ui.w;
    const Own<R> own(ui, h);
    constexpr int W = U * TPA;  // columns per round
    uint32_t e[U], en[U];
    R4 u[U];
#pragma unroll
    for (int q = 0; q < U; ++q) e[q] = (l + q * TPA < cap) ? list(l + q * TPA) : 0u;
    const int nn = *nnb_i;
#pragma unroll
    for (int q = 0; q < U; ++q) en[q] = (l + W + q * TPA < nn) ? list(l + W + q * TPA) : 0u;
#pragma unroll
    for (int q = 0; q < U; ++q) u[q] = (l < nn) ? fetch(q == 0 || l + q * TPA < nn ? e[q] : e[0]) : ui;
    for (int k = l; k < nn; k += W) {
        // in flight while this round is computed: the next round's records
        // and the columns of the round after
        const int k1 = k + W;
        R4 un[U];
        uint32_t e2[U];
#pragma unroll
        for (int q = 0; q < U; ++q) un[q] = (k1 < nn) ? fetch(q == 0 || k1 + q * TPA < nn ? en[q] : en[0]) : ui;
#pragma unroll
        for (int q = 0; q < U; ++q) e2[q] = (k1 + W + q * TPA < nn) ? list(k1 + W + q * TPA) : 0u;
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const PairIn<R> p = own.to(u[q], e[q]);
            if ((q == 0 || k + q * TPA < nn) && within(p.r2, rc2)) {
                R rinv, r;
                inv_r(p.r2, rinv, r);
                const R Fpj = u[q].w;
                R phv, phd, fdj, fdi;
                if (KIND == KIND_TYPES) {
                    static_assert(KIND != KIND_TYPES || !ENERGY, "energies take the general kernels");
                    R t;
                    const int kk = tab.interval(g, r, t);
                    tab.slopes_types(L.ntypes, g.nint, ti, (int)tab.type8[e[q] & kIndexMask], kk, t, fdi, fdj, phd);
                    phv = (R)0;
                } else if (KIND == KIND_ANY) {
                    const int j = (int)(e[q] & kIndexMask);
                    const int tj = B.type[s][j];
                    spline_r(T.phi[pair_index(L.ntypes, ti, tj)], B.coef, r, phv, phd);
                    fdj = spline_r_der(T.f[tj], B.coef, r);
                    fdi = (tj == ti) ? fdj : spline_r_der(T.f[ti], B.coef, r);
                } else {
                    R t;
                    const int kk = tab.interval(g, r, t);
                    if (ENERGY) {
                        R4 cf, cp;
                        tab.fphi(kk, cf, cp);
                        fdj = fma(t, fma(t, (R)3 * cf.w, (R)2 * cf.z), cf.y);
                        phd = fma(t, fma(t, (R)3 * cp.w, (R)2 * cp.z), cp.y);
                        phv = fma(t, fma(t, fma(t, cp.w, cp.z), cp.y), cp.x);
                    } else {
                        tab.slopes(kk, t, fdj, phd);
                        phv = (R)0;
                    }
                    fdi = fdj;
                }
                const R sij = fma(Fpj, fdi, fma(Fpi, fdj, phd));
                const R sr = sij * rinv;
                f[0] = fma(sr, p.dx, f[0]);
                f[1] = fma(sr, p.dy, f[1]);
                f[2] = fma(sr, p.dz, f[2]);
                if (ENERGY) {
                    const R hs = (R)(-0.5) * sr;
                    e7[0] += (R)0.5 * phv;
                    e7[1] = fma(hs * p.dx, p.dx, e7[1]);
                    e7[2] = fma(hs * p.dy, p.dy, e7[2]);
                    e7[3] = fma(hs * p.dz, p.dz, e7[3]);
                    e7[4] = fma(hs * p.dx, p.dy, e7[4]);
                    e7[5] = fma(hs * p.dx, p.dz, e7[5]);
                    e7[6] = fma(hs * p.dy, p.dz, e7[6]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            e[q] = en[q];
            en[q] = e2[q];
            u[q] = un[q];
        }
    }
}

// Integration of Eq. 5 for the components this lane owns (c = l, l + TPA,
// ... < 3) once the lanes' forces are summed: MODE_CLOSE* applies the closing
// half kick v += F dt/(2m); MODE_CLOSE_OPEN also the next step's opening
// half kick and the drift x += v dt, writing the next record and the
// displacement since the last list build; MODE_MEASURE only stores F.
template <class R, int MODE, bool ENERGY, int TPA>
__device__ __forceinline__ void integrate(const Bufs<R> &B, const Launch &L, int s, int sp, int i, int l, int ti,
                                          const R (&f)[3], double &ke, float &d2)
{
    if (l == 0 && !isfinite(f[0] + f[1] + f[2])) atomicOr(&B.st->error, ERR_NONFINITE);
    const double kq = L.half_kick[ti];
    for (int c = l; c < 3; c += TPA) {
        const R fc = (c == 0) ? f[0] : ((c == 1) ? f[1] : f[2]);
        if (MODE == MODE_MEASURE || MODE == MODE_CLOSE) B.fcache[c][i] = fc;
        double v = B.v[s][c][i];
        if (MODE != MODE_MEASURE) {
            if (std::is_same<R, float>::value && MODE == MODE_CLOSE_OPEN && !ENERGY) {
                // both half kicks at once: 2 (F dt/(2m)) is exact in FP32
                v += (double)((R)2 * (fc * (R)kq));
            } else {
                v = fma((double)fc, kq, v);
            }
        }
        if (ENERGY) ke += L.ke_factor[ti] * v * v;
        if (MODE == MODE_CLOSE_OPEN && (ENERGY || !std::is_same<R, float>::value)) v = fma((double)fc, kq, v);
        if (MODE != MODE_MEASURE) B.v[s][c][i] = v;
        if (MODE == MODE_CLOSE_OPEN) {
            const double dn = fma(v, L.dt, B.d[c][i]);
            B.d[c][i] = dn;
            const R u = B.uref[c][i] + (R)dn;
            reinterpret_cast<R *>(B.shadow[sp ^ 1] + i)[c] = u;
            if constexpr (sizeof(R) == 8) reinterpret_cast<float *>(B.rec32[sp ^ 1] + i)[c] = (float)u;
            const float gc = (float)dn;
            d2 += gc * gc;
        }
    }
}

template <class R, bool ENERGY>
__device__ __forceinline__ void force_block_end(const Bufs<R> &B, const Launch &L, const R (&e7)[7], double ke,
                                                float d2max, bool open)
{
    if (ENERGY) {
        // the kinetic energy is formed in FP64 and carried as a pair of R
        const R ke_hi = (R)ke;
        const R ke_lo = (R)(ke - (double)ke_hi);
        const R v8[8] = {e7[0], ke_hi, e7[1], e7[2], e7[3], e7[4], e7[5], e7[6]};
        const R lo8[8] = {0, ke_lo, 0, 0, 0, 0, 0, 0};
        block_sums_t<8, R>(v8, B.partials, L.pstride, 1, lo8);
    }
    if (open) block_max_disp(d2max, &B.st->maxdisp2);
}

// The atom's density and force sums over its whole list: FP32 walks the list,
// FP64 its columns in range.  All lanes of the warp must call; `active`: the
// lane has an atom.
template <class R, int KIND, int TPA, int U, class Fetch, class Tab>
__device__ __forceinline__ R density_atom(const Bufs<R> &B, const Geom &G, const Launch &L, const R (&h)[3], R rc2, int s,
                                          int sp, int i, int l, bool active, const Fetch &fetch, const Tab &tab)
{
    const ListGlobal list{B.list + i, L.ld};
    if constexpr (sizeof(R) == 8) {
        const int width = blockDim.x / TPA;
        uint32_t *buf = compact_smem + threadIdx.x / TPA;
        const int nn = active ? B.nnb[i] : 0;
        const typename V4<R>::T ui = active ? B.shadow[sp][i] : mk4<R>(0, 0, 0, 0);
        const float4 uf = active ? B.rec32[sp][i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float bound = compact_bound(G, uf);
        const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)nn);
        R rho = (R)0;
        for (int k0 = 0; k0 < most; k0 += kCompactColumns) {
            const int cnt = compact_columns<TPA>(G, B.rec32[sp], uf, bound, k0, nn, l, list, buf, width);
            rho = density_lane<R, KIND, TPA, U>(B, h, rc2, s, &cnt, cnt, l, ui, ListCompact{buf, width}, fetch, tab,
                                                 rho);
            __syncwarp();  // the buffer is free for the next columns
        }
        return rho;
    } else {
        return active ? density_lane<R, KIND, TPA, U>(B, h, rc2, s, B.nnb + i, L.cap, l, B.shadow[sp][i], list, fetch,
                                                       tab)
                      : (R)0;
    }
}

template <class R, int KIND, bool ENERGY, int TPA, int U, class Fetch, class Tab>
__device__ __forceinline__ void force_atom(const Bufs<R> &B, const Geom &G, const Launch &L, const R (&h)[3], R rc2,
                                           int s, int sp, int i, int l, int ti, bool active, const Fetch &fetch,
                                           R (&f)[3], R (&e7)[7], const Tab &tab)
{
    const ListGlobal list{B.list + i, L.ld};
    if constexpr (sizeof(R) == 8) {
        const int width = blockDim.x / TPA;
        uint32_t *buf = compact_smem + threadIdx.x / TPA;
        const int nn = active ? B.nnb[i] : 0;
        const typename V4<R>::T ui = active ? B.shadow[sp][i] : mk4<R>(0, 0, 0, 0);
        const float4 uf = active ? B.rec32[sp][i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float bound = compact_bound(G, uf);
        const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)nn);
        for (int k0 = 0; k0 < most; k0 += kCompactColumns) {
            const int cnt = compact_columns<TPA>(G, B.rec32[sp], uf, bound, k0, nn, l, list, buf, width);
            force_lane<R, KIND, ENERGY, TPA, U>(B, L, h, rc2, s, &cnt, cnt, l, ti, ui, ListCompact{buf, width}, fetch, f,
                                                 e7, tab);
            __syncwarp();
        }
    } else if (active) {
        force_lane<R, KIND, ENERGY, TPA, U>(B, L, h, rc2, s, B.nnb + i, L.cap, l, ti, B.shadow[sp][i], list, fetch, f,
                                             e7, tab);
    }
}

// ---- L2 prefetch of a warp's streams ----

__device__ __forceinline__ void prefetch_l2(const void *p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(p)));
}

// Ask L2 for the lines a warp of the atom-parallel passes streams from
// device memory, atoms [a0, a0 + m): the list columns up to the longest list
// of the last build and, in the force pass, the velocities, displacements
// and reference coordinates its integration reads.  A hint: nothing waits on
// it, and every address lies inside its array.  Systems whose streams stay in
// L2 from pass to pass (list, velocities, displacements, reference
// coordinates and records of all atoms, in FP32 4 bytes a neighbour and 92 an
// atom, below L.prefetch_from = 0.8 of L2) gain nothing from the hints and pay
// for them: us a step with and without, BCC 118,638 atoms (23 MB) 44.8 and 42.5,
// 453,962 (89 MB) 112.0 and 107.6, 574,992 (113 MB) 136.5 and 136.9, 686,000
// (134 MB) 155.4 and 163.5; FCC 256,000 (79 MB) 129 and 123.5, 470,596 (145 MB)
// 215.5 and 224.  The FP64 path always asks (314,928 atoms: 547 and 560).
template <class R, bool FORCE>
__device__ __forceinline__ void prefetch_warp_streams(const Bufs<R> &B, const Launch &L, int s, int a0, int m,
                                                      int ncol)
{
    if (a0 >= L.n || (long long)L.n * (4 * (long long)ncol + 92) < L.prefetch_from) return;
    const int lane = threadIdx.x & 31;
    for (int k = lane; k < ncol; k += 32) prefetch_l2(B.list + (size_t)k * L.ld + a0);
    if (FORCE) {
        // 128-byte lines: 16 doubles or 128 / sizeof(R) reference coordinates
        const int last = min(a0 + m, L.n) - 1;
        const int k = lane;
        if (k < 6) {
            const int c = k % 3;
            const int a = (k < 3) ? a0 : min(a0 + 16, last);
            prefetch_l2(B.v[s][c] + a);
            prefetch_l2(B.d[c] + a);
        } else if (k < 9) {
            prefetch_l2(B.uref[k - 6] + a0);
        } else if (k < 12 && sizeof(R) == 8) {
            prefetch_l2(B.uref[k - 9] + min(a0 + 16, last));
        }
    }
}

// ---- atom-parallel schedule ----

// Pairs in flight per lane: the type-dependent path needs more registers a pair.
template <class R, int KIND> struct PairsInFlight {
    static constexpr int density = KIND == KIND_ANY ? 2 : 3;
    // (type pairs: one, whose 64-byte row already holds more registers; 184,320
    // atoms 35.0 us, 42.5 with two)
    static constexpr int force = KIND == KIND_TYPES && sizeof(R) == 4 ? 1 : 2;
};

template <class R, int KIND, bool ENERGY, int TPA, bool TEX>
__global__ void __launch_bounds__(256) k_density(Bufs<R> B, Geom G, Launch L)
{
    using R4 = typename V4<R>::T;
    constexpr int U = PairsInFlight<R, KIND>::density;
    R h[3];
    load_h<R>(G, h);
    const DevState *st = B.st;
    const int sp = st->sp, s = st->set;
    R4 *sw = B.shadow[sp];
    const int width = blockDim.x / TPA;
    const int i0 = blockIdx.x * width;
    prefetch_warp_streams<R, false>(B, L, s, i0 + (threadIdx.x >> 5) * (32 / TPA), 32 / TPA, min(st->max_nnb, L.cap));
    const int i = i0 + threadIdx.x / TPA, l = threadIdx.x % TPA;
    const bool active = i < L.n;
    const int ti = (KIND != KIND_ONE && active) ? B.type[s][i] : 0;
    const R rc2 = g_rc2<R>(G);
    const TabGlobal<R> tab(B);
    R rho;
    if constexpr (TEX)
        rho = density_atom<R, KIND, TPA, U>(B, G, L, h, rc2, s, sp, i, l, active,
                                             TexFetch{(cudaTextureObject_t)B.tex_shadow[sp]}, tab);
    else
        rho = density_atom<R, KIND, TPA, U>(B, G, L, h, rc2, s, sp, i, l, active, GlobalFetch<R>{sw}, tab);
    rho = lane_sum<TPA>(rho);
    R e_embed = (R)0;
    if (active && l == 0) e_embed = embed<R>(B, sw, i, ti, rho);
    if (ENERGY) {
        const R v[1] = {e_embed};
        block_sums_t<1, R>(v, B.partials, L.pstride, 0);
    }
}

template <class R, int KIND, int MODE, bool ENERGY, int TPA>
__global__ void __launch_bounds__(256) k_force(Bufs<R> B, Geom G, Launch L)
{
    using R4 = typename V4<R>::T;
    constexpr int U = PairsInFlight<R, KIND>::force;
    R h[3];
    load_h<R>(G, h);
    const DevState *st = B.st;
    const int sp = st->sp, s = st->set;
    const R4 *sw = B.shadow[sp];
    const int width = blockDim.x / TPA;
    const int i0 = blockIdx.x * width;
    prefetch_warp_streams<R, true>(B, L, s, i0 + (threadIdx.x >> 5) * (32 / TPA), 32 / TPA, min(st->max_nnb, L.cap));
    const int i = i0 + threadIdx.x / TPA, l = threadIdx.x % TPA;
    const bool active = i < L.n;
    const int ti = (KIND != KIND_ONE && active) ? B.type[s][i] : 0;
    const R rc2 = g_rc2<R>(G);
    R f[3] = {0, 0, 0};
    R e7[7] = {0, 0, 0, 0, 0, 0, 0};
    force_atom<R, KIND, ENERGY, TPA, U>(B, G, L, h, rc2, s, sp, i, l, ti, active, GlobalFetch<R>{sw}, f, e7,
                                         TabGlobal<R>(B));
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] = lane_sum<TPA>(f[c]);
    double ke = 0.0;
    float d2 = 0.f;
    if (active) integrate<R, MODE, ENERGY, TPA>(B, L, s, sp, i, l, ti, f, ke, d2);
    force_block_end<R, ENERGY>(B, L, e7, ke, lane_sum<TPA>(d2), MODE == MODE_CLOSE_OPEN);
}

// ---- half lists (force symmetry): each pair once, the other end's term
// added through fixed-point accumulators ----
//
// A pair (i, j) sits in one list only: that of the atom that sees the other
// in the upper half space (the list build decides it exactly).  Its
// density term f(r) (one type: the same for both ends) and its force term
// s_ij (x_j - x_i)/r are formed once; i keeps its share in registers (a sum
// in a fixed order, stored in own[i]), j's share goes into acc_*[j] as a
// 64-bit integer in units of 2^-32 by an atomic add.  Integer sums do not
// depend on the order of the adds, so the totals, and every result, are
// bitwise reproducible.  A second pass per quantity adds own and acc (FP64),
// zeroes acc for the next use, and carries on as the full-list passes do:
// the embedding derivative F'(rho) into the record, or the integration.

constexpr float kFixScale = 4294967296.0f;       // 2^32 fixed-point units per unit
constexpr double kFixUnit = 1.0 / 4294967296.0;  // one unit
constexpr float kFixLimit = 16777216.0f;         // 2^24: largest pair term the accumulators take

__device__ __forceinline__ unsigned long long to_fixed(float x)
{
    return (unsigned long long)__float2ll_rn(x * kFixScale);
}

__device__ __forceinline__ double from_fixed(unsigned long long a)
{
    return (double)(long long)a * kFixUnit;
}

// rho_i's own terms and the scatter of j's; one lane per atom.
__global__ void __launch_bounds__(256) k_density_half(Bufs<float> B, Geom G, Launch L)
{
    constexpr int U = 3;
    float h[3];
    load_h<float>(G, h);
    const DevState *st = B.st;
    const int sp = st->sp, s = st->set;
    const float4 *sw = B.shadow[sp];
    const int i0 = blockIdx.x * blockDim.x;
    prefetch_warp_streams<float, false>(B, L, s, i0 + (threadIdx.x & ~31), 32, min(st->max_nnb, L.cap));
    const int i = i0 + threadIdx.x;
    if (i >= L.n) return;
    const SplineDesc<float> g = B.tables->fphi;
    const float rc2 = g_rc2<float>(G);
    const float4 ui = sw[i];
    const uint32_t *lp = B.list + i;
    const int nn = B.nnb[i];
    float rho = 0.f;
    bool range_ok = true;
    for (int k = 0; k < nn; k += U) {
        uint32_t e[U];
        float4 u[U];
#pragma unroll
        for (int q = 0; q < U; ++q) e[q] = (k + q < nn) ? lp[(size_t)(k + q) * L.ld] : 0u;
#pragma unroll
        for (int q = 0; q < U; ++q) u[q] = sw[(q == 0 || k + q < nn ? e[q] : e[0]) & kIndexMask];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const PairIn<float> pv = pair_vector<float>(ui, u[q], entry_shift<float>(e[q], h));
            if ((q == 0 || k + q < nn) && pv.r2 < rc2) {
                float rinv, r;
                inv_r(pv.r2, rinv, r);
                float t;
                const int kk = segment(g, r, t);
                const float4 c = B.coef_f[kk];
                const float v = fma(t, fma(t, fma(t, c.w, c.z), c.y), c.x);
                rho += v;
                range_ok = range_ok && fabsf(v) < kFixLimit;
                atomicAdd(B.acc_rho + (e[q] & kIndexMask), to_fixed(v));
            }
        }
    }
    if (!range_ok) atomicOr(&B.st->error, ERR_NONFINITE);
    B.own[i].x = rho;
}

// rho_i = own + accumulated, F'(rho_i) into the record, F(rho_i) for the
// energy; the accumulator is zeroed for the next pass.
template <bool ENERGY>
__global__ void __launch_bounds__(256) k_embed_half(Bufs<float> B, Launch L)
{
    const DevState *st = B.st;
    float4 *sw = B.shadow[st->sp];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float e_embed = 0.f;
    if (i < L.n) {
        const double rho = (double)B.own[i].x + from_fixed(B.acc_rho[i]);
        B.acc_rho[i] = 0ull;
        e_embed = embed<float>(B, sw, i, 0, (float)rho);
    }
    if (ENERGY) {
        const float v[1] = {e_embed};
        block_sums_t<1, float>(v, B.partials, L.pstride, 0);
    }
}

// F_i's own terms of Eq. 4 and the scatter of j's (-s_ij d / r); with ENERGY
// the pair energy phi(r) and the virial of each pair, counted once.
template <bool ENERGY>
__global__ void __launch_bounds__(256) k_force_half(Bufs<float> B, Geom G, Launch L)
{
    constexpr int U = 2;
    float h[3];
    load_h<float>(G, h);
    const DevState *st = B.st;
    const int sp = st->sp, s = st->set;
    const float4 *sw = B.shadow[sp];
    const int i0 = blockIdx.x * blockDim.x;
    prefetch_warp_streams<float, true>(B, L, s, i0 + (threadIdx.x & ~31), 32, min(st->max_nnb, L.cap));
    const int i = i0 + threadIdx.x;
    const SplineDesc<float> g = B.tables->fphi;
    const float rc2 = g_rc2<float>(G);
    float f0 = 0.f, f1 = 0.f, f2 = 0.f;
    float e7[7] = {0, 0, 0, 0, 0, 0, 0};
    if (i < L.n) {
        const float4 ui = sw[i];
        const float Fpi = ui.w;
        const uint32_t *lp = B.list + i;
        const int nn = B.nnb[i];
        bool range_ok = true;
        for (int k = 0; k < nn; k += U) {
            uint32_t e[U];
            float4 u[U];
#pragma unroll
            for (int q = 0; q < U; ++q) e[q] = (k + q < nn) ? lp[(size_t)(k + q) * L.ld] : 0u;
#pragma unroll
            for (int q = 0; q < U; ++q) u[q] = sw[(q == 0 || k + q < nn ? e[q] : e[0]) & kIndexMask];
#pragma unroll
            for (int q = 0; q < U; ++q) {
                const PairIn<float> pv = pair_vector<float>(ui, u[q], entry_shift<float>(e[q], h));
                if ((q == 0 || k + q < nn) && pv.r2 < rc2) {
                    float rinv, r;
                    inv_r(pv.r2, rinv, r);
                    float t;
                    const int kk = segment(g, r, t);
                    float4 cf, cp;
                    load_row2<float>(B.coef2 + 2 * kk, cf, cp);
                    const float fd = fma(t, fma(t, 3.f * cf.w, 2.f * cf.z), cf.y);
                    const float pd = fma(t, fma(t, 3.f * cp.w, 2.f * cp.z), cp.y);
                    const float sr = fma(u[q].w + Fpi, fd, pd) * rinv;
                    const float gx = sr * pv.dx, gy = sr * pv.dy, gz = sr * pv.dz;
                    f0 += gx;
                    f1 += gy;
                    f2 += gz;
                    range_ok = range_ok && fabsf(gx) < kFixLimit && fabsf(gy) < kFixLimit && fabsf(gz) < kFixLimit;
                    unsigned long long *aj = B.acc_f + 3 * (size_t)(e[q] & kIndexMask);
                    atomicAdd(aj + 0, to_fixed(-gx));
                    atomicAdd(aj + 1, to_fixed(-gy));
                    atomicAdd(aj + 2, to_fixed(-gz));
                    if (ENERGY) {
                        e7[0] += fma(t, fma(t, fma(t, cp.w, cp.z), cp.y), cp.x);
                        const float hs = -sr;
                        e7[1] = fma(hs * pv.dx, pv.dx, e7[1]);
                        e7[2] = fma(hs * pv.dy, pv.dy, e7[2]);
                        e7[3] = fma(hs * pv.dz, pv.dz, e7[3]);
                        e7[4] = fma(hs * pv.dx, pv.dy, e7[4]);
                        e7[5] = fma(hs * pv.dx, pv.dz, e7[5]);
                        e7[6] = fma(hs * pv.dy, pv.dz, e7[6]);
                    }
                }
            }
        }
        if (!range_ok) atomicOr(&B.st->error, ERR_NONFINITE);
        B.own[i] = make_float4(f0, f1, f2, 0.f);
    }
    if (ENERGY) {
        const float pe[1] = {e7[0]};
        block_sums_t<1, float>(pe, B.partials, L.pstride, 1);
        const float w6[6] = {e7[1], e7[2], e7[3], e7[4], e7[5], e7[6]};
        block_sums_t<6, float>(w6, B.partials, L.pstride, 3);
    }
}

// F_i = own + accumulated (zeroed for the next pass), then the integration
// of the full-list force pass (kicks, drift, next record, cached forces,
// kinetic energy and largest displacement as MODE asks).
template <int MODE, bool ENERGY>
__global__ void __launch_bounds__(256) k_integrate_half(Bufs<float> B, Launch L)
{
    const DevState *st = B.st;
    const int sp = st->sp, s = st->set;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double ke = 0.0;
    float d2 = 0.f;
    if (i < L.n) {
        const float4 o = B.own[i];
        unsigned long long *ai = B.acc_f + 3 * (size_t)i;
        const float f[3] = {(float)((double)o.x + from_fixed(ai[0])), (float)((double)o.y + from_fixed(ai[1])),
                            (float)((double)o.z + from_fixed(ai[2]))};
        ai[0] = 0ull;
        ai[1] = 0ull;
        ai[2] = 0ull;
        integrate<float, MODE, ENERGY, 1>(B, L, s, sp, i, 0, 0, f, ke, d2);
    }
    if (ENERGY) {
        const float ke_hi = (float)ke;
        const float v[1] = {ke_hi};
        const float lo[1] = {(float)(ke - (double)ke_hi)};
        block_sums_t<1, float>(v, B.partials, L.pstride, 2, lo);
    }
    if (MODE == MODE_CLOSE_OPEN) block_max_disp(d2, &B.st->maxdisp2);
}

template <int MODE, bool ENERGY>
void force_half(const Bufs<float> &B, const Geom &G, const Launch &L)
{
    dim3 g(L.nb_f), b(L.block_f);
    k_force_half<ENERGY><<<g, b, 0, L.stream>>>(B, G, L);
    k_integrate_half<MODE, ENERGY><<<g, b, 0, L.stream>>>(B, L);
}

// ---- dispatch ----

template <class R, int KIND, bool ENERGY, bool TEX>
void density_tpa_fetch(const Bufs<R> &B, const Geom &G, const Launch &L)
{
    dim3 g(L.nb_d), b(L.block_d);
    switch (L.tpa_d) {
    case 1: k_density<R, KIND, ENERGY, 1, TEX><<<g, b, compact_bytes<R>(L.block_d, 1), L.stream>>>(B, G, L); break;
    case 2: k_density<R, KIND, ENERGY, 2, TEX><<<g, b, compact_bytes<R>(L.block_d, 2), L.stream>>>(B, G, L); break;
    case 4: k_density<R, KIND, ENERGY, 4, TEX><<<g, b, compact_bytes<R>(L.block_d, 4), L.stream>>>(B, G, L); break;
    default: k_density<R, KIND, ENERGY, 8, TEX><<<g, b, compact_bytes<R>(L.block_d, 8), L.stream>>>(B, G, L); break;
    }
}

// Records through the texture path where both record buffers have a texture
// object (FP32), through the load path otherwise (FP64).
template <class R, int KIND, bool ENERGY>
void density_tpa(const Bufs<R> &B, const Geom &G, const Launch &L)
{
    if constexpr (std::is_same<R, float>::value) {
        if (B.tex_shadow[0] && B.tex_shadow[1]) {
            density_tpa_fetch<R, KIND, ENERGY, true>(B, G, L);
            return;
        }
    }
    density_tpa_fetch<R, KIND, ENERGY, false>(B, G, L);
}

template <class R, int KIND, int MODE, bool ENERGY>
void force_tpa(const Bufs<R> &B, const Geom &G, const Launch &L)
{
    dim3 g(L.nb_f), b(L.block_f);
    switch (L.tpa_f) {
    case 1: k_force<R, KIND, MODE, ENERGY, 1><<<g, b, compact_bytes<R>(L.block_f, 1), L.stream>>>(B, G, L); break;
    case 2: k_force<R, KIND, MODE, ENERGY, 2><<<g, b, compact_bytes<R>(L.block_f, 2), L.stream>>>(B, G, L); break;
    case 4: k_force<R, KIND, MODE, ENERGY, 4><<<g, b, compact_bytes<R>(L.block_f, 4), L.stream>>>(B, G, L); break;
    default: k_force<R, KIND, MODE, ENERGY, 8><<<g, b, compact_bytes<R>(L.block_f, 8), L.stream>>>(B, G, L); break;
    }
}

template <class R, int KIND>
void force_modes_plain(const Bufs<R> &B, const Geom &G, const Launch &L, int mode)
{
    if (mode == MODE_MEASURE) force_tpa<R, KIND, MODE_MEASURE, false>(B, G, L);
    else if (mode == MODE_CLOSE) force_tpa<R, KIND, MODE_CLOSE, false>(B, G, L);
    else force_tpa<R, KIND, MODE_CLOSE_OPEN, false>(B, G, L);
}

template <class R, int KIND>
void force_modes(const Bufs<R> &B, const Geom &G, const Launch &L, int mode, bool energy)
{
    if (!energy) force_modes_plain<R, KIND>(B, G, L, mode);
    else if (mode == MODE_MEASURE) force_tpa<R, KIND, MODE_MEASURE, true>(B, G, L);
    else if (mode == MODE_CLOSE) force_tpa<R, KIND, MODE_CLOSE, true>(B, G, L);
    else force_tpa<R, KIND, MODE_CLOSE_OPEN, true>(B, G, L);
}

}  // namespace

template <class R>
int launch_density(const Bufs<R> &B, const Geom &G, const Launch &L, bool energy)
{
    if constexpr (std::is_same<R, float>::value) {
        if (L.half) {
            dim3 g(L.nb_d), b(L.block_d);
            k_density_half<<<g, b, 0, L.stream>>>(B, G, L);
            if (energy) k_embed_half<true><<<g, b, 0, L.stream>>>(B, L);
            else k_embed_half<false><<<g, b, 0, L.stream>>>(B, L);
            return 2;
        }
    }
    // with energies several types take the general kernels (one step of a call)
    if (L.multi == KIND_TYPES && !energy) {
        density_tpa<R, KIND_TYPES, false>(B, G, L);
    } else if (L.multi) {
        if (energy) density_tpa<R, KIND_ANY, true>(B, G, L);
        else density_tpa<R, KIND_ANY, false>(B, G, L);
    } else {
        if (energy) density_tpa<R, KIND_ONE, true>(B, G, L);
        else density_tpa<R, KIND_ONE, false>(B, G, L);
    }
    return 1;
}

template <class R>
int launch_force(const Bufs<R> &B, const Geom &G, const Launch &L, int mode, bool energy)
{
    if constexpr (std::is_same<R, float>::value) {
        if (L.half) {
            if (mode == MODE_MEASURE) {
                if (energy) force_half<MODE_MEASURE, true>(B, G, L);
                else force_half<MODE_MEASURE, false>(B, G, L);
            } else if (mode == MODE_CLOSE) {
                if (energy) force_half<MODE_CLOSE, true>(B, G, L);
                else force_half<MODE_CLOSE, false>(B, G, L);
            } else {
                if (energy) force_half<MODE_CLOSE_OPEN, true>(B, G, L);
                else force_half<MODE_CLOSE_OPEN, false>(B, G, L);
            }
            return 2;
        }
    }
    if (L.multi == KIND_TYPES && !energy) force_modes_plain<R, KIND_TYPES>(B, G, L, mode);
    else if (L.multi) force_modes<R, KIND_ANY>(B, G, L, mode, energy);
    else force_modes<R, KIND_ONE>(B, G, L, mode, energy);
    return 1;
}


}  // namespace eammd
