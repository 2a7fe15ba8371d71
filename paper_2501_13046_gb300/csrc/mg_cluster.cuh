// mg_cluster.cuh -- the bottom of a V-cycle in one thread-block cluster.
//
// The levels of at most ~20^3 cells do little work per step, so a launch per colour pass (7-8 us at
// 16^3, of which the arithmetic is a few hundred nanoseconds) and a single CTA for the last two
// levels (29 us per cycle at 8^3 + 4^3) are bound by latency.  Here a cluster of 8 CTAs runs
// them all: pre-sweeps, restriction, the dense coarsest solve, prolongation and post-sweeps of
// every level from `the first level that fits` down.  Every CTA holds the whole correction of
// every level in its shared memory; a step's cells are split over the CTAs, and a new value is
// written to all 8 copies through distributed shared memory, so neighbours are always local reads
// and no halo exists.  One step costs its longest thread's stencil (4400 cycles at 16^3, 1900 at 8^3), its
// stores (~1500) and one or two cluster barriers: 42 us per V(1,1) cycle from 16^3 down in 4th order back to back
// (Robin 76; 56 and 96 cold, between other kernels), where the per-level kernels took 78.  FP64 from 8^3 down: 29 us
// against 175 us in one CTA.  The cluster barriers are hardware barriers of one launch, whose 8 CTAs run together by
// definition and all reach every one of them: no wait on a flag, so no iteration limit.
//
// A warp takes one row of the operator (psi, W_x, W_y or W_z) at 32 cells, so a thread's chain is
// one row's taps (13 or 45 in 4th order), not all four rows' 148.  Shared-memory layout of a field:
// the cells of even x, then those of odd x, so the 32 cells of one colour (x stride 2) lie side by
// side.  The boundary rule maps each coordinate by itself (wrap, clamp, mirror), so a
// tap's address is the sum of three per-axis offsets formed once per cell; the Robin ratio
// comes from a table over the level padded by 2.
//
// Operator, colour order and Jacobi-within-colour reads are those of the per-kernel path.
#pragma once
#include "mg_coarse.cuh"

namespace ctt {

constexpr int kClusterCtas = 8, kClusterThreads = 512;
static_assert(kClusterCtas == 8, "the restriction's 8 lanes of a coarse cell write one CTA's copy each");
constexpr int kClusterLevels = 3;               // levels above the coarsest handled at most
constexpr int kClusterCells = 8000;             // cells of the first level at most (20^3)
constexpr int kClusterIts = (kClusterCells / 2 / kClusterCtas + 127) / 128;   // cells per thread and colour

template <typename T>
struct ClusterLevel {
    Geo g;
    Coef<T> cf;
    const T *ab;   // psi-row coefficients (global, colour-split)
};

template <typename T>
struct ClusterArgs {
    ClusterLevel<T> lev[kClusterLevels];
    Geo gc;                 // the coarsest level
    int nl;                 // levels above it
    int zero;               // the first level's correction starts at zero, else at e_in
    int nu_pre, nu_post;
    const T *f, *e_in;      // the first level's right-hand side and correction (global, colour-split)
    T *e_out;
    const T *Gpsi, *GW;     // the coarsest level's inverses
    int mpsi, mw;
};

// Storage of a split level's field: x parity halves of planes, a plane padded to 16 mod 32 words so that the
// children of a coarse cell (two rows of two planes) lie in different banks.
__host__ __device__ inline int cluster_plane(const Geo &g)
{
    const int p = (g.n[0] >> 1) * g.n[1];
    return p + ((16 - p) & 31);
}
__host__ __device__ inline int cluster_field(const Geo &g, bool split)
{
    return split ? 2 * cluster_plane(g) * g.n[2] : g.n[0] * g.n[1] * g.n[2];
}

inline int cluster_share(int items) { return (items + kClusterCtas - 1) / kClusterCtas; }

// Shared-memory elements: per level the correction (4N), from the second on the right-hand side (4N), the
// CTA's own a, b (and the first level's f) of both colours, the Robin ratios; the coarsest f and e.  Then, in
// ints: per level its axis tables (n + 4 offsets per axis) and the own cells' coordinates.
inline size_t cluster_smem_bytes(const Geo *lev, int nl, const Geo &gc, int robin, size_t tb)
{
    auto axes = [](const Geo &g) { return (size_t)g.n[0] + g.n[1] + g.n[2] + 12; };
    size_t s = 8 * (size_t)gc.n[0] * gc.n[1] * gc.n[2], ints = axes(gc);
    for (int l = 0; l < nl; ++l) {
        const size_t N = (size_t)lev[l].n[0] * lev[l].n[1] * lev[l].n[2], share = (size_t)cluster_share((int)(N / 2));
        s += (l ? 8 : 4) * (size_t)cluster_field(lev[l], true) + (l ? 2 : 6) * 2 * share + fused_ratio_cells(lev[l], robin);
        ints += axes(lev[l]) + 2 * share;
    }
    return s * tb + ints * sizeof(int);
}

// The level whose bottom the cluster takes: the first one that is small enough, whose copies fit a CTA's shared
// memory, and of which a cluster with that much per CTA can be placed on this device (placeable(bytes); a
// partition may have too few free SMs per cluster).  -1: none, the per-level kernels run every level.
template <class Placeable>
inline int cluster_level(const Geo *lev, int nlev, int robin, size_t tb, Placeable placeable)
{
    const int Lc = nlev - 1;
    for (int l = Lc > kClusterLevels ? Lc - kClusterLevels : 0; l < Lc; ++l) {
        const size_t bytes = cluster_smem_bytes(lev + l, Lc - l, lev[Lc], robin, tb);
        if ((size_t)lev[l].n[0] * lev[l].n[1] * lev[l].n[2] <= (size_t)kClusterCells && bytes <= kMaxCoarseSmem &&
            placeable(bytes))
            return l;
    }
    return -1;
}

// ---------------------------------------------------------------- cluster primitives
// All threads of the cluster; orders memory both ways: what was written before it is seen after it, and
// what was read before it is not overwritten by a write after it (a relaxed arrival orders neither).
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// v to the same shared-memory place of CTA `rank`
template <typename T>
__device__ __forceinline__ void cluster_store(T *p, unsigned rank, T v)
{
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(sm_addr(p)), "r"(rank));
    if constexpr (sizeof(T) == 4) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
    else asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

template <typename T>
__device__ __forceinline__ void cluster_store_all(T *p, T v)
{
#pragma unroll
    for (unsigned r = 0; r < kClusterCtas; ++r) cluster_store(p, r, v);
}

// ---------------------------------------------------------------- taps
// Axis tables of a level: entry p + 2 of axis a is the offset that coordinate p (-2 .. n + 1) adds to a cell's
// place, after the boundary rule (see bc_cell); bit 30 marks a mirror image.
constexpr int kClusterMirror = 1 << 30;

template <int BC>
__device__ __forceinline__ int cluster_axis_entry(const Geo &g, int a, int p, bool split)
{
    const int n = g.n[a], nxh = split ? g.n[0] >> 1 : g.n[0], pl = split ? cluster_plane(g) : g.n[0] * g.n[1];
    int flag = 0;
    if constexpr (BC == BC_PERIODIC) {
        p += p < 0 ? n : (p >= n ? -n : 0);
    } else {
        if (BC == BC_SYM && p < 0 && ((g.reflect >> a) & 1)) {
            p = -1 - p;
            flag = kClusterMirror;
        } else {
            p = min(max(p, 0), n - 1);
        }
    }
    return flag | (a == 0 ? (split ? ((p & 1) ? pl * g.n[2] : 0) + (p >> 1) : p) : a == 1 ? p * nxh : p * pl);
}

// Per-axis offsets of the cells i - 2 .. i + 2, and, on boxes with faces, the place in the ratio table and
// which of them are mirrored.
template <int BC>
struct ClusterNb {
    int o[3][5];
    int r, rsy, rsz;   // ratio table: the cell itself, strides along y and z
    int mir;           // bit 5 a + d: the cell at offset d - 2 along axis a is a mirror image

    __device__ __forceinline__ void init(const Geo &g, const int *tab, int i, int j, int k)
    {
        const int *t[3] = {tab + i, tab + g.n[0] + 4 + j, tab + g.n[0] + g.n[1] + 8 + k};
        mir = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int d = 0; d < 5; ++d) {
                o[a][d] = t[a][d];
                if constexpr (BC == BC_SYM) {
                    if (o[a][d] & kClusterMirror) mir |= 1 << (5 * a + d);
                    o[a][d] &= kClusterMirror - 1;
                }
            }
        rsy = g.n[0] + 4;
        rsz = rsy * (g.n[1] + 4);
        r = i + 2 + (j + 2) * rsy + (k + 2) * rsz;
    }
    __device__ __forceinline__ int centre() const { return o[0][2] + o[1][2] + o[2][2]; }
};

// Field fi (0 = u, 1..3 = W_x..W_z) around a cell.
template <typename T, int BC>
struct ClusterAcc {
    const T *f, *rt;
    const ClusterNb<BC> *nb;
    int fi;
    __device__ __forceinline__ T operator()(int dx, int dy, int dz) const
    {
        T v = f[nb->o[0][dx + 2] + nb->o[1][dy + 2] + nb->o[2][dz + 2]];
        if constexpr (BC != BC_PERIODIC)
            v *= rt[nb->r + dx + dy * nb->rsy + dz * nb->rsz];
        if constexpr (BC == BC_SYM) {
            const int a = fi - 1, d = a == 0 ? dx : a == 1 ? dy : dz;
            if (fi > 0 && ((nb->mir >> (5 * a + d + 2)) & 1)) v = -v;
        }
        return v;
    }
};

// Row `row` of J e at a cell (0: psi, 1 + A: the row of W_A), as apply_J; e: the level's 4 fields, F apart.
template <typename T, int ORDER, int BC>
__device__ __forceinline__ T cluster_row(int row, const T *e, int F, const T *rt, const ClusterNb<BC> &nb, T ca, T cb,
                                         const Coef<T> &cf, T &ctr)
{
    auto acc = [&](int f) { return ClusterAcc<T, BC>{e + f * F, rt, &nb, f}; };
    auto lap = [&](const ClusterAcc<T, BC> &w, T &dxx, T &dyy, T &dzz) {
        ctr = w(0, 0, 0);
        dxx = d2<ORDER, 0, T>(w, ctr) * cf.ih2[0];
        dyy = d2<ORDER, 1, T>(w, ctr) * cf.ih2[1];
        dzz = d2<ORDER, 2, T>(w, ctr) * cf.ih2[2];
        return dxx + dyy + dzz;
    };
    T dxx, dyy, dzz;
    if (row == 0) {
        const T l = lap(acc(0), dxx, dyy, dzz);
        return ca * l + cb * ctr;
    }
    const T third = (T)(1.0 / 3.0);
    if (row == 1) {
        const T l = lap(acc(1), dxx, dyy, dzz);
        const T mx = dmix<ORDER, 0, 1, T>(acc(2)) * (cf.ih[0] * cf.ih[1]) + dmix<ORDER, 0, 2, T>(acc(3)) * (cf.ih[0] * cf.ih[2]);
        return l + (dxx + mx) * third;
    }
    if (row == 2) {
        const T l = lap(acc(2), dxx, dyy, dzz);
        const T mx = dmix<ORDER, 1, 0, T>(acc(1)) * (cf.ih[1] * cf.ih[0]) + dmix<ORDER, 1, 2, T>(acc(3)) * (cf.ih[1] * cf.ih[2]);
        return l + (dyy + mx) * third;
    }
    const T l = lap(acc(3), dxx, dyy, dzz);
    const T mx = dmix<ORDER, 2, 0, T>(acc(1)) * (cf.ih[2] * cf.ih[0]) + dmix<ORDER, 2, 1, T>(acc(2)) * (cf.ih[2] * cf.ih[1]);
    return l + (dzz + mx) * third;
}

// place of cell (i, j, k) in a field: even x, then odd x (split levels); x fastest (the coarsest)
__device__ __forceinline__ int cluster_place(const Geo &g, int i, int j, int k, bool split)
{
    if (!split) return i + g.n[0] * (j + g.n[1] * k);
    const int pl = cluster_plane(g);
    return ((i & 1) ? pl * g.n[2] : 0) + k * pl + j * (g.n[0] >> 1) + (i >> 1);
}

// ---------------------------------------------------------------- the kernel
template <typename T, int ORDER, int BC>
__global__ void __launch_bounds__(kClusterThreads) k_cluster_cycle(const __grid_constant__ ClusterArgs<T> A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = warp & 3, sub = (warp >> 2) * 32 + lane;
    const int rank = (int)cluster_rank();
    const int Nc = A.gc.n[0] * A.gc.n[1] * A.gc.n[2];
    constexpr int kStep = kClusterThreads / 4;   // cells per round: every warp quad takes 32 cells x 4 rows
    // shared-memory pointers
    T *e[kClusterLevels], *fl[kClusterLevels], *own[kClusterLevels], *rt[kClusterLevels];
    T *sp = reinterpret_cast<T *>(smem_raw);
    T *fc = sp, *ec = fc + 4 * Nc;
    sp = ec + 4 * Nc;
#pragma unroll
    for (int l = 0; l < kClusterLevels; ++l) {
        if (l >= A.nl) break;
        const Geo &g = A.lev[l].g;
        const int N = g.n[0] * g.n[1] * g.n[2], per = (N / 2 + kClusterCtas - 1) / kClusterCtas;
        const int F = cluster_field(g, true);
        e[l] = sp;
        sp += 4 * F;
        fl[l] = sp;
        if (l) sp += 4 * F;
        own[l] = sp;                    // [a, b (, f_0..3)][colour][per]
        sp += (l ? 2 : 6) * 2 * per;
        rt[l] = sp;
        if (BC != BC_PERIODIC) sp += (g.n[0] + 4) * (g.n[1] + 4) * (g.n[2] + 4);
    }
    int *tab[kClusterLevels + 1], *ijk[kClusterLevels];   // axis tables; own cells, [colour][per], 10 bits per axis
    int *ip = reinterpret_cast<int *>(sp);
#pragma unroll
    for (int l = 0; l <= kClusterLevels; ++l) {
        if (l > A.nl) break;
        const Geo &g = l == A.nl ? A.gc : A.lev[l].g;
        tab[l] = ip;
        ip += g.n[0] + g.n[1] + g.n[2] + 12;
        if (l < A.nl) {
            ijk[l] = ip;
            ip += 2 * ((g.n[0] * g.n[1] * g.n[2] / 2 + kClusterCtas - 1) / kClusterCtas);
        }
    }
    // cell m of a colour (pair order): its coordinates
    auto cell = [](const Geo &g, int colour, int m, int &i, int &j, int &k) {
        const int nxh = g.n[0] >> 1, r = m / nxh;
        j = r % g.n[1];
        k = r / g.n[1];
        i = 2 * (m - r * nxh) + ((colour + j + k) & 1);
    };
    auto unpack = [](int v, int &i, int &j, int &k) {
        i = v & 1023;
        j = (v >> 10) & 1023;
        k = v >> 20;
    };
    // start: tables, own coefficients, ratios, corrections (zero, or e_in on the first level)
    for (int l = 0; l <= A.nl; ++l) {
        const Geo &g = l == A.nl ? A.gc : A.lev[l].g;
        const int n0 = g.n[0] + 4, n01 = n0 + g.n[1] + 4, n = n01 + g.n[2] + 4;
        for (int t = tid; t < n; t += kClusterThreads) {
            const int a = t < n0 ? 0 : t < n01 ? 1 : 2, p = t - (a == 0 ? 0 : a == 1 ? n0 : n01) - 2;
            tab[l][t] = cluster_axis_entry<BC>(g, a, p, l < A.nl);
        }
    }
#pragma unroll
    for (int l = 0; l < kClusterLevels; ++l) {
        if (l >= A.nl) break;
        const Geo &g = A.lev[l].g;
        const int N = g.n[0] * g.n[1] * g.n[2], Nh = N / 2, per = (Nh + kClusterCtas - 1) / kClusterCtas;
        for (int t = tid; t < 2 * per; t += kClusterThreads) {
            const int c = t / per, m = rank * per + (t - c * per);
            if (m < Nh) {
                const int q = c * Nh + m;
                int i, j, k;
                cell(g, c, m, i, j, k);
                ijk[l][t] = i | (j << 10) | (k << 20);
                own[l][t] = A.lev[l].ab[q];
                own[l][2 * per + t] = A.lev[l].ab[N + q];
                if (l == 0)
                    for (int a = 0; a < 4; ++a) own[l][(2 + a) * 2 * per + t] = A.f[a * N + q];
            }
        }
        const bool from = l == 0 && !A.zero;
        if (from) {
            for (int t = tid; t < N; t += kClusterThreads) {
                const int c = t >= Nh, m = t - c * Nh;
                int i, j, k;
                cell(g, c, m, i, j, k);
                const int p = cluster_place(g, i, j, k, true);
                for (int a = 0; a < 4; ++a) e[l][a * cluster_field(g, true) + p] = A.e_in[a * N + t];
            }
        } else {
            for (int t = tid; t < 4 * cluster_field(g, true); t += kClusterThreads) e[l][t] = 0;
        }
        if constexpr (BC != BC_PERIODIC) {
            const int m0 = g.n[0] + 4, m1 = g.n[1] + 4, M = m0 * m1 * (g.n[2] + 4);
            for (int t = tid; t < M; t += kClusterThreads) {
                const int c[3] = {t % m0 - 2, (t / m0) % m1 - 2, t / (m0 * m1) - 2};
                int b[3], mirror;
                rt[l][t] = bc_cell<BC>(g, c, b, mirror) ? robin_ratio<T>(g, b[0], b[1], b[2], c[0], c[1], c[2]) : (T)1;
            }
        }
    }
    cluster_barrier();

    // nu sweeps of level l; zero: the level's correction is still zero
    auto sweeps = [&](int l, int nu, bool zero) {
        const Geo &g = A.lev[l].g;
        const Coef<T> &cf = A.lev[l].cf;
        const int N = g.n[0] * g.n[1] * g.n[2], Nh = N / 2, F = cluster_field(g, true), per = (Nh + kClusterCtas - 1) / kClusterCtas;
        const int m0 = rank * per, m1 = min(m0 + per, Nh);
#pragma unroll 1
        for (int s = 0; s < 2 * nu; ++s) {
            const int colour = s & 1;
            T nv[kClusterIts];
            int place[kClusterIts];
#pragma unroll
            for (int it = 0; it < kClusterIts; ++it) {
                const int lm = sub + it * kStep, m = m0 + lm;
                if (lm >= per || m >= m1) continue;
                int i, j, k;
                const int t = colour * per + lm;
                unpack(ijk[l][t], i, j, k);
                ClusterNb<BC> nb;
                nb.init(g, tab[l], i, j, k);
                const int p = nb.centre();
                place[it] = p;
                const T ca = own[l][t], cb = own[l][2 * per + t];
                const T fv = l == 0 ? own[l][(2 + row) * 2 * per + t] : fl[l][row * F + p];
                T Je = 0, ctr = 0;
                if (!(zero && s == 0)) {
                    Je = cluster_row<T, ORDER, BC>(row, e[l], F, rt[l], nb, ca, cb, cf, ctr);
                }
                T dl, kW[3];
                relax_factors<BC>(cf.fd, g, i, j, k, true, cf.dl, cf.idW, cf.iom, dl, kW);
                nv[it] = row == 0 ? ctr + (fv - Je) / ((ca * dl + cb) * cf.iom)
                                  : ctr + (fv - Je) * (row == 1 ? kW[0] : row == 2 ? kW[1] : kW[2]);
            }
            // every CTA has read the old values (a pass reads cells of its own colour: distance 2, mixed terms)
            if (!(zero && s == 0)) cluster_barrier();
#pragma unroll
            for (int it = 0; it < kClusterIts; ++it) {
                const int lm = sub + it * kStep, m = m0 + lm;
                if (lm >= per || m >= m1) continue;
                cluster_store_all(e[l] + row * F + place[it], nv[it]);
            }
            cluster_barrier();
        }
    };

#pragma unroll 1
    for (int l = 0; l < A.nl; ++l) {
        sweeps(l, A.nu_pre, l > 0 || A.zero);
        // residual and its 8-child means: 8 lanes per coarse cell, one child each, then one copy each
        const Geo &g = A.lev[l].g;
        const bool last = l + 1 == A.nl;
        const Geo &gn = last ? A.gc : A.lev[l + 1].g;
        const int N = g.n[0] * g.n[1] * g.n[2], Nn = gn.n[0] * gn.n[1] * gn.n[2], F = cluster_field(g, true);
        const int per = (Nn + kClusterCtas - 1) / kClusterCtas, q1 = min((rank + 1) * per, Nn);
        T *fn = last ? fc : fl[l + 1];
        const int d = lane & 7;
        struct Child {   // its inputs from global memory are fetched one round ahead
            int I, J, K, sq;
            T ca, cb, fv;
        } next;
        auto fetch = [&](int q, Child &c) {
            if (q >= q1) return;
            const int r2 = q / gn.n[0];
            c.I = q - r2 * gn.n[0];
            c.K = r2 / gn.n[1];
            c.J = r2 - c.K * gn.n[1];
            const int i = 2 * c.I + (d & 1), j = 2 * c.J + ((d >> 1) & 1), k = 2 * c.K + (d >> 2);
            const int lin = i + g.n[0] * (j + g.n[1] * k);
            c.sq = (((i + j + k) & 1) ? N / 2 : 0) + (lin >> 1);
            c.ca = row == 0 ? A.lev[l].ab[c.sq] : (T)0;
            c.cb = row == 0 ? A.lev[l].ab[N + c.sq] : (T)0;
            c.fv = l == 0 ? A.f[row * N + c.sq] : (T)0;
        };
        const int qa = rank * per + (warp >> 2) * 4 + (lane >> 3);
        fetch(qa, next);
        for (int q0 = rank * per + (warp >> 2) * 4; q0 < q1; q0 += kClusterThreads / 32) {
            const int q = q0 + (lane >> 3);
            const Child c = next;
            fetch(q + kClusterThreads / 32, next);
            T r = 0;
            if (q < q1) {
                ClusterNb<BC> nb;
                nb.init(g, tab[l], 2 * c.I + (d & 1), 2 * c.J + ((d >> 1) & 1), 2 * c.K + (d >> 2));
                const T fv = l == 0 ? c.fv : fl[l][row * F + nb.centre()], ca = c.ca, cb = c.cb;
                T ctr;
                r = fv - cluster_row<T, ORDER, BC>(row, e[l], F, rt[l], nb, ca, cb, A.lev[l].cf, ctr);
            }
            for (int o = 1; o < 8; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
            if (q < q1) cluster_store(fn + row * cluster_field(gn, !last) + cluster_place(gn, c.I, c.J, c.K, !last), (unsigned)d, r * (T)0.125);
        }
        cluster_barrier();
    }
    // coarsest level: e_c = G f_c, one warp per row, the rows split over the CTAs
    {
        const int per = (4 * Nc + kClusterCtas - 1) / kClusterCtas, r1 = min((rank + 1) * per, 4 * Nc);
        for (int r = rank * per + warp; r < r1; r += kClusterThreads / 32) {
            const bool psi = r < Nc;
            const T *gr = psi ? A.Gpsi + (size_t)r * A.mpsi : A.GW + (size_t)(r - Nc) * A.mw;
            const T *fr = psi ? fc : fc + Nc;
            const int len = psi ? Nc : 3 * Nc;
            T acc = 0;
            for (int j = lane; j < len; j += 32) acc = fma(gr[j], fr[j], acc);
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane < kClusterCtas) cluster_store(ec + r, (unsigned)lane, acc);
        }
        cluster_barrier();
    }
#pragma unroll 1
    for (int l = A.nl - 1; l >= 0; --l) {
        // trilinear prolongation (3/4, 1/4 per axis; coarse boundary values from the boundary rule)
        const Geo &g = A.lev[l].g;
        const bool last = l + 1 == A.nl;
        const Geo &gn = last ? A.gc : A.lev[l + 1].g;
        const T *en = last ? ec : e[l + 1];
        const int N = g.n[0] * g.n[1] * g.n[2], Nh = N / 2, F = cluster_field(g, true), Fn = cluster_field(gn, !last);
        const int per = (Nh + kClusterCtas - 1) / kClusterCtas, m0 = rank * per, m1 = min(m0 + per, Nh);
        for (int t = sub; t < 2 * per; t += kStep) {
            const int c = t / per, m = m0 + (t - c * per);
            if (m >= m1) continue;
            int i, j, k;
            unpack(ijk[l][t], i, j, k);
            const int ia[3][2] = {{i >> 1, (i >> 1) + ((i & 1) ? 1 : -1)}, {j >> 1, (j >> 1) + ((j & 1) ? 1 : -1)},
                                  {k >> 1, (k >> 1) + ((k & 1) ? 1 : -1)}};
            const int *tn = tab[l + 1];
            int o[3][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                o[0][h] = tn[ia[0][h] + 2];
                o[1][h] = tn[gn.n[0] + 4 + ia[1][h] + 2];
                o[2][h] = tn[gn.n[0] + gn.n[1] + 8 + ia[2][h] + 2];
            }
            T s = 0;
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                const int q[3] = {o[0][d & 1], o[1][(d >> 1) & 1], o[2][d >> 2]};
                T w = (T)(((d & 1) ? 0.25 : 0.75) * ((d & 2) ? 0.25 : 0.75) * ((d & 4) ? 0.25 : 0.75));
                if constexpr (BC != BC_PERIODIC) {
                    const int cc[3] = {ia[0][d & 1], ia[1][(d >> 1) & 1], ia[2][d >> 2]};
                    int b[3], mirror;
                    if (bc_cell<BC>(gn, cc, b, mirror)) w *= robin_ratio<T>(gn, b[0], b[1], b[2], cc[0], cc[1], cc[2]);
                    w = bc_signed<BC>(w, mirror, row);
                }
                s = fma(w, en[row * Fn + ((q[0] + q[1] + q[2]) & (kClusterMirror - 1))], s);
            }
            T *p = e[l] + row * F + cluster_place(g, i, j, k, true);
            cluster_store_all(p, *p + s);   // (a CTA's own cells: no other thread reads or writes them in this step)
        }
        cluster_barrier();
        sweeps(l, A.nu_post, false);
    }
    {
        const Geo &g = A.lev[0].g;
        const int N = g.n[0] * g.n[1] * g.n[2], Nh = N / 2;
        const int per = (Nh + kClusterCtas - 1) / kClusterCtas, m0 = rank * per, m1 = min(m0 + per, Nh);
        for (int t = sub; t < 2 * per; t += kStep) {
            const int c = t / per, m = m0 + (t - c * per);
            if (m >= m1) continue;
            int i, j, k;
            unpack(ijk[0][t], i, j, k);
            A.e_out[row * N + c * Nh + m] = e[0][row * cluster_field(g, true) + cluster_place(g, i, j, k, true)];
        }
    }
    // (the last barrier came after every remote store: no CTA leaves while another still writes to it)
}

}  // namespace ctt
