// mg_outer.cuh -- FP64 outer residual of the CTT constraints in one fused, tiled pass.
//
// On GB300 an FP64 instruction issues at 2 lanes per clock per SM (conversions to and from FP64
// too), integer and FP32 instructions at 64 to 128, so a residual written in FP64 arithmetic is
// bound by its FP64 instruction count: the two-kernel form this replaces spent ~160 of them per
// cell, 130 on the linear stencils (128^3: 95 us for q, div W, then 589 us; 256^3 Robin 0.6 + 4.8 ms).
// Here the stencils run on 64-bit integers.  Each CTA brings the planes of (u, W) of its tile into
// shared memory as fixed-point numbers in units of 2^(E - 56), E the exponent of the largest value
// the CTA has met so far (one E for u, one for the three W_i: every momentum row and At_ij takes
// all components).  The stencil weights are small integers (1/12 and 1/h^2 are applied at the
// end), so sums are exact: |x| < 2^57 units and a 4th-order second difference has weights of
// total size 64.  A double within 4 binary orders of E is represented exactly, a smaller one to
// 2^(E - 57), against the 2^(E - 48) an FP64 sum of the same taps rounds by (16 f + 16 f is
// formed first).  Only the results are converted: Lap u, the three momentum rows, AtAt.  What is
// left in FP64 is ~40 instructions per cell (powers of psi, the source terms, the block sums):
// 128^3 periodic 240 us (integer part alone 165 us, the FP64 part's floor ~150 us).
//
// March: 16 x 8 cells per plane, one thread per cell, planes along z through a ring of ORDER + 1
// slots (4 CTAs per SM: their integer and FP64 phases overlap).  The mixed term (1/3) d_i d_j W_j uses
// D_i D_j = D_i o D_j:
//   row x: D_x B + D_z C,  row y: D_y A + D_z D,  row z: D_z (A + B)
// with A = D_x W_x, B = D_y W_y, C = D_x W_z, D = D_y W_z formed once per plane; A and B are
// shared with the neighbouring cells through shared memory, beside the z history of A + B, C and D.
// A cell's FP64 tail runs one plane later, among the integer stencils of the next cell.  Boundary values
// (periodic wrap, Robin, mirror, extrapolation) are filled in when a plane is loaded, in FP64 by the
// rule of fetch_bc, so every cell takes this path.
//
// Values that are NaN or infinite have no fixed-point form: a CTA that meets one finishes its
// remaining planes with the direct FP64 stencils (outer_cell), which propagate it cell by cell.
// Fields below 2^-383 (5e-116) everywhere in a tile are held in units of 2^-439.
#pragma once
#include <algorithm>

#include "mg_kernels.cuh"

namespace ctt {

constexpr int kOutX = 16, kOutY = 8, kOutThreads = kOutX * kOutY;
constexpr int kOutMaxZ = 32;          // planes per CTA at most
constexpr int kOutMinExp = 640;       // smallest E (biased): units and their squares stay normal numbers
constexpr int kOutBadExp = 0x7ff;     // biased exponent of NaN and infinity

template <int ORDER> __host__ __device__ constexpr int outer_w() { return kOutX + ORDER; }        // tile + halo
template <int ORDER> __host__ __device__ constexpr int outer_rows() { return kOutY + ORDER; }
template <int ORDER> __host__ __device__ constexpr int outer_plane() { return 4 * outer_w<ORDER>() * outer_rows<ORDER>(); }
template <int ORDER> __host__ __device__ constexpr size_t outer_smem_bytes()
{   // the ring of planes; A (tile columns, all rows) and B (all columns, tile rows) of the centre plane; the
    // z history of A + B, C and D, ORDER planes of the tile's cells
    return ((size_t)(ORDER + 1) * outer_plane<ORDER>() + (size_t)kOutX * outer_rows<ORDER>() +
            (size_t)kOutY * outer_w<ORDER>() + (size_t)3 * ORDER * kOutThreads) * sizeof(long long);
}

// The state and the sources, plain arrays (rho2 may be null: zero).
struct OuterIn {
    const double *u, *W, *rho0, *rho2, *S;
};

// Integer weights: with unequal spacings each axis' difference is scaled by its share of the
// smallest spacing's weight (ratios <= 1 in 64-bit fixed point, the high half of a 64 x 64
// product); with equal spacings (iso) the shares are 1 and shifts suffice.
struct OuterInt {
    int iso;
    long long wl[3];      // Lap u: (hmin/h_a)^2
    long long w3[3][3];   // row A: (3 + delta_Aa) (hmin/h_a)^2
    long long gq[3];      // hmin/h_a, first derivatives inside the mixed term
    long long gm[3];      // ... outside it, with its 1/6 (order 4) or 1/4 (order 2)
    long long ga[3];      // ... of At_ij
    double cu, cm, ca;    // 1/(c hmin^2), a third of it (c = 12 or 1); 1/(c1 hmin) (c1 = 12 or 2)
};

inline OuterInt make_outer_int(const Geo &g, int order)
{
    OuterInt o;
    const double hmin = fmin(g.h[0], fmin(g.h[1], g.h[2])), hmax = fmax(g.h[0], fmax(g.h[1], g.h[2]));
    o.iso = hmax <= hmin * (1.0 + 4.5e-16);   // the same spacing up to the rounding of (hi - lo) / n
    auto fix = [](long double v, int bits) {  // v 2^bits, at most 2^63 - 1
        const long double s = ldexpl(v, bits);
        return s >= 9223372036854775807.0L ? 9223372036854775807LL : (long long)(s + 0.5L);
    };
    for (int a = 0; a < 3; ++a) {
        const long double r = (long double)hmin / (long double)g.h[a];
        o.wl[a] = fix(r * r, 62);
        for (int A = 0; A < 3; ++A) o.w3[A][a] = fix((A == a ? 4.0L : 3.0L) * r * r, 60);
        o.gq[a] = fix(r, 59);
        o.gm[a] = order == 4 ? fix(r / 6.0L, 64) : fix(r, 62);
        o.ga[a] = fix(r, 63);
    }
    o.cu = 1.0 / ((order == 4 ? 12.0 : 1.0) * hmin * hmin);
    o.cm = o.cu / 3.0;
    o.ca = 1.0 / ((order == 4 ? 12.0 : 2.0) * hmin);
    return o;
}

// Launch shape: planes per CTA.  A CTA loads ORDER planes more than it finishes and starts with a
// load of its own (~3 planes' time in all); up to four CTAs share an SM, and a plane of k of them
// takes about max(1, 0.67 k) times a plane of one (measured, 32^3 to 256^3: within 5% of the best zc).
struct OuterGrid {
    int ntx, nty, zc;
};

inline OuterGrid outer_grid(const Geo &g)
{
    constexpr int sms = 152;   // a constant: the workspace (one partial row per CTA) is sized without a device
    OuterGrid t;
    t.ntx = (g.n[0] + kOutX - 1) / kOutX;
    t.nty = (g.n[1] + kOutY - 1) / kOutY;
    t.zc = kOutMaxZ;
    double best = 0.0;
    for (int zc = kOutMaxZ; zc >= 2; --zc) {
        const long long ctas = (long long)t.ntx * t.nty * ((g.n[2] + zc - 1) / zc);
        const double cost = std::max(1.0, 0.67 * (double)((ctas + sms - 1) / sms)) * (zc + 3);
        if (best == 0.0 || cost < best) {
            best = cost;
            t.zc = zc;
        }
    }
    return t;
}

inline int outer_ctas(const Geo &g, const OuterGrid &t) { return t.ntx * t.nty * ((g.n[2] + t.zc - 1) / t.zc); }

// ---------------------------------------------------------------- integer stencils
// taps of one axis around a cell: p1, m1 at distance 1, p2, m2 at 2 (order 4)
template <int ORDER> struct IAxis { long long m1, p1, m2, p2; };

template <int ORDER>
__device__ __forceinline__ IAxis<ORDER> itaps(const long long *c, int s)
{
    if constexpr (ORDER == 4) return {c[-s], c[s], c[-2 * s], c[2 * s]};
    else return {c[-s], c[s], 0, 0};
}

// 12 h D f (order 4) or 2 h D f
template <int ORDER>
__device__ __forceinline__ long long id1(const IAxis<ORDER> &t)
{
    if constexpr (ORDER == 4) return ((t.p1 - t.m1) << 3) - (t.p2 - t.m2);
    else return t.p1 - t.m1;
}

// 12 h^2 D2 f (order 4) or h^2 D2 f; k0 = 30 f or 2 f
template <int ORDER>
__device__ __forceinline__ long long id2(const IAxis<ORDER> &t, long long k0)
{
    if constexpr (ORDER == 4) return ((t.p1 + t.m1) << 4) - (t.p2 + t.m2) - k0;
    else return t.p1 + t.m1 - k0;
}

template <int ORDER>
__device__ __forceinline__ long long ik0(long long f)
{
    if constexpr (ORDER == 4) return (f << 5) - (f << 1);
    else return f << 1;
}

// x in units of 2^(E - 56): an FP64 bit pattern of biased exponent <= E, rounded to nearest.  (The
// implicit bit that zero and denormal numbers do not have is shifted out: E >= kOutMinExp.)
__device__ __forceinline__ long long to_fixed(double x, int E)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mh = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;   // mantissa, leading one at bit 62
    const unsigned long long t = ((unsigned long long)mh << 32) | (lo << 10);
    const int d = min(E - (int)((hi >> 20) & 0x7ffu) + 5, 63);
    const long long v = (long long)(((t >> d) + 1) >> 1);
    return (int)hi < 0 ? -v : v;
}

__device__ __forceinline__ double pow2_biased(int e) { return __hiloint2double(e << 20, 0); }   // 2^(e - 1023)

// ---------------------------------------------------------------- out-of-line parts
// Boundary value of field fi (0 = u, 1..3 = W_i) at a cell outside the box.
template <int BC>
__device__ __noinline__ double outer_ghost(const double *f, int fi, const Geo &g, int i, int j, int k)
{
    return fetch_bc<double, BC>(f, fi, g, i, j, k);
}

// The direct FP64 form at a cell: out = (Lap u, AtAt, momentum rows).
template <int ORDER, int BC>
__device__ __noinline__ void outer_direct(const Geo &g, const Coef<double> &cf, const double *u, const double *W, int i,
                                          int j, int k, double *out)
{
    const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
    const size_t p = (size_t)i + (size_t)g.n[0] * ((size_t)j + (size_t)g.n[1] * k);
    AccB<double, BC> a0{u, 0, &g, i, j, k}, a1{W, 1, &g, i, j, k}, a2{W + N, 2, &g, i, j, k},
        a3{W + 2 * N, 3, &g, i, j, k};
    double lu, aa, mom[3];
    outer_cell<ORDER>(a0, a1, a2, a3, cf, lu, aa, mom, g.by ? g.by + p : nullptr, N);
    out[0] = lu;
    out[1] = aa;
    out[2] = mom[0];
    out[3] = mom[1];
    out[4] = mom[2];
}

// What the tail of a cell reads besides the stencils' results.
struct OuterSrc {
    double bg, u, rho0, rho2, S[3];   // psi = bg + u (added where it is used: nothing waits for the loads before)
};

__device__ __forceinline__ OuterSrc outer_src(const Geo &g, const OuterIn &in, size_t N, size_t p, int i, int j, int k)
{
    OuterSrc s;
    s.bg = psi_bg(g, i, j, k, p);
    s.u = in.u[p];
    s.rho0 = in.rho0[p];
    s.rho2 = in.rho2 ? in.rho2[p] : 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) s.S[a] = in.S[a * N + p];
    return s;
}

// The FP64 tail of a cell: nonlin = (1/8) psi^-7 AtAt + 2 pi (rho0 psi^5 + rho2 psi), s = 8 pi psi^6 S_i, p5 = psi^5.
__device__ __forceinline__ double outer_nonlin(const OuterSrc &c, double aa, double s[3], double &p5)
{
    const double psi = c.bg + c.u, p2 = psi * psi, p4 = p2 * p2;
    p5 = p4 * psi;
    const double p6 = p5 * psi, s8 = (8.0 * kPi) * p6;
#pragma unroll
    for (int a = 0; a < 3; ++a) s[a] = s8 * c.S[a];
    return fma(2.0 * kPi, fma(c.rho0, p5, c.rho2 * psi), (0.125 * aa) * recip_f64(p6 * psi));
}

// ---------------------------------------------------------------- the fused residual
//   R0 = Lap u + (1/8) psi^-7 AtAt + 2 pi (rho0 psi^5 + rho2 psi)     (F_psi before the K^2 term)
//   R1..3 = Lap W_i + (1/3) d_i d_j W_j - 8 pi psi^6 S_i                 (F_W before adding m_i)
//   R4 = AtAt (null: not stored; pass 2 forms the linearisation coefficient from it)
// and, on periodic boxes, one row of 5 partial sums per CTA; the last CTA finishes the outer
// scalars when fin.s is set.
template <int ORDER, int BC>
__global__ void __launch_bounds__(kOutThreads, 4)
    k_outer_residual(Geo g, Coef<double> cf, OuterInt oi, OuterIn in, double *__restrict__ R, double *__restrict__ R4,
                     double *__restrict__ partial, OuterGrid tg, OuterFin fin)
{
    constexpr int H = ORDER / 2, W = outer_w<ORDER>(), RW = outer_rows<ORDER>(), FE = W * RW, PE = outer_plane<ORDER>(),
                  NS = ORDER + 1;
    constexpr int NE = (FE + kOutThreads - 1) / kOutThreads;   // loaded elements per thread, field and plane
    constexpr int SHU = ORDER == 4 ? 2 : 0, SH3 = ORDER == 4 ? 4 : 0, QS = ORDER == 4 ? 5 : 0;   // pre-shifts of sums
    static_assert(2 * H * kOutX + 2 * H * kOutY <= kOutThreads, "one halo value of A or B per thread");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    long long *ring = reinterpret_cast<long long *>(smem_raw);
    long long *sA = ring + NS * PE, *sB = sA + kOutX * RW;      // A[row][kOutX], B[row of the tile][W]
    long long *hist = sB + kOutY * W + threadIdx.x;             // [A + B, C, D][plane % ORDER][thread]
    __shared__ int sE[2][2];                                    // [plane parity][u, W]: largest exponent of a plane

    const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], tid = threadIdx.x;
    const size_t plane = (size_t)nx * ny;
    int b = blockIdx.x;
    const int x0 = (b % tg.ntx) * kOutX;
    b /= tg.ntx;
    const int y0 = (b % tg.nty) * kOutY;
    const int z0 = (b / tg.nty) * tg.zc, z1 = min(z0 + tg.zc, nz), NP = z1 - z0 + 2 * H;
    const int lx = tid & (kOutX - 1), ly = tid / kOutX, i = x0 + lx, j = y0 + ly;
    const bool act = i < nx && j < ny;

    // loaded elements: in-plane offset of the (wrapped) cell, -1 beyond the halo, -2 a ghost of a box with faces
    int off[NE];
#pragma unroll
    for (int t = 0; t < NE; ++t) {
        const int e = tid + t * kOutThreads;
        int x = x0 - H + e % W, y = y0 - H + e / W;
        off[t] = -1;
        if (e < FE && x < nx + H && y < ny + H) {
            if constexpr (BC == BC_PERIODIC) {
                x += x < 0 ? nx : (x >= nx ? -nx : 0);
                y += y < 0 ? ny : (y >= ny ? -ny : 0);
                off[t] = x + nx * y;
            } else {
                off[t] = (x >= 0 && x < nx && y >= 0 && y < ny) ? x + nx * y : -2;
            }
        }
    }
    double raw[4][NE];
    auto load = [&](int p) {
        int z = z0 - H + p;
        bool zg = false;
        if constexpr (BC == BC_PERIODIC) z += z < 0 ? nz : (z >= nz ? -nz : 0);
        else zg = z < 0 || z >= nz;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const double *field = f == 0 ? in.u : in.W + (size_t)(f - 1) * N;
#pragma unroll
            for (int t = 0; t < NE; ++t) {
                raw[f][t] = 0.0;
                if (off[t] == -1) continue;
                if (BC != BC_PERIODIC && (zg || off[t] < 0)) {
                    const int e = tid + t * kOutThreads;
                    raw[f][t] = outer_ghost<BC>(field, f, g, x0 - H + e % W, y0 - H + e / W, z);
                } else {
                    raw[f][t] = (field + plane * z)[off[t]];
                }
            }
        }
    };
    auto reduce_exp = [&](int p) {   // into sE[p & 1]
        unsigned eu = 0, ew = 0;     // (the sign bit dropped, the largest high word has the largest exponent)
#pragma unroll
        for (int t = 0; t < NE; ++t) {
            eu = max(eu, (unsigned)__double2hiint(raw[0][t]) << 1);
#pragma unroll
            for (int f = 1; f < 4; ++f) ew = max(ew, (unsigned)__double2hiint(raw[f][t]) << 1);
        }
        eu = __reduce_max_sync(0xffffffffu, eu >> 21);
        ew = __reduce_max_sync(0xffffffffu, ew >> 21);
        if ((tid & 31) == 0) {
            atomicMax(&sE[p & 1][0], (int)eu);
            atomicMax(&sE[p & 1][1], (int)ew);
        }
    };
    int Eu = kOutMinExp, Ew = kOutMinExp;
    double wu, wm, wa, waa;   // units of Lap u, of the momentum rows, of At_ij, of the squares' high halves
    auto set_units = [&]() {
        wu = oi.cu * pow2_biased(Eu - 56 + SHU);
        wm = oi.cm * pow2_biased(Ew - 56 + SH3);
        wa = oi.ca * pow2_biased(Ew - 56);
        waa = wa * wa * pow2_biased(1023 + 64);
    };
    set_units();
    double acc[5] = {0, 0, 0, 0, 0};
    // the stencils' results at the centre cell of the last plane, finished one plane later: their FP64
    // tail then runs interleaved with the integer stencils of the next cell
    double cl = 0.0, cm[3] = {0.0, 0.0, 0.0}, ca = 0.0;
    auto finish = [&](const OuterSrc &c, size_t P, bool on) {
        double s[3], p5;
        const double nonlin = outer_nonlin(c, ca, s, p5), r0 = fma(cl, wu, nonlin);
        double r[3];
#pragma unroll
        for (int A = 0; A < 3; ++A) r[A] = fma(cm[A], wm, -s[A]);
        if (fin.periodic) {   // (other boxes use no sums)
            acc[0] += on ? nonlin : 0.0;
            acc[1] += on ? p5 : 0.0;
#pragma unroll
            for (int A = 0; A < 3; ++A) acc[2 + A] += on ? s[A] : 0.0;
        }
        if (on) {
            R[P] = r0;
#pragma unroll
            for (int A = 0; A < 3; ++A) R[(1 + A) * N + P] = r[A];
            if (R4) R4[P] = ca;
        }
    };

    if (tid < 4) sE[tid >> 1][tid & 1] = 0;
    load(0);
    __syncthreads();
    reduce_exp(0);
    __syncthreads();
    int bad = -1;
    int slot = 0;   // p % NS
    const int cell = (ly + H) * W + lx + H;
    const size_t P0 = (size_t)i + (size_t)nx * j + plane * z0;
    for (int p = 0; p < NP; ++p) {
        // phase 0: plane p into the ring in the current units (grown when it holds larger values),
        // A and B of the centre plane p - H for the tile's neighbours
        const int eu = sE[p & 1][0], ew = sE[p & 1][1];
        if (max(eu, ew) == kOutBadExp) { bad = p; break; }
        if (eu > Eu || ew > Ew) {   // rare: rescale what the ring, the history and the registers hold
            const int du = min(62, max(0, eu - Eu)), dw = min(62, max(0, ew - Ew));
            if (p > 0) {
                for (int e = tid; e < NS * PE; e += kOutThreads) {
                    const int d = (e % PE) < FE ? du : dw;
                    ring[e] = (ring[e] + ((1LL << d) >> 1)) >> d;
                }
#pragma unroll
                for (int k = 0; k < 3 * ORDER; ++k) hist[k * kOutThreads] >>= dw;
                cl *= pow2_biased(1023 - du);
#pragma unroll
                for (int A = 0; A < 3; ++A) cm[A] *= pow2_biased(1023 - dw);
                __syncthreads();
            }
            Eu = max(Eu, eu);
            Ew = max(Ew, ew);
            set_units();
        }
        const bool full = p >= 2 * H;
        const int zprev = max(0, p - 1 - 2 * H);   // the cell whose tail runs now (plane z0 + zprev)
        const size_t Pp = P0 + plane * zprev;
        OuterSrc src{1.0, 0.0, 0.0, 0.0, {0.0, 0.0, 0.0}};
        if (full && act) src = outer_src(g, in, N, Pp, i, j, z0 + zprev);
        {
            long long *dst = ring + slot * PE + tid;
#pragma unroll
            for (int f = 0; f < 4; ++f)
#pragma unroll
                for (int t = 0; t < NE; ++t)
                    if (tid + t * kOutThreads < FE) dst[f * FE + t * kOutThreads] = to_fixed(raw[f][t], f == 0 ? Eu : Ew);
        }
        if (p + 1 < NP) load(p + 1);
        const int cs = slot >= H ? slot - H : slot - H + NS;   // slot of the centre plane
        const long long *q = ring + cs * PE + cell;
        long long gxx = 0, gyy = 0;   // D_x W_x, D_y W_y at the cell
        auto q0 = [&](long long a, int ax) { return oi.iso ? a >> QS : __mul64hi(a << (5 - QS), oi.gq[ax]); };
        if (full) {
            gxx = id1<ORDER>(itaps<ORDER>(q + FE, 1));
            gyy = id1<ORDER>(itaps<ORDER>(q + 2 * FE, W));
            sA[(ly + H) * kOutX + lx] = q0(gxx, 0);
            sB[ly * W + lx + H] = q0(gyy, 1);
            const long long *c1 = ring + cs * PE + FE, *c2 = c1 + FE;   // W_x, W_y
            if (tid < 2 * H * kOutX) {   // A in the rows above and below the tile
                const int r = tid / kOutX, row = r < H ? r : r + kOutY;
                sA[row * kOutX + lx] = q0(id1<ORDER>(itaps<ORDER>(c1 + row * W + H + lx, 1)), 0);
            } else if (tid < 2 * H * (kOutX + kOutY)) {   // B in the columns left and right of it
                const int e = tid - 2 * H * kOutX, c = e % (2 * H), col = c < H ? c : c + kOutX, row = e / (2 * H);
                sB[row * W + col] = q0(id1<ORDER>(itaps<ORDER>(c2 + (H + row) * W + col, W)), 1);
            }
        }
        __syncthreads();
        // phase 1: the new plane's first derivatives; the previous cell's FP64 tail and the centre
        // plane's cell, in one block
        if (tid < 2) sE[p & 1][tid] = 0;
        long long ns, nc, nd;   // A + B, C, D of the new plane (p = centre + H)
        {
            const long long *n = ring + slot * PE + cell;
            const long long a = id1<ORDER>(itaps<ORDER>(n + FE, 1)), bb = id1<ORDER>(itaps<ORDER>(n + 2 * FE, W));
            const long long c = id1<ORDER>(itaps<ORDER>(n + 3 * FE, 1)), d = id1<ORDER>(itaps<ORDER>(n + 3 * FE, W));
            ns = oi.iso ? (a + bb) >> QS : q0(a, 0) + q0(bb, 1);
            nc = q0(c, 0);
            nd = q0(d, 1);
        }
        if (full && act) {
            finish(src, Pp, p > 2 * H);
            // z taps: planes of the ring, as offsets from the centre plane
            int zo[2 * H];
#pragma unroll
            for (int s = 0; s < 2 * H; ++s) {
                const int dz = s < H ? s - H : s - H + 1;
                int sl = cs + dz;
                sl += sl < 0 ? NS : (sl >= NS ? -NS : 0);
                zo[s] = (sl - cs) * PE;
            }
            auto ztaps = [&](const long long *c) -> IAxis<ORDER> {
                if constexpr (ORDER == 4) return {c[zo[1]], c[zo[2]], c[zo[0]], c[zo[3]]};
                else return {c[zo[0]], c[zo[1]], 0, 0};
            };
            // Lap u
            long long lu;
            {
                const long long k0 = ik0<ORDER>(q[0]);
                const long long dx = id2<ORDER>(itaps<ORDER>(q, 1), k0), dy = id2<ORDER>(itaps<ORDER>(q, W), k0),
                                dz = id2<ORDER>(ztaps(q), k0);
                // (the small constants centre the rounding of the shifts)
                if (oi.iso) lu = (dx >> SHU) + (dy >> SHU) + (dz >> SHU) + (SHU ? 1 : 0);
                else
                    lu = __mul64hi(dx << (2 - SHU), oi.wl[0]) + __mul64hi(dy << (2 - SHU), oi.wl[1]) +
                         __mul64hi(dz << (2 - SHU), oi.wl[2]) + 1;
            }
            cl = (double)lu;
            // momentum rows, Lap W_A + (1/3) D_AA W_A part, and the first derivatives of W_A
            long long m[3], g9[3][3];   // g9[a][A] = D_a W_A
#pragma unroll
            for (int A = 0; A < 3; ++A) {
                const long long *w = q + (1 + A) * FE;
                const long long k0 = ik0<ORDER>(w[0]);
                const IAxis<ORDER> tx = itaps<ORDER>(w, 1), ty = itaps<ORDER>(w, W), tz = ztaps(w);
                const long long d0 = id2<ORDER>(tx, k0), d1 = id2<ORDER>(ty, k0), d2 = id2<ORDER>(tz, k0);
                g9[0][A] = A == 0 ? gxx : id1<ORDER>(tx);
                g9[1][A] = A == 1 ? gyy : id1<ORDER>(ty);
                g9[2][A] = id1<ORDER>(tz);
                if (oi.iso) {
                    const long long e0 = d0 >> SH3, e1 = d1 >> SH3, e2 = d2 >> SH3, s = e0 + e1 + e2;
                    m[A] = (s << 1) + s + (A == 0 ? e0 : A == 1 ? e1 : e2) + (SH3 ? 5 : 0);
                } else {
                    m[A] = __mul64hi(d0 << (4 - SH3), oi.w3[A][0]) + __mul64hi(d1 << (4 - SH3), oi.w3[A][1]) +
                           __mul64hi(d2 << (4 - SH3), oi.w3[A][2]) + 1;
                }
            }
            // mixed terms; z derivatives from the history (planes p - 1 .. p - ORDER) and the new plane
            {
                const IAxis<ORDER> bx = itaps<ORDER>(sB + ly * W + lx + H, 1), ay = itaps<ORDER>(sA + (ly + H) * kOutX + lx, kOutX);
                auto zt = [&](int f, long long newest) -> IAxis<ORDER> {
                    auto h = [&](int back) { return hist[(f * ORDER + (unsigned)(p - back) % ORDER) * kOutThreads]; };
                    if constexpr (ORDER == 4) return {h(3), h(1), h(4), newest};
                    else return {h(2), newest, 0, 0};
                };
                const long long xb = id1<ORDER>(bx), ya = id1<ORDER>(ay), zs = id1<ORDER>(zt(0, ns)),
                                zc = id1<ORDER>(zt(1, nc)), zd = id1<ORDER>(zt(2, nd));
                if (oi.iso) {
                    constexpr long long kSixth = 0x2AAAAAAAAAAAAAABLL;   // 2^64 / 6
                    auto fold = [&](long long v) { return ORDER == 4 ? __mul64hi(v, kSixth) : v >> 2; };
                    m[0] += fold(xb + zc);
                    m[1] += fold(ya + zd);
                    m[2] += fold(zs);
                } else {
                    m[0] += __mul64hi(xb, oi.gm[0]) + __mul64hi(zc, oi.gm[2]);
                    m[1] += __mul64hi(ya, oi.gm[1]) + __mul64hi(zd, oi.gm[2]);
                    m[2] += __mul64hi(zs, oi.gm[2]);
                }
            }
#pragma unroll
            for (int A = 0; A < 3; ++A) cm[A] = (double)m[A];
            // At_ab = D_a W_b + D_b W_a - (2/3) delta_ab div W, then AtAt
            if (!oi.iso) {
#pragma unroll
                for (int a = 0; a < 3; ++a)
#pragma unroll
                    for (int A = 0; A < 3; ++A) g9[a][A] = __mul64hi(g9[a][A] << 1, oi.ga[a]);
            }
            constexpr long long kThird = 0x5555555555555555LL;   // 2^64 / 3
            const long long third = __mul64hi(g9[0][0] + g9[1][1] + g9[2][2], kThird);
            long long at[6] = {(g9[0][0] - third) << 1, (g9[1][1] - third) << 1, (g9[2][2] - third) << 1,
                               g9[0][1] + g9[1][0], g9[0][2] + g9[2][0], g9[1][2] + g9[2][1]};
            if (g.by) {   // with the punctures' analytic part, in FP64
                const double *by = g.by + Pp + (p > 2 * H ? plane : 0);
                double v[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) v[c] = fma((double)at[c], wa, by[c * N]);
                ca = fma(2.0, fma(v[3], v[3], fma(v[4], v[4], v[5] * v[5])), fma(v[0], v[0], fma(v[1], v[1], v[2] * v[2])));
            } else {      // squares of the entries shifted up to 61 bits, high halves of the products
                long long any = 0;
#pragma unroll
                for (int c = 0; c < 6; ++c) any |= at[c] ^ (at[c] >> 63);
                const int sh = __clzll(any) - 3;
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    const long long v = sh < 0 ? at[c] >> -sh : at[c] << sh;
                    at[c] = __mul64hi(v, v);
                }
                const long long sq = at[0] + at[1] + at[2] + ((at[3] + at[4] + at[5]) << 1);
                ca = sq == 0 ? 0.0 : (double)sq * (waa * pow2_biased(1023 - 2 * sh));
            }
        }
        {   // the oldest plane of the history (last read above) becomes the newest
            long long *h = hist + (unsigned)p % ORDER * kOutThreads;
            h[0] = ns;
            h[ORDER * kOutThreads] = nc;
            h[2 * ORDER * kOutThreads] = nd;
        }
        if (p + 1 < NP) reduce_exp(p + 1);
        __syncthreads();
        slot = slot + 1 == NS ? 0 : slot + 1;
    }
    const int done = bad >= 0 ? max(0, bad - 2 * H) : z1 - z0;   // planes whose stencils are done
    if (act) {
        if (done > 0) finish(outer_src(g, in, N, P0 + plane * (done - 1), i, j, z0 + done - 1), P0 + plane * (done - 1), true);
        for (int k = z0 + done; k < z1; ++k) {   // after a NaN or an infinity: directly
            const size_t P = P0 + plane * (k - z0);
            double o[5];
            outer_direct<ORDER, BC>(g, cf, in.u, in.W, i, j, k, o);
            wu = wm = 1.0;
            cl = o[0];
            ca = o[1];
#pragma unroll
            for (int A = 0; A < 3; ++A) cm[A] = o[2 + A];
            finish(outer_src(g, in, N, P, i, j, k), P, true);
        }
    }
    if (fin.periodic) {
        double r[5];
        block_sum<5>(acc, r);
        if (tid == 0)
            for (int a = 0; a < 5; ++a) partial[blockIdx.x * 5 + a] = r[a];
    }
    if (fin.s && finalize_last<5, false>(partial, fin.periodic ? gridDim.x : 0, fin.s->sums, &fin.s->ticket[0]) && tid == 0)
        outer_scalars(fin.s, N, fin.kmode_integrability, fin.K2_fixed, fin.periodic);
}

}  // namespace ctt
