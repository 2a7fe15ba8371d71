// mg_outer.cuh -- FP64 outer residual of the CTT constraints in one fused, tiled pass.
//
// On GB300 an FP64 instruction issues at 2 lanes per clock per SM (conversions to and from FP64
// too), integer and FP32 instructions at 64 to 128, so a residual written in FP64 arithmetic is
// bound by its FP64 instruction count: the two-kernel form this replaces spent ~160 of them per
// cell, 130 on the linear stencils (128^3: 95 us for q, div W, then 589 us; 256^3 Robin 0.6 + 4.8 ms).
// Here the stencils run on 64-bit integers.  Each CTA brings the planes of (u, W) of its tile into
// shared memory as fixed-point numbers in units of 2^(E - 59), one E per field: the exponent of the field's
// largest value in the planes of the stencil.  The weights are small integers (1/8 of the usual 16, 30, 1; the
// spacings are applied at the end), so that with |x| < 2^60 units no sum leaves 64 bits.  A double within 7 binary
// orders of E is represented exactly and a smaller one to half a unit; the eighths of the outer taps are
// truncated to a unit, the sum over the axes of a row to 8 units where its differences exceed the taps.  Sums of
// one field are converted once; sums of different fields are added in FP64 with their own units.
//
// Precision cell by cell: the limit is a cell's own taps, whatever larger values the tile holds.  A cell
// with no tap of 2^53 units in some field is left to FP64 (outer_direct) and done at the end of the CTA, such cells
// packed into full warps; that is one cell in thousands of smooth fields (a field and its gradient small together),
// and all cells outside a steep peak.  Where the values of a whole window have fallen kOutFall
// binary orders below E, the march starts anew in smaller units (it costs about three planes).  Zeros stay exact.
// Every cell is held to a bound from its own taps by tests/test_gpu_outer_local.py, which also prints the errors.
//
// What is left in FP64 is 51 instructions per cell (powers of psi, the source terms, the sums of different fields,
// the block sums), 170 us of that pipe at 128^3 periodic; the kernel takes 312 us there (the two FP64 kernels 684), 2016
// instructions per warp and cell.  (One unit for all fields that never fell took 256 us and lost a cell's digits behind
// every peak of its tile.)
//
// March: 16 x 8 cells per plane, one thread per cell, planes along z through a ring of ORDER + 1
// slots (4 CTAs per SM: their integer and FP64 phases overlap).  The mixed term (1/3) d_i d_j W_j uses
// D_i D_j = D_i o D_j:
//   row x: D_x B + D_z C,  row y: D_y A + D_z D,  row z: D_z A + D_z B
// with A = D_x W_x, B = D_y W_y, C = D_x W_z, D = D_y W_z; A and B of the centre plane are shared with the
// neighbouring cells through shared memory, beside the z history of B, C and D (A's z neighbours are formed again
// from the ring: a fourth history would leave three CTAs per SM).  A cell's FP64 tail runs one plane later,
// among the integer stencils of the next cell.  Boundary values (periodic wrap, Robin, mirror, extrapolation) are
// filled in when a plane is loaded, in FP64 by the rule of fetch_bc, so every cell takes this path.
//
// Values that are NaN or infinite have no fixed-point form: a CTA that meets one leaves its remaining planes to the
// direct FP64 stencils, which propagate it cell by cell.
#pragma once
#include <algorithm>

#include "mg_kernels.cuh"

namespace ctt {

constexpr int kOutX = 16, kOutY = 8, kOutThreads = kOutX * kOutY;
constexpr int kOutMaxZ = 32;          // planes per CTA at most
constexpr int kOutMinExp = 640;       // smallest E (biased): units and their squares stay normal numbers
constexpr int kOutZeroExp = kOutMinExp - 1;   // E of a field that is zero in the whole window
constexpr int kOutFall = 4;           // a march starts anew where the window's largest exponent has fallen this far below E
constexpr int kOutBadExp = 0x7ff;     // biased exponent of NaN and infinity

template <int ORDER> __host__ __device__ constexpr int outer_w() { return kOutX + ORDER; }        // tile + halo
template <int ORDER> __host__ __device__ constexpr int outer_rows() { return kOutY + ORDER; }
template <int ORDER> __host__ __device__ constexpr int outer_plane() { return 4 * outer_w<ORDER>() * outer_rows<ORDER>(); }
template <int ORDER> __host__ __device__ constexpr size_t outer_smem_bytes()
{   // the ring of planes; A (tile columns, all rows) and B (all columns, tile rows) of the centre plane; the
    // z history of B, C and D, ORDER planes of the tile's cells
    return ((size_t)(ORDER + 1) * outer_plane<ORDER>() + (size_t)kOutX * outer_rows<ORDER>() +
            (size_t)kOutY * outer_w<ORDER>() + (size_t)3 * ORDER * kOutThreads) * sizeof(long long);
}

// The smallest |high word| of a cell's largest tap: 2^53 units.  Above, rounding the taps to the unit, at most 2^-53 of
// the largest, adds less to a second difference than FP64's own rounding of the weighted sums (order 4, random and
// smooth taps: rms 2.2 and 1.5 such units at the limit, against 3.1 and 4.4; half as much per binary order above it).
constexpr int kOutEnough = 1 << 21;

// The state and the sources, plain arrays (rho2 may be null: zero).
struct OuterIn {
    const double *u, *W, *rho0, *rho2, *S;
};

// Weights.  Inside a second difference, and for At_ij, the axes' differences are added as integers: with
// unequal spacings each is scaled by its share of the smallest spacing's weight (ratios <= 1 in 64-bit
// fixed point, the high half of a 64 x 64 product); with equal spacings (iso) the shares are 1 and shifts
// suffice.  Sums of different fields have different units: they are added in FP64 with the weights w.
constexpr int kOutWeights = 13;
struct OuterInt {
    int iso;
    long long wl[3];      // Lap u: (hmin/h_a)^2
    long long w3[3][3];   // row A: (3 + delta_Aa) (hmin/h_a)^2
    long long ga[3];      // At_ij: hmin/h_a
    double w[kOutWeights];   // (see outer_weight_field; the shifts' powers of 2 folded in)
    double ca, ca2;       // of At_ij, 1 / (c1 hmin), and its square
};

// The field (0 = u, 1..3 = W_i) in whose unit weight t counts: Lap u, rows x, y, z, then the mixed terms
// D_x D_y W_y, D_x D_z W_z | D_y D_x W_x, D_y D_z W_z | D_z D_x W_x, D_z D_y W_y; at last rows x, y, z without the shift.
__host__ __device__ constexpr int outer_weight_field(int t)
{
    return t < 4 ? t : t >= 10 ? t - 9 : t == 6 || t == 8 ? 1 : t == 4 || t == 9 ? 2 : 3;
}

// Right shifts of second differences before they are added, so that no sum leaves 64 bits: of u; of W in rough cells.
template <int ORDER> __host__ __device__ constexpr int outer_shu() { return ORDER == 4 ? 2 : 1; }
template <int ORDER> __host__ __device__ constexpr int outer_sh3() { return ORDER == 4 ? 4 : 3; }

inline OuterInt make_outer_int(const Geo &g, int order)
{
    OuterInt o;
    const double hmin = fmin(g.h[0], fmin(g.h[1], g.h[2])), hmax = fmax(g.h[0], fmax(g.h[1], g.h[2]));
    // equal spacings, or one unit of the last place apart as (hi - lo) / n may leave them: their mean is then as near to
    // each as a rounded 1/h^2 is to its own
    o.iso = hmax <= nextafter(hmin, hmax);
    const long double hb = o.iso ? ((long double)hmin + (long double)hmax) / 2 : (long double)hmin;
    auto fix = [](long double v, int bits) {  // v 2^bits, at most 2^63 - 1
        const long double s = ldexpl(v, bits);
        return s >= 9223372036854775807.0L ? 9223372036854775807LL : (long long)(s + 0.5L);
    };
    for (int a = 0; a < 3; ++a) {
        const long double r = (long double)hmin / (long double)g.h[a];
        o.wl[a] = fix(r * r, 62);
        for (int A = 0; A < 3; ++A) o.w3[A][a] = fix((A == a ? 4.0L : 3.0L) * r * r, 60);
        o.ga[a] = fix(r, 63);
    }
    // (id2 is c2 h^2 D2, id1 is c1 h D)
    const long double c2 = order == 4 ? 1.5L : 1.0L, c1 = order == 4 ? 1.5L : 2.0L;
    const int shu = order == 4 ? outer_shu<4>() : outer_shu<2>(), sh3 = order == 4 ? outer_sh3<4>() : outer_sh3<2>();
    o.w[0] = (double)(ldexpl(1.0L, shu) / (c2 * hb * hb));
    for (int A = 0; A < 3; ++A) {
        o.w[1 + A] = (double)(ldexpl(1.0L, sh3) / (3.0L * c2 * hb * hb));
        o.w[10 + A] = (double)(1.0L / (3.0L * c2 * hb * hb));
    }
    constexpr int pair[6][2] = {{0, 1}, {0, 2}, {1, 0}, {1, 2}, {2, 0}, {2, 1}};
    for (int t = 0; t < 6; ++t)
        o.w[4 + t] = (double)(1.0L / (3.0L * c1 * c1 * (long double)g.h[pair[t][0]] * (long double)g.h[pair[t][1]]));
    o.ca = (double)(1.0L / (c1 * hb));
    o.ca2 = (double)(1.0L / (c1 * c1 * hb * hb));
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

// 1.5 h D f (order 4) or 2 h D f
template <int ORDER>
__device__ __forceinline__ long long id1(const IAxis<ORDER> &t)
{
    if constexpr (ORDER == 4) return (t.p1 - t.m1) - ((t.p2 - t.m2) >> 3);
    else return t.p1 - t.m1;
}

// 1.5 h^2 D2 f (order 4) or h^2 D2 f; k0 = (30 / 8) f or 2 f.  (Partial sums may wrap, the result does not: weights of
// total size 8 or 4 on values below 2^60.)
template <int ORDER>
__device__ __forceinline__ long long id2(const IAxis<ORDER> &t, unsigned long long k0)
{
    typedef unsigned long long U;
    if constexpr (ORDER == 4) return (long long)((((U)t.p1 + (U)t.m1) << 1) - (U)((t.p2 + t.m2) >> 3) - k0);
    else return (long long)((U)t.p1 + (U)t.m1 - k0);
}

template <int ORDER>
__device__ __forceinline__ unsigned long long ik0(long long f)
{
    if constexpr (ORDER == 4) return ((unsigned long long)f << 2) - (unsigned long long)(f >> 2);
    else return (unsigned long long)f << 1;
}

// x in units of 2^(E - 59), so below 2^60: an FP64 bit pattern of biased exponent <= E, rounded to nearest.  (The
// implicit bit that zero and denormal numbers do not have is shifted out: E >= kOutMinExp.)
__device__ __forceinline__ long long to_fixed(double x, int E)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mh = (__funnelshift_l(lo, hi, 10) & 0x3fffffffu) | 0x40000000u;   // mantissa, leading one at bit 62
    const unsigned long long t = ((unsigned long long)mh << 32) | (lo << 10);
    const int d = min(E - (int)((hi >> 20) & 0x7ffu) + 2, 63);
    const long long v = (long long)(((t >> d) + 1) >> 1);
    return (int)hi < 0 ? -v : v;
}

// x / 2^S, rounded to nearest
template <int S>
__device__ __forceinline__ long long rshift(long long x)
{
    if constexpr (S == 0) return x;
    else return (x + (1LL << (S - 1))) >> S;
}

__device__ __forceinline__ double pow2_biased(int e) { return __hiloint2double(e << 20, 0); }   // 2^(e - 1023)

// Sums of second differences over the axes, in units of the weights w.  (The products' floors are centred by one unit, none
// where all differences are zero.)  Lap u:
template <int ORDER>
__device__ __forceinline__ long long isum_u(const OuterInt &oi, const IAxis<ORDER> &x, const IAxis<ORDER> &y,
                                            const IAxis<ORDER> &z, long long c)
{
    constexpr int S = outer_shu<ORDER>();
    const unsigned long long k0 = ik0<ORDER>(c);
    const long long d0 = id2<ORDER>(x, k0), d1 = id2<ORDER>(y, k0), d2 = id2<ORDER>(z, k0);
    if (oi.iso) return rshift<S>(d0) + rshift<S>(d1) + rshift<S>(d2);
    return __mul64hi(d0 << (2 - S), oi.wl[0]) + __mul64hi(d1 << (2 - S), oi.wl[1]) + __mul64hi(d2 << (2 - S), oi.wl[2]) +
           ((d0 | d1 | d2) != 0);
}

// Row A: three times Lap W_A + (1/3) D_AA W_A, weights of total size 10.  Differences below 2^59 need no shift before the
// sum; above (a rough cell: its differences are larger than its taps) they are shifted and rough is set.
template <int ORDER>
__device__ __forceinline__ long long isum_w(const OuterInt &oi, int A, const IAxis<ORDER> &x, const IAxis<ORDER> &y,
                                            const IAxis<ORDER> &z, long long c, bool &rough)
{
    constexpr int S = outer_sh3<ORDER>();
    const unsigned long long k0 = ik0<ORDER>(c);
    long long d0 = id2<ORDER>(x, k0), d1 = id2<ORDER>(y, k0), d2 = id2<ORDER>(z, k0);
    auto mag = [](long long d) { return (int)(d >> 32) ^ ((int)(d >> 32) >> 31); };
    rough = (mag(d0) | mag(d1) | mag(d2)) >= (1 << 27);
    if (oi.iso) {
        if (rough) {
            d0 = rshift<S>(d0);
            d1 = rshift<S>(d1);
            d2 = rshift<S>(d2);
        }
        const long long s = d0 + d1 + d2;
        return (s << 1) + s + (A == 0 ? d0 : A == 1 ? d1 : d2);
    }
    const int l = rough ? 4 - S : 4;
    return __mul64hi(d0 << l, oi.w3[A][0]) + __mul64hi(d1 << l, oi.w3[A][1]) + __mul64hi(d2 << l, oi.w3[A][2]) +
           ((d0 | d1 | d2) != 0);
}

// ---------------------------------------------------------------- out-of-line parts
// Boundary value of field fi (0 = u, 1..3 = W_i) at a cell outside the box.
template <int BC>
__device__ __noinline__ double outer_ghost(const double *f, int fi, const Geo &g, int i, int j, int k)
{
    return fetch_bc<double, BC>(f, fi, g, i, j, k);
}

// A field around a cell whose taps all lie inside the box.
struct OuterInner {
    const double *p;
    int sy;
    size_t sz;
    __device__ __forceinline__ double operator()(int dx, int dy, int dz) const
    {
        return p[dx + dy * sy + dz * (long long)sz];
    }
};
template <int H>
__device__ __forceinline__ bool outer_inner(const Geo &g, int i, int j, int k)
{
    return min(min(min(i, j), k), min(min(g.n[0] - 1 - i, g.n[1] - 1 - j), g.n[2] - 1 - k)) >= H;
}

// The direct FP64 form at a cell: out = (Lap u, momentum rows, AtAt).
template <int ORDER, int BC>
__device__ __noinline__ void outer_direct(const Geo &g, const Coef<double> &cf, const double *u, const double *W, int i,
                                          int j, int k, double *out)
{
    const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
    const size_t p = (size_t)i + (size_t)g.n[0] * ((size_t)j + (size_t)g.n[1] * k);
    double lu, aa, mom[3];
    const double *by = g.by ? g.by + p : nullptr;
    if (outer_inner<ORDER / 2>(g, i, j, k)) {
        const size_t sz = (size_t)g.n[0] * g.n[1];
        const OuterInner a0{u + p, g.n[0], sz}, a1{W + p, g.n[0], sz}, a2{W + N + p, g.n[0], sz},
            a3{W + 2 * N + p, g.n[0], sz};
        outer_cell<ORDER>(a0, a1, a2, a3, cf, lu, aa, mom, by, N);
    } else {
        AccB<double, BC> a0{u, 0, &g, i, j, k}, a1{W, 1, &g, i, j, k}, a2{W + N, 2, &g, i, j, k},
            a3{W + 2 * N, 3, &g, i, j, k};
        outer_cell<ORDER>(a0, a1, a2, a3, cf, lu, aa, mom, by, N);
    }
    out[0] = lu;
    out[1] = mom[0];
    out[2] = mom[1];
    out[3] = mom[2];
    out[4] = aa;
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

// The FP64 tail of a cell: aterm = (1/8) psi^-7 AtAt, m2 = rho2 psi, s8 = 8 pi psi^6, p5 = psi^5.
struct OuterTail {
    double aterm, m2, s8, p5;
};
__device__ __forceinline__ OuterTail outer_tail(const OuterSrc &c, double aa)
{
    const double psi = c.bg + c.u, p2 = psi * psi, p4 = p2 * p2, p5 = p4 * psi, p6 = p5 * psi;
    return {(0.125 * aa) * recip_f64(p6 * psi), c.rho2 * psi, (8.0 * kPi) * p6, p5};
}

// ---------------------------------------------------------------- the fused residual
//   R0 = Lap u + (1/8) psi^-7 AtAt + 2 pi rho2 psi     (F_psi without its psi^5 terms, see f_psi)
//   R1..3 = Lap W_i + (1/3) d_i d_j W_j - 8 pi psi^6 S_i                 (F_W before adding m_i)
//   R4 = AtAt (null: not stored; pass 2 forms the linearisation coefficient from it)
// and, on periodic boxes, one row of 5 partial sums per CTA; the last CTA finishes the outer
// scalars when fin.s is set.
template <int ORDER, int BC>
__global__ void __launch_bounds__(kOutThreads, 4)
    k_outer_residual(const __grid_constant__ Geo g, const __grid_constant__ Coef<double> cf,
                     const __grid_constant__ OuterInt oi, OuterIn in, double *__restrict__ R, double *__restrict__ R4,
                     double *__restrict__ partial, OuterGrid tg, OuterFin fin)
{
    constexpr int H = ORDER / 2, W = outer_w<ORDER>(), RW = outer_rows<ORDER>(), FE = W * RW, PE = outer_plane<ORDER>(),
                  NS = ORDER + 1;
    constexpr int NE = (FE + kOutThreads - 1) / kOutThreads;   // loaded elements per thread, field and plane
    static_assert(2 * H * kOutX + 2 * H * kOutY <= kOutThreads, "one halo value of A or B per thread");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    long long *ring = reinterpret_cast<long long *>(smem_raw);
    long long *sA = ring + NS * PE, *sB = sA + kOutX * RW;      // A[row][kOutX], B[row of the tile][W]
    long long *hist = sB + kOutY * W + threadIdx.x;             // [B, C, D][plane % ORDER][thread]
    __shared__ int4 sM[8];                                      // [plane % 8]: largest |high word| of u, W_x, W_y, W_z
    __shared__ double wt[kOutWeights];                          // weights in the current units
    __shared__ int4 sE, sT;                                     // exponents of the units; kOutEnough, or 0 for a zero field

    const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], tid = threadIdx.x;
    const size_t plane = (size_t)nx * ny;
    int b = blockIdx.x;
    const int x0 = (b % tg.ntx) * kOutX;
    b /= tg.ntx;
    const int y0 = (b % tg.nty) * kOutY;
    const int zb = (b / tg.nty) * tg.zc, z1 = min(zb + tg.zc, nz);
    int z0 = zb;             // first plane of the current march
    unsigned later = 0;      // bit k: the thread's cell in plane zb + k is left to FP64 (kOutMaxZ planes at most)
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
    auto reduce_max = [&](int p) {   // into sM[p % 8]
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            unsigned m = 0;
#pragma unroll
            for (int t = 0; t < NE; ++t) m = max(m, (unsigned)__double2hiint(raw[f][t]) & 0x7fffffffu);
            m = __reduce_max_sync(0xffffffffu, m);
            if ((tid & 31) == 0) atomicMax(reinterpret_cast<int *>(&sM[p & 7]) + f, (int)m);
        }
    };
    double acc[5] = {0, 0, 0, 0, 0};
    // the results at the centre cell of the last plane, finished one plane later: their FP64 tail then runs
    // interleaved with the integer stencils of the next cell
    double cl = 0.0, cm[3] = {0.0, 0.0, 0.0}, ca = 0.0;
    auto finish = [&](const OuterSrc &c, size_t P, bool on) {
        const OuterTail t = outer_tail(c, ca);
        if (fin.periodic) {   // (other boxes use no sums)
            acc[0] += on ? fma(2.0 * kPi, fma(c.rho0, t.p5, t.m2), t.aterm) : 0.0;
            acc[1] += on ? t.p5 : 0.0;
            const double s8on = on ? t.s8 : 0.0;
#pragma unroll
            for (int A = 0; A < 3; ++A) acc[2 + A] = fma(s8on, c.S[A], acc[2 + A]);
        }
        if (on) {
            R[P] = fma(2.0 * kPi, t.m2, t.aterm + cl);
#pragma unroll
            for (int A = 0; A < 3; ++A) R[(1 + A) * N + P] = fma(-t.s8, c.S[A], cm[A]);
            if (R4) R4[P] = ca;
        }
    };

    // A march from plane z0 on: it ends at z1, or earlier where values have left the ring that were far larger than what is
    // left (the next march starts there, in smaller units), or at a plane that holds a NaN or an infinity.
    bool bad = false;
    while (z0 < z1 && !bad) {
        const int NP = z1 - z0 + 2 * H;
        __syncthreads();
        if (tid < 32) reinterpret_cast<int *>(sM)[tid] = 0;
        load(0);
        __syncthreads();
        reduce_max(0);
        __syncthreads();
        int slot = 0;              // p % NS
        int done = z1 - z0;        // cells whose stencils this march forms
        const int cell = (ly + H) * W + lx + H;
        const size_t P0 = (size_t)i + (size_t)nx * j + plane * z0;
        for (int p = 0; p < NP; ++p) {
            // phase 0: plane p into the ring in the current units (grown when it holds larger values),
            // A and B of the centre plane p - H for the tile's neighbours
            int E[4];
            {
                int top[4] = {0, 0, 0, 0};   // largest |high word| of each field in the planes p - 2 H .. p
#pragma unroll
                for (int s = 0; s <= 2 * H; ++s) {
                    const int4 m = sM[(p - s) & 7];
                    top[0] = max(top[0], m.x);
                    top[1] = max(top[1], m.y);
                    top[2] = max(top[2], m.z);
                    top[3] = max(top[3], m.w);
                }
                const int4 old = sE;
                const int was[4] = {old.x, old.y, old.z, old.w};
                int up = 0, down = 0, all = 0;
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    const int e = top[f] == 0 ? kOutZeroExp : max(top[f] >> 20, kOutMinExp);
                    all = max(all, top[f] >> 20);
                    E[f] = p > 0 ? max(e, was[f]) : e;
                    up |= E[f] ^ was[f];
                    down = max(down, E[f] - e);
                }
                bad = all == kOutBadExp;
                if (bad || (down >= kOutFall && p > 2 * H)) {
                    done = max(0, p - 2 * H);
                    break;
                }
                if (up || p == 0) {   // rare: rescale what the ring and the history hold
                    int rise[4];
#pragma unroll
                    for (int f = 0; f < 4; ++f) rise[f] = min(62, E[f] - was[f]);
                    if (p > 0) {
                        for (int e = tid; e < NS * PE; e += kOutThreads) {
                            const int f = (e % PE) / FE;
                            const int d = f == 0 ? rise[0] : f == 1 ? rise[1] : f == 2 ? rise[2] : rise[3];
                            ring[e] = (ring[e] + ((1LL << d) >> 1)) >> d;
                        }
#pragma unroll
                        for (int k = 0; k < 3 * ORDER; ++k) {
                            const int d = k < ORDER ? rise[2] : rise[3];
                            hist[k * kOutThreads] = (hist[k * kOutThreads] + ((1LL << d) >> 1)) >> d;
                        }
                    }
                    __syncthreads();   // (every thread has read the old exponents)
                    if (tid == 0) {
                        auto enough = [](int e) { return e == kOutZeroExp ? 0 : kOutEnough; };
                        sE = make_int4(E[0], E[1], E[2], E[3]);
                        sT = make_int4(enough(E[0]), enough(E[1]), enough(E[2]), enough(E[3]));
                    }
                    if (tid < kOutWeights) {
                        const int f = outer_weight_field(tid);
                        wt[tid] = oi.w[tid] * pow2_biased((f == 0 ? E[0] : f == 1 ? E[1] : f == 2 ? E[2] : E[3]) - 59);
                    }
                }
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
                        if (tid + t * kOutThreads < FE) dst[f * FE + t * kOutThreads] = to_fixed(raw[f][t], E[f]);
            }
            if (p + 1 < NP) load(p + 1);
            const int cs = slot >= H ? slot - H : slot - H + NS;   // slot of the centre plane
            const long long *q = ring + cs * PE + cell;
            long long gxx = 0, gyy = 0;   // D_x W_x, D_y W_y at the cell
            if (full) {
                gxx = id1<ORDER>(itaps<ORDER>(q + FE, 1));
                gyy = id1<ORDER>(itaps<ORDER>(q + 2 * FE, W));
                sA[(ly + H) * kOutX + lx] = gxx;
                sB[ly * W + lx + H] = gyy;
                const long long *c1 = ring + cs * PE + FE, *c2 = c1 + FE;   // W_x, W_y
                if (tid < 2 * H * kOutX) {   // A in the rows above and below the tile
                    const int r = tid / kOutX, row = r < H ? r : r + kOutY;
                    sA[row * kOutX + lx] = id1<ORDER>(itaps<ORDER>(c1 + row * W + H + lx, 1));
                } else if (tid < 2 * H * (kOutX + kOutY)) {   // B in the columns left and right of it
                    const int e = tid - 2 * H * kOutX, c = e % (2 * H), col = c < H ? c : c + kOutX, row = e / (2 * H);
                    sB[row * W + col] = id1<ORDER>(itaps<ORDER>(c2 + (H + row) * W + col, W));
                }
            }
            __syncthreads();
            // phase 1: the new plane's first derivatives; the previous cell's FP64 tail and the centre
            // plane's cell, in one block
            if (tid < 4) reinterpret_cast<int *>(&sM[(p + 2) & 7])[tid] = 0;
            long long nb, nc, nd;   // B, C, D of the new plane (p = centre + H)
            {
                const long long *n = ring + slot * PE + cell;
                nb = id1<ORDER>(itaps<ORDER>(n + 2 * FE, W));
                nc = id1<ORDER>(itaps<ORDER>(n + 3 * FE, 1));
                nd = id1<ORDER>(itaps<ORDER>(n + 3 * FE, W));
            }
            auto remember = [&]() {   // the history's oldest plane becomes the newest
                long long *h = hist + (unsigned)p % ORDER * kOutThreads;
                h[0] = nb;
                h[ORDER * kOutThreads] = nc;
                h[2 * ORDER * kOutThreads] = nd;
            };
            if (!(full && act)) {
                remember();
            } else {
                finish(src, Pp, p > 2 * H && !((later >> (z0 - zb + zprev)) & 1));
                const int4 e4 = sE;
                const int Ew[3] = {e4.y, e4.z, e4.w};
                const bool wide = max(max(Ew[0], Ew[1]), Ew[2]) > min(min(Ew[0], Ew[1]), Ew[2]) + 2;
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
                // Whether the taps of a field reach kOutEnough: its centre and outermost taps, and where the components'
                // units are far apart (a row may then see the mixed term of a much coarser component) also those in
                // either plane of a mixed term.  (High words; a field that is zero in the whole window is exact.)
                bool small = false;
                auto reaches = [&](int f, const IAxis<ORDER> &x, const IAxis<ORDER> &y, const IAxis<ORDER> &z,
                                   long long c) {
                    auto line = [&](const IAxis<ORDER> &t) {   // largest |high word|
                        const int l = (int)((ORDER == 4 ? t.m2 : t.m1) >> 32), r = (int)((ORDER == 4 ? t.p2 : t.p1) >> 32);
                        const int h = (int)(c >> 32);
                        return max(max(max(l, r), h), ~min(min(l, r), h));
                    };
                    const int a[3] = {line(x), line(y), line(z)};
                    const int own = f == 0 ? 0 : a[f - 1], o1 = f == 0 ? 0 : a[f % 3], o2 = f == 0 ? 0 : a[(f + 1) % 3];
                    const int m = f > 0 && wide ? max(own, min(o1, o2)) : max(max(a[0], a[1]), a[2]);
                    small = small || m < reinterpret_cast<const int *>(&sT)[f];
                };
                {
                    const IAxis<ORDER> tx = itaps<ORDER>(q, 1), ty = itaps<ORDER>(q, W), tz = ztaps(q);
                    reaches(0, tx, ty, tz, q[0]);
                    cl = (double)isum_u<ORDER>(oi, tx, ty, tz, q[0]) * wt[0];
                }
                double mix[3];
                // mixed terms; z derivatives from the history (planes p - 1 .. p - ORDER) and the new plane, those
                // of A from the ring
                {
                    const IAxis<ORDER> bx = itaps<ORDER>(sB + ly * W + lx + H, 1);
                    const IAxis<ORDER> ay = itaps<ORDER>(sA + (ly + H) * kOutX + lx, kOutX);
                    auto zt = [&](int f, long long newest) -> IAxis<ORDER> {
                        auto h = [&](int back) { return hist[(f * ORDER + (unsigned)(p - back) % ORDER) * kOutThreads]; };
                        if constexpr (ORDER == 4) return {h(3), h(1), h(4), newest};
                        else return {h(2), newest, 0, 0};
                    };
                    IAxis<ORDER> az{0, 0, 0, 0};
                    {
                        auto dx = [&](int s) { return id1<ORDER>(itaps<ORDER>(q + FE + zo[s], 1)); };
                        if constexpr (ORDER == 4) az = {dx(1), dx(2), dx(0), dx(3)};
                        else az = {dx(0), dx(1), 0, 0};
                    }
                    const long long xb = id1<ORDER>(bx), ya = id1<ORDER>(ay), za = id1<ORDER>(az),
                                    zb = id1<ORDER>(zt(0, nb)), zc = id1<ORDER>(zt(1, nc)), zd = id1<ORDER>(zt(2, nd));
                    mix[0] = fma((double)xb, wt[4], (double)zc * wt[5]);
                    mix[1] = fma((double)ya, wt[6], (double)zd * wt[7]);
                    mix[2] = fma((double)za, wt[8], (double)zb * wt[9]);
                    remember();
                }
                // momentum rows, Lap W_A + (1/3) D_AA W_A part, and the first derivatives of W_A
                long long g9[3][3];   // g9[a][A] = D_a W_A
#pragma unroll
                for (int A = 0; A < 3; ++A) {
                    const long long *w = q + (1 + A) * FE;
                    const IAxis<ORDER> tx = itaps<ORDER>(w, 1), ty = itaps<ORDER>(w, W), tz = ztaps(w);
                    reaches(1 + A, tx, ty, tz, w[0]);
                    g9[0][A] = A == 0 ? gxx : id1<ORDER>(tx);
                    g9[1][A] = A == 1 ? gyy : id1<ORDER>(ty);
                    g9[2][A] = id1<ORDER>(tz);
                    bool rough;
                    const long long m = isum_w<ORDER>(oi, A, tx, ty, tz, w[0], rough);
                    cm[A] = fma((double)m, wt[(rough ? 1 : 10) + A], mix[A]);
                }
                // At_ab = D_a W_b + D_b W_a - (2/3) delta_ab div W, then AtAt.  The components' derivatives first in one
                // unit, 2^(U - 59), in which the largest of them has its top bit at 60.
                int U = -(1 << 20);
#pragma unroll
                for (int A = 0; A < 3; ++A) {
                    long long any = 0;
#pragma unroll
                    for (int a = 0; a < 3; ++a) any |= g9[a][A] ^ (g9[a][A] >> 63);
                    if (any) U = max(U, Ew[A] + 3 - __clzll(any));
                }
#pragma unroll
                for (int A = 0; A < 3; ++A) {
                    const int n = Ew[A] - U, l = min(63, max(n, 0)), r = min(63, max(-n, 0));
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        g9[a][A] = g9[a][A] << l >> r;
                        if (!oi.iso) g9[a][A] = __mul64hi(g9[a][A] << 1, oi.ga[a]);   // (after the shift: no bits are lost)
                    }
                }
                constexpr long long kThird = 0x5555555555555555LL;   // 2^64 / 3
                const long long third = __mul64hi(g9[0][0] + g9[1][1] + g9[2][2], kThird);
                long long at[6] = {(g9[0][0] - third) << 1, (g9[1][1] - third) << 1, (g9[2][2] - third) << 1,
                                   g9[0][1] + g9[1][0], g9[0][2] + g9[2][0], g9[1][2] + g9[2][1]};
                if (g.by) {   // with the punctures' analytic part, in FP64
                    const double *by = g.by + Pp + (p > 2 * H ? plane : 0);
                    const double wa = oi.ca * pow2_biased(min(2046, max(0, U - 59)));
                    double v[6];
#pragma unroll
                    for (int c = 0; c < 6; ++c) v[c] = fma((double)at[c], wa, by[c * N]);
                    ca = fma(2.0, fma(v[3], v[3], fma(v[4], v[4], v[5] * v[5])),
                             fma(v[0], v[0], fma(v[1], v[1], v[2] * v[2])));
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
                    const int e = 2 * (U - 1082) + 64 - 2 * sh;
                    ca = sq == 0 ? 0.0 : (double)sq * oi.ca2 * pow2_biased(min(2046, max(0, e + 1023)));
                }
                if (small) later |= 1u << (z0 - zb + p - 2 * H);
            }
            if (p + 1 < NP) reduce_max(p + 1);
            __syncthreads();
            slot = slot + 1 == NS ? 0 : slot + 1;
        }
        if (act && done > 0 && !((later >> (z0 - zb + done - 1)) & 1)) {
            const size_t P = P0 + plane * (done - 1);
            finish(outer_src(g, in, N, P, i, j, z0 + done - 1), P, true);
        }
        z0 += done;
    }
    // The cells left to FP64, and those of the planes not reached because of a NaN or an infinity: listed in shared memory
    // (in a fixed order), so that they fill whole warps.
    if (!act) later = 0;
    else if (z0 < z1) later |= (0xffffffffu >> (32 - (z1 - z0))) << (z0 - zb);
    if (__syncthreads_or(later != 0)) {
        __shared__ int base[kOutThreads / 32];
        unsigned short *list = reinterpret_cast<unsigned short *>(smem_raw);
        static_assert(kOutThreads * kOutMaxZ * sizeof(unsigned short) <= outer_smem_bytes<2>(), "the list fits");
        const int own = __popc(later), lane = tid & 31;
        int before = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, before, o);
            before += lane >= o ? v : 0;
        }
        if (lane == 31) base[tid >> 5] = before;
        __syncthreads();
        before -= own;
        int total = 0;
#pragma unroll
        for (int w = 0; w < kOutThreads / 32; ++w) {
            before += w < (tid >> 5) ? base[w] : 0;
            total += base[w];
        }
        for (unsigned m = later; m; m &= m - 1) list[before++] = (unsigned short)(tid | ((__ffs(m) - 1) << 8));
        __syncthreads();
        for (int e = tid; e < total; e += kOutThreads) {
            const int t = list[e] & 255, k = zb + (list[e] >> 8), ci = x0 + (t & (kOutX - 1)), cj = y0 + t / kOutX;
            const size_t P = (size_t)ci + (size_t)nx * cj + plane * k;
            double v[5];
            outer_direct<ORDER, BC>(g, cf, in.u, in.W, ci, cj, k, v);
            cl = v[0];
#pragma unroll
            for (int A = 0; A < 3; ++A) cm[A] = v[1 + A];
            ca = v[4];
            finish(outer_src(g, in, N, P, ci, cj, k), P, true);
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
