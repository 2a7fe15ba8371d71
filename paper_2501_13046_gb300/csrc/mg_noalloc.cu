// mg_noalloc.cu -- constraint norms of a caller-held state without any device allocation.
//
// For callers that must not allocate device memory: the scratch of this entry point (the
// four FP64 pass-1 fields, the per-block reduction partials and the reduced scalars) lives in
// one file-scope device array, sized for grids of at most kNoallocMaxCells cells, that every
// GPU loading the library holds until the process exits.  The arithmetic is that of the
// context path (mg_residual_norms): the same per-cell residual, integrability K^2 and
// momentum-source means, and max-norms of H and M.
#include <mutex>

#include "mg_common.cuh"

namespace ctt {
namespace {

constexpr size_t kNoallocMaxCells = 64 * 64 * 64;                 // 262,144 cells
constexpr size_t kNoallocR = 4 * kNoallocMaxCells;                // pass-1 output, 4 FP64 fields
constexpr size_t kNoallocPartials = 4096 * 5;                      // block partials: 5 per CTA of the residual
constexpr size_t kNoallocScalars = 64;                            // >= sizeof(Scalars) / 8
constexpr size_t kNoallocDoubles = kNoallocR + kNoallocPartials + kNoallocScalars;   // 8.55 MB
static_assert(kNoallocPartials >= (size_t)kRedBlocks * 4, "the norms' partials fit too");
static_assert(sizeof(Scalars) <= kNoallocScalars * sizeof(double), "scalar slot too small");

static __device__ __align__(256) double g_noalloc_scratch[kNoallocDoubles];

// Host code cannot use g_noalloc_scratch as a device address; each device's address is
// looked up once, with that device current, and cached here.
constexpr int kMaxDevices = 64;
std::mutex g_addr_mu;
double *g_addr[kMaxDevices] = {};

mg_status scratch_address(double **out)
{
    int dev = -1;
    CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(MG_ERR_UNSUPPORTED, "device index out of range");
    std::lock_guard<std::mutex> lock(g_addr_mu);
    if (!g_addr[dev]) {
        void *p = nullptr;
        CK(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        g_addr[dev] = static_cast<double *>(p);
    }
    *out = g_addr[dev];
    return MG_OK;
}

// Maxima of |H| and |M_i|, finished in the last block.
__global__ void __launch_bounds__(256) k_noalloc_norms(Geo g, const double *__restrict__ u,
                                                       const double *__restrict__ R,
                                                       const double *__restrict__ rho0, Scalars *s,
                                                       double *__restrict__ partial)
{
    const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
    const double nk = -s->K2 / 12.0, m[3] = {s->msrc[0], s->msrc[1], s->msrc[2]};
    unsigned long long mxu[4] = {0, 0, 0, 0};
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < N; p += (size_t)gridDim.x * blockDim.x) {
        int i = (int)(p % g.n[0]);
        size_t rest = p / g.n[0];
        int j = (int)(rest % g.n[1]);
        int k = (int)(rest / g.n[1]);
        double psi = psi_background(g, i, j, k) + u[p];
        double p2 = psi * psi, p4 = p2 * p2, p5 = p4 * psi;
        const PsiInverse inv = psi_inverse(psi, p5);
        max_abs(mxu[0], -8.0 * inv.i5 * f_psi(R[p], rho0[p], p5, nk));
#pragma unroll
        for (int a = 0; a < 3; ++a) max_abs(mxu[1 + a], inv.i6 * (R[(1 + a) * N + p] + m[a]));
    }
    double mx[4], r[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) mx[a] = max_value(mxu[a]);
    block_max<4>(mx, r);
    if (threadIdx.x == 0)
        for (int a = 0; a < 4; ++a) partial[blockIdx.x * 4 + a] = r[a];
    finalize_last<4, true>(partial, gridDim.x, s->norms, &s->ticket[1]);
}

mg_status check_config(const mg_config *c)
{
    if (!c) return fail(MG_ERR_INVALID_ARG, "null config");
    for (int a = 0; a < 3; ++a)
        if (c->n[a] < 3 || !(c->hi[a] > c->lo[a])) return fail(MG_ERR_INVALID_ARG, "bad grid size or box");
    if (c->order != 2 && c->order != 4) return fail(MG_ERR_INVALID_ARG, "order must be 2 or 4");
    if (c->bc != MG_BC_PERIODIC && c->bc != MG_BC_ROBIN) return fail(MG_ERR_INVALID_ARG, "bad bc");
    if (c->k_mode != MG_K_FIXED && c->k_mode != MG_K_INTEGRABILITY) return fail(MG_ERR_INVALID_ARG, "bad k_mode");
    if (c->k_mode == MG_K_INTEGRABILITY && c->bc != MG_BC_PERIODIC)
        return fail(MG_ERR_INVALID_ARG, "integrability K needs a periodic box");
    if (c->npunct < 0 || c->npunct > 2) return fail(MG_ERR_INVALID_ARG, "npunct must be 0..2");
    if (c->npunct > 0 && c->bc == MG_BC_PERIODIC) return fail(MG_ERR_UNSUPPORTED, "punctures need Robin boundaries");
    for (int p = 0; p < c->npunct; ++p)
        for (int a = 0; a < 3; ++a)
            if (c->punct_P[p][a] != 0.0 || c->punct_S[p][a] != 0.0)
                return fail(MG_ERR_UNSUPPORTED, "Bowen-York punctures are not supported by the allocation-free norms");
    if (c->reflect != 0) return fail(MG_ERR_UNSUPPORTED, "symmetry planes are not supported by the allocation-free norms");
    if (c->extrap != 0)
        return fail(MG_ERR_UNSUPPORTED, "extrapolating faces are not supported by the allocation-free norms");
    if (!std::isfinite(c->K)) return fail(MG_ERR_INVALID_ARG, "K not finite");
    // each product is checked before the next one is formed, so no cell count wraps around
    const char *msg = "mg_residual_norms_noalloc: the grid exceeds the static scratch limit of 262144 cells (64^3)";
    for (int a = 0; a < 3; ++a)
        if ((size_t)c->n[a] > kNoallocMaxCells) return fail(MG_ERR_INVALID_ARG, msg);
    const size_t n01 = (size_t)c->n[0] * c->n[1];
    if (n01 > kNoallocMaxCells || n01 * c->n[2] > kNoallocMaxCells) return fail(MG_ERR_INVALID_ARG, msg);
    return MG_OK;
}

}  // namespace
}  // namespace ctt

using namespace ctt;

extern "C" mg_status mg_residual_norms_noalloc(const mg_config *cfg, const double *u, const double *W,
                                               const double *rho0, const double *rho2, const double *S,
                                               double out[4], double *K2, void *cuda_stream)
{
    CKS(check_config(cfg));
    if (!u || !W || !rho0 || !S || !out) return fail(MG_ERR_INVALID_ARG, "null pointer");
    double *scratch = nullptr;
    CKS(scratch_address(&scratch));
    cudaStream_t st = (cudaStream_t)cuda_stream;
    Geo g;
    std::memset(&g, 0, sizeof(g));
    for (int a = 0; a < 3; ++a) {
        g.n[a] = cfg->n[a];
        g.lo[a] = cfg->lo[a];
        g.h[a] = (cfg->hi[a] - cfg->lo[a]) / cfg->n[a];
        g.lof[a] = (float)g.lo[a];
        g.hf[a] = (float)g.h[a];
    }
    g.npunct = cfg->npunct;
    for (int p = 0; p < cfg->npunct; ++p) {
        g.pm[p] = cfg->punct_m[p];
        for (int a = 0; a < 3; ++a) g.px[p][a] = cfg->punct_x[p][a];
    }
    const size_t N = (size_t)g.n[0] * g.n[1] * g.n[2];
    double *R = scratch;
    double *partial = scratch + kNoallocR;
    Scalars *sc = reinterpret_cast<Scalars *>(scratch + kNoallocR + kNoallocPartials);
    // the scalars are read back below: start them at zero on every call
    CK(cudaMemsetAsync(sc, 0, sizeof(Scalars), st));
    const int g1 = grid_for(N, kRedBlocks);
    const OuterGrid tg = outer_grid(g);
    if ((size_t)outer_ctas(g, tg) * 5 > kNoallocPartials)   // (at most 3641 CTAs on 262144 cells: 3 x 29127 x 3)
        return fail(MG_ERR_INVALID_ARG, "mg_residual_norms_noalloc: too many tiles for the static scratch");
    const OuterIn in{u, W, rho0, rho2, S};
    const OuterFin fin{sc, cfg->k_mode == MG_K_INTEGRABILITY, cfg->bc == MG_BC_PERIODIC, cfg->K * cfg->K};
    cudaError_t attr = cudaSuccess;
    auto launch1 = [&](auto O, auto B) {
        constexpr int ORDER = decltype(O)::value, BC = decltype(B)::value;
        attr = cudaFuncSetAttribute(k_outer_residual<ORDER, BC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)outer_smem_bytes<ORDER>());
        k_outer_residual<ORDER, BC><<<outer_ctas(g, tg), kOutThreads, outer_smem_bytes<ORDER>(), st>>>(
            g, make_coef<double>(g, cfg->order), make_outer_int(g, cfg->order), in, R, nullptr, partial, tg, fin);
    };
    using I2 = std::integral_constant<int, 2>;
    using I4 = std::integral_constant<int, 4>;
    using P = std::integral_constant<int, BC_PERIODIC>;
    using Rb = std::integral_constant<int, BC_ROBIN>;
    if (cfg->order == 2) {
        if (cfg->bc == MG_BC_PERIODIC) launch1(I2(), P()); else launch1(I2(), Rb());
    } else {
        if (cfg->bc == MG_BC_PERIODIC) launch1(I4(), P()); else launch1(I4(), Rb());
    }
    CK(attr);
    k_noalloc_norms<<<g1, kThreads, 0, st>>>(g, u, R, rho0, sc, partial);
    CK(cudaGetLastError());
    Scalars h;
    CK(cudaMemcpyAsync(&h, sc, sizeof(Scalars), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    for (int a = 0; a < 4; ++a) out[a] = h.norms[a];
    if (K2) *K2 = h.K2;
    return MG_OK;
}
