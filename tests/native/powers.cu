// The reciprocal and the negative powers of psi that the residual and the constraints use, and the powers of the
// correctly rounded 1/psi, on device arrays.
#include "mg_common.cuh"

static __global__ void k_recip(const double *x, double *y, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = ctt::recip_f64(x[i]);
}

// out: [psi^-5, psi^-6, psi^-7][n], then the same three from 1/psi
static __global__ void k_powers(const double *psi, double *out, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double p = psi[i], p2 = p * p, p5 = p2 * p2 * p, p6 = p5 * p;
        const ctt::PsiInverse v = ctt::psi_inverse(p, p5);
        out[i] = v.i5;
        out[n + i] = v.i6;
        out[2 * n + i] = ctt::recip_f64(p6 * p);
        const double q = 1.0 / p, q2 = q * q, q5 = q2 * q2 * q;
        out[3 * n + i] = q5;
        out[4 * n + i] = q5 * q;
        out[5 * n + i] = q2 * q2 * q2 * q;
    }
}

extern "C" int recip(const double *x, double *y, int n)
{
    k_recip<<<256, 256>>>(x, y, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int powers(const double *psi, double *out, int n)
{
    k_powers<<<256, 256>>>(psi, out, n);
    return (int)cudaDeviceSynchronize();
}
