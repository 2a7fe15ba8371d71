// k_sum4 on device arrays: means[a] of four contiguous fields of N values.
#include "mg_common.cuh"

template <typename T>
static int sum4(const T *x, long long N, double *partial, double *means, unsigned *ticket)
{
    const int per = 16 / (int)sizeof(T);
    ctt::k_sum4<T><<<ctt::grid_for((N + per - 1) / per, ctt::kSumBlocks), ctt::kThreads>>>(x, (size_t)N, partial, means, ticket);
    return (int)cudaDeviceSynchronize();
}
extern "C" int sum4_f32(const float *x, long long N, double *p, double *m, unsigned *t) { return sum4(x, N, p, m, t); }
extern "C" int sum4_f64(const double *x, long long N, double *p, double *m, unsigned *t) { return sum4(x, N, p, m, t); }
extern "C" int sum4_blocks() { return ctt::kSumBlocks; }
