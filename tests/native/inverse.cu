// k_invert_registers on the left block of an augmented matrix (row stride 2m), by its register tile R.
#include "mg_common.cuh"

template <typename T>
static int invert(const T *aug, int m, T *inv)
{
    if (m <= 32) ctt::k_invert_registers<T, 1><<<1, 256>>>(aug, m, inv);
    else if (m <= 64) ctt::k_invert_registers<T, 2><<<1, 256>>>(aug, m, inv);
    else if (m <= 96) ctt::k_invert_registers<T, 3><<<1, 256>>>(aug, m, inv);
    else ctt::k_invert_registers<T, 5><<<1, 256>>>(aug, m, inv);
    return (int)cudaDeviceSynchronize();
}
extern "C" int invert_f32(const float *a, int m, float *i) { return invert(a, m, i); }
extern "C" int invert_f64(const double *a, int m, double *i) { return invert(a, m, i); }
