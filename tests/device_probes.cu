// Device functions of the library under test, element by element over arrays, for the tests.
#include "elbm_device.cuh"

namespace {

__global__ void k_div(const double *a, const double *b, double *out, double *ieee, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = eelbm::div_(a[k], b[k]), ieee[k] = __ddiv_rn(a[k], b[k]);
}
__global__ void k_sqrt(const double *a, double *out, double *ieee, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = eelbm::sqrt_(a[k]), ieee[k] = __dsqrt_rn(a[k]);
}
// out: S3..S6 of a thread's q populations (f, x: q rows of n), both lanes summed as by a node
__global__ void k_power_sums(const float *f, const float *x, float *out, int n, int q)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    eelbm::PowerSums s;
    for (int i = 0; i < q; i += 2) {
        const bool pad = i + 1 == q;
        s.add(make_float2(f[i * n + k], pad ? 1.0f : f[(i + 1) * n + k]), make_float2(x[i * n + k], pad ? 0.0f : x[(i + 1) * n + k]));
    }
    const float2 v[4] = {s.S3, s.S4, s.S5, s.S6};
    for (int j = 0; j < 4; ++j) out[j * n + k] = v[j].x + v[j].y;
}
int finish()
{
    const cudaError_t e = cudaGetLastError();
    return int(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
unsigned blocks(int n) { return unsigned((n + 127) / 128); }

} // namespace

extern "C" {
int probe_div(const double *a, const double *b, double *out, double *ieee, int n)
{
    k_div<<<blocks(n), 128>>>(a, b, out, ieee, n);
    return finish();
}
int probe_sqrt(const double *a, double *out, double *ieee, int n)
{
    k_sqrt<<<blocks(n), 128>>>(a, out, ieee, n);
    return finish();
}
int probe_power_sums(const float *f, const float *x, float *out, int n, int q)
{
    k_power_sums<<<blocks(n), 128>>>(f, x, out, n, q);
    return finish();
}
}
