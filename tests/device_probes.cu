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
}
