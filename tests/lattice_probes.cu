// Device functions of one lattice's kernels, element by element over arrays, for the tests
// (built with ELBM_DIM 2 or 3).
#define ELBM_SUFFIX probed
#define ELBM_PART 0 // no launchers
#include "elbm_kernels.cuh"

namespace {

using namespace eelbm;

__global__ void k_rcp64(const double *rho, double *out, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = probed::rcp64(rho[k]);
}
// v: Q rows of n stored values; out: rho, then D rows of rho u (1 + D rows)
template <bool kDev>
__global__ void k_exact_sums(const float *v, double *out, int n, float R)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    float f[probed::Q];
    double rho = 0.0, j[3] = {0.0, 0.0, 0.0};
    for (int i = 0; i < probed::Q; ++i) f[i] = v[i * n + k];
    if (!probed::exact_sums<kDev>(f, R, (probed::Q == 9 ? 36.0 : 216.0) * double(R), rho, j)) rho = j[0] = j[1] = j[2] = -1.0;
    out[k] = rho;
    for (int a = 0; a < probed::D; ++a) out[(1 + a) * n + k] = j[a];
}
int finish()
{
    const cudaError_t e = cudaGetLastError();
    return int(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
unsigned blocks(int n) { return unsigned((n + 127) / 128); }

} // namespace

extern "C" {
int probe_rcp64(const double *rho, double *out, int n)
{
    k_rcp64<<<blocks(n), 128>>>(rho, out, n);
    return finish();
}
int probe_exact_sums(const float *v, double *out, int n, float R)
{
    if (R == 0.0f) k_exact_sums<false><<<blocks(n), 128>>>(v, out, n, R);
    else k_exact_sums<true><<<blocks(n), 128>>>(v, out, n, R);
    return finish();
}
}
