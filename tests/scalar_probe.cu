// The device arithmetic of ugks_device.cuh and ugks_scalar.cuh on arrays, for
// test_gpu_scalar.py: out[i] of in[i], one element per thread.
#include "ugks_scalar.cuh"

using namespace ugks;

__global__ void k_exp_neg(const double *in, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = exp_neg(in[i]);
}

// in (dt, x), out q1..q5
__global__ void k_time_integrals(const double *in, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double q[5];
    time_integrals(in[2 * i], in[2 * i + 1], q);
    for (int j = 0; j < 5; ++j) out[5 * i + j] = q[j];
}

// in W (4 values in 2D, 5 in 3D), out U, T, lam and the Maxwellian's prefactor
template <int D> __global__ void k_prim(const double *in, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Prim p = prim_of(in + (size_t)i * (D + 2), D);
    double *o = out + (size_t)i * (D + 3);
    for (int d = 0; d < D; ++d) o[d] = p.U[d];
    o[D] = p.T;
    o[D + 1] = p.lam;
    o[D + 2] = pref_of(p.rho, p.lam, D);
}

using Kernel = void (*)(const double *, double *, int);

// host arrays in[n][nin], out[n][nout]; a CUDA error code
extern "C" int scalar_probe(int what, const double *in, int nin, double *out, int nout, int n)
{
    const Kernel kernels[] = {k_exp_neg, k_time_integrals, k_prim<2>, k_prim<3>};
    if (what < 0 || what >= (int)(sizeof(kernels) / sizeof(kernels[0])) || n <= 0) return (int)cudaErrorInvalidValue;
    double *di = nullptr, *dout = nullptr;
    cudaError_t e = cudaMalloc(&di, sizeof(double) * nin * (size_t)n);
    if (e == cudaSuccess) e = cudaMalloc(&dout, sizeof(double) * nout * (size_t)n);
    if (e == cudaSuccess) e = cudaMemcpy(di, in, sizeof(double) * nin * (size_t)n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        kernels[what]<<<(n + 127) / 128, 128>>>(di, dout, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, sizeof(double) * nout * (size_t)n, cudaMemcpyDeviceToHost);
    cudaFree(di);
    cudaFree(dout);
    return (int)e;
}
