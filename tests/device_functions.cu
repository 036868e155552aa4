// Device functions of the local solve, one element per thread, for tests/test_gpu_device_functions.py.
#include "local.cuh"

namespace {
__global__ void k_pow(long n, const double *__restrict__ x, const double *__restrict__ y, double *__restrict__ table,
                      double *__restrict__ cuda) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    table[i] = evp::pow_tab(x[i], y[i]);
    cuda[i] = pow(x[i], y[i]);
}

// sg: 6 x n stresses in the crystal frame; k32, k64: 21 x n tangents (packed lower)
__global__ void k_tangent(long n, const double *__restrict__ sg, evp::Cubic<double> cub, double tauc, evp::MatConst mc,
                          float *__restrict__ k32, double *__restrict__ k64) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    evp::Problem<double> pb;
    pb.cu = cub;
    pb.R = nullptr;   // the evaluation itself does not rotate
    const double etr[6] = {0, 0, 0, 0, 0, 0};
    double s[6];
    for (int c = 0; c < 6; ++c) s[c] = sg[c * n + i];
    evp::Eval<double, float> e32;
    evp::Eval<double> e64;
    evp::evaluate(pb, etr, tauc, 1.0 / tauc, s, mc, e32);
    evp::evaluate(pb, etr, tauc, 1.0 / tauc, s, mc, e64);
    for (int q = 0; q < 21; ++q) {
        k32[q * n + i] = e32.K[q];
        k64[q * n + i] = e64.K[q];
    }
}
}  // namespace

extern "C" int dev_pow(long n, const double *x, const double *y, double *table, double *cuda, void *stream) {
    k_pow<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(n, x, y, table, cuda);
    return (int)cudaGetLastError();
}
extern "C" int dev_tangent(long n, const double *sg, double d, double s12, double s44, double tauc, double gdot0,
                           double dt, double exponent, int n_int, float *k32, double *k64, void *stream) {
    evp::MatConst mc{};
    mc.gdot0 = gdot0;
    mc.n = exponent;
    mc.dt = dt;
    mc.n_int = n_int;
    k_tangent<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(n, sg, evp::Cubic<double>{d, s12, s44}, tauc,
                                                                             mc, k32, k64);
    return (int)cudaGetLastError();
}
