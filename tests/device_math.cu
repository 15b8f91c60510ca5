// Host entry of the device arithmetic of dfv_device.cuh, function by function,
// for test_gpu_device_math.py (built there with the library's own flags).
#include <cstring>

#include <cuda_runtime.h>

#include "dfv_device.cuh"

using namespace dfv;

namespace {

enum { RCP, DIV, QUOT, SQRT, SQRT_RATIO, ARTANH, COSH, SINHC, EXPM1, WIDEN, NARROW, MIN, MAX, PRED, LESS, POWER };

__global__ void k_eval(int id, const double *a, const double *b, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = a[i], y = b[i];
    double r = 0.0, s = 0.0;
    switch (id) {
    case RCP: r = m_rcp(x); break;
    case DIV: r = m_div(x, y); break;
    case QUOT: r = m_quot(x, y); break;
    case SQRT: r = m_sqrt(x); break;
    case SQRT_RATIO: r = m_sqrt_ratio(x, y); break;
    case ARTANH: r = artanh_ratio(x); break;
    case COSH: coshm1_sinhc(x, r, s); r += 1.0; break;
    case SINHC: coshm1_sinhc(x, s, r); break;
    case EXPM1: r = expm1_near0(x); break;
    case WIDEN: r = m_widen(__uint_as_float((unsigned)__double_as_longlong(x))); break;
    case NARROW: r = __longlong_as_double((long long)__float_as_uint(m_narrow(x))); break;
    case MIN: r = m_min(x, y); break;
    case MAX: r = m_max(x, y); break;
    case PRED: r = m_pos(x) + 2 * m_neg(x) + 4 * m_ge0(x) + 8 * m_zero(x) + 16 * m_over1(x); break;
    case LESS: r = m_less(x, y); break;
    default: r = m_whole_pow(x, (int)y); break;
    }
    out[i] = r;
}

// the end of a step for a solid's cell at rest, FP32 with a strain plane: A in
// and out, rho times the strain that the return adds
__global__ void k_finish(GridP g, float *A, float *strain, int n)
{
    using L = Lay<2, 1, 2>;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float o[L::NVAR], c;
    for (int v = 0; v < L::NVAR; v++) o[v] = 0.f;
    o[L::IAR] = (float)g.mat[0].rho0;
    o[L::IE] = 1e5f;
    for (int k = 0; k < L::NV; k++) o[L::IV + k] = A[(size_t)k * n + i];
    solid_finish<float, 2, 1, 2>(g, 1e-9, o, c);
    for (int k = 0; k < L::NV; k++) A[(size_t)k * n + i] = o[L::IV + k];
    strain[i] = o[L::IH];
}

}  // namespace

extern "C" int dm_eval(int id, const double *a, const double *b, double *out, int n)
{
    double *d = nullptr;
    const size_t bytes = sizeof(double) * (size_t)n;
    cudaError_t e = cudaMalloc(&d, 3 * bytes);
    if (e == cudaSuccess) e = cudaMemcpy(d, a, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + n, b, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_eval<<<(n + 255) / 256, 256>>>(id, d, d + n, d + 2 * (size_t)n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, d + 2 * (size_t)n, bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}

extern "C" int dm_finish(double rho0, double K0, double G0, double sigY, float *A, float *strain, int n)
{
    GridP g;
    memset(&g, 0, sizeof(g));
    g.dim = 2;
    for (int d = 0; d < 3; d++) g.dx[d] = g.inv_dx[d] = 1.0;
    g.mat[0].kind = 2;
    g.mat[0].rho0 = rho0;
    g.mat[0].K0 = K0;
    g.mat[0].G0 = G0;
    g.mat[0].alpha = g.mat[0].beta = 1.0;
    g.mat[0].Gamma0 = 2.0;
    g.mat[0].sigY = sigY;
    apply_options(g, 1, 1.6, 0, 0, 0, 0);
    finish_params(g);
    float *d = nullptr;
    const size_t bytes = sizeof(float) * (size_t)n;
    cudaError_t e = cudaMalloc(&d, 6 * bytes);
    if (e == cudaSuccess) e = cudaMemcpy(d, A, 5 * bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_finish<<<(n + 255) / 256, 256>>>(g, d, d + 5 * (size_t)n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(A, d, 5 * bytes, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(strain, d + 5 * (size_t)n, bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
