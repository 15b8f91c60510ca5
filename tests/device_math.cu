// Host entry of the device arithmetic of dfv_device.cuh, function by function,
// for test_gpu_device_math.py (built there with the library's own flags).
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
