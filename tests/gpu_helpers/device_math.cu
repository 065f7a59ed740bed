// Test helper: the library's own FP32 division and square root (lll_device.cuh)
// against FP64, and the root that draw_increment takes against the decision in
// FP64.  Built and loaded by tests/test_gpu_device_math.py only.
#include <cstdint>

#include <cuda_runtime.h>

#include "../../paper_1006_3340_gb300/csrc/lll_internal.h"
#include "../../paper_1006_3340_gb300/csrc/lll_device.cuh"

using namespace lll;

// Distance of y from the exact value `want` in spacings of FP32 at it.
__device__ double spacings(float y, double want)
{
    const double a = fabs(want);
    const double ulp = a < 1.1754943508222875e-38 ? 1.401298464324817e-45 : exp2(floor(log2(a)) - 23.0);
    return fabs((double)y - want) / ulp;
}

// what: 0 quotient(a, b), 1 square_root(a), 2 a / b, 3 sqrtf(a)
__global__ void math_kernel(int what, const float *a, const float *b, int count, double *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const double x = a[i], y = b[i];
    if (what == 0) err[i] = spacings(quotient(a[i], b[i]), x / y);
    else if (what == 1) err[i] = spacings(square_root(a[i]), sqrt(x));
    else if (what == 2) err[i] = spacings(a[i] / b[i], x / y);
    else err[i] = spacings(sqrtf(a[i]), sqrt(x));
}

// Draws of `count` paths at step k: how many increments are nearer to the root
// that the FP64 decision does not take, how many draws lie within `band` of the
// threshold (relative), and how many differ between the two forms of the draw.
__global__ void root_kernel(PathArgs a, uint32_t k, int count, double band, unsigned long long *wrong,
                            unsigned long long *near, unsigned long long *differ)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= count) return;
    const uint4 w = philox4x32_10(make_uint4(k, a.inst, (uint32_t)p, 0u), a.key0, a.key1);
    const double m = a.ig_md, l = a.ig_ld, u0 = u01d(w.x), u1 = u01d(w.y), u2 = u01d(w.z);
    const double r = sqrt(-2.0 * log(u0)), z1 = r * cospi(2.0 * u1), z2 = r * sinpi(2.0 * u1), nu = z1 * z1;
    const double large = m + m * m * nu / (2.0 * l) + m / (2.0 * l) * sqrt(4.0 * m * l * nu + m * m * nu * nu);
    const double small = m * m / large;
    const double t = u2 * (m + small);
    const bool take_small = u2 <= m / (m + small);
    auto increment = [&](double V) { return (double)a.nig_beta * V + sqrt(V) * z2 + (double)a.nig_muh; };
    const double right = increment(take_small ? small : large), other = increment(take_small ? large : small);
    const float out_of_line = draw_increment<false>(a, (uint64_t)p, k), in_line = draw_increment<true>(a, (uint64_t)p, k);
    const double got = out_of_line;
    if (fabs(t - m) < band * m) atomicAdd(near, 1ull);
    if (fabs(right - other) > 1e-4 * (fabs(right) + fabs(other)) && fabs(got - right) > fabs(got - other)) atomicAdd(wrong, 1ull);
    if (__float_as_uint(out_of_line) != __float_as_uint(in_line)) atomicAdd(differ, 1ull);
}

extern "C" int device_math(int what, const float *a, const float *b, int count, double *err)
{
    float *da = nullptr, *db = nullptr;
    double *de = nullptr;
    cudaError_t e = cudaMalloc((void **)&da, 4 * (size_t)count);
    if (e == cudaSuccess) e = cudaMalloc((void **)&db, 4 * (size_t)count);
    if (e == cudaSuccess) e = cudaMalloc((void **)&de, 8 * (size_t)count);
    if (e == cudaSuccess) e = cudaMemcpy(da, a, 4 * (size_t)count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(db, b, 4 * (size_t)count, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        math_kernel<<<(count + 127) / 128, 128>>>(what, da, db, count, de);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(err, de, 8 * (size_t)count, cudaMemcpyDeviceToHost);
    cudaFree(da);
    cudaFree(db);
    cudaFree(de);
    return (int)e;
}

// Increments of the normal inverse Gaussian driver (m, l: mean and shape of the
// mixing variable over a step).
extern "C" int device_roots(double m, double l, double beta, double muh, unsigned key, unsigned k, int count, double band,
                            unsigned long long *wrong, unsigned long long *near, unsigned long long *differ)
{
    PathArgs a{};
    a.driver = 0;
    a.key0 = key;
    a.ig_m = (float)m; a.ig_m2 = (float)(m * m); a.ig_hl = (float)(m / (2.0 * l));
    a.ig_fl = (float)(4.0 * m * l); a.ig_md = m; a.ig_ld = l;
    a.nig_beta = (float)beta; a.nig_muh = (float)muh;
    unsigned long long *d = nullptr, h[3] = {0, 0, 0};
    cudaError_t e = cudaMalloc((void **)&d, sizeof h);
    if (e == cudaSuccess) e = cudaMemset(d, 0, sizeof h);
    if (e == cudaSuccess) {
        root_kernel<<<(count + 127) / 128, 128>>>(a, k, count, band, d, d + 1, d + 2);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost);
    cudaFree(d);
    *wrong = h[0];
    *near = h[1];
    *differ = h[2];
    return (int)e;
}
