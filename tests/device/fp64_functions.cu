// The short FP64 functions of cph_device.cuh and cph_kernels.cuh against CUDA's, over
// their domains with the edges of their intervals.  Prints a line for each:
// name, largest absolute error, largest relative error (log64: the larger of |log x|
// and 2^-7 in place of |log x|).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include <cuda_runtime.h>

#include "cph_kernels.cuh"

using namespace cph;

#define OK(x)                                                                                          \
    do {                                                                                               \
        const cudaError_t e_ = (x);                                                                    \
        if (e_ != cudaSuccess) { std::printf("CUDA: %s\n", cudaGetErrorString(e_)); std::exit(1); }    \
    } while (0)

enum { kRcp, kRsqrt, kLog, kExp, kExpTab, kTanh, kSin, kCos, kFix, kFunctions };

__global__ void eval(int f, const double* x, double* mine, double* ref, int n) {
    __shared__ double2 tab[kTab64];
    load_tab64(tab, threadIdx.x, blockDim.x);
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    double a = 0.0, b = 0.0, s, c, s0, c0;
    switch (f) {
    case kRcp: a = rcp64(v); b = 1.0 / v; break;
    case kRsqrt: a = rsqrt64(v); b = rsqrt(v); break;
    case kLog: a = log64(v, tab); b = log(v); break;
    case kExp: a = exp64(v); b = exp(v); break;
    case kExpTab: a = exp64(v, tab); b = exp(v); break;
    case kTanh: a = tanh64(v); b = tanh(v); break;
    case kSin:
    case kCos: {
        const uint32_t w = (uint32_t)(long long)v;
        sincos64(w, s, c);
        sincospi(2.0 * unit_open(w), &s0, &c0);
        a = f == kSin ? s : c;
        b = f == kSin ? s0 : c0;
        break;
    }
    case kFix: a = (double)(fix32((float)v) - to_fixed((float)v, (float)kScaleE)); break;
    }
    mine[i] = a;
    ref[i] = b;
}

static std::mt19937_64 rng(11);
static double uni(double lo, double hi) { return lo + (hi - lo) * std::uniform_real_distribution<double>()(rng); }
static void around(std::vector<double>& v, double x) {
    v.push_back(x);
    v.push_back(std::nextafter(x, -INFINITY));
    v.push_back(std::nextafter(x, INFINITY));
}

static std::vector<double> points(int f) {
    std::vector<double> v;
    const int n = 400000;
    switch (f) {
    case kRcp:
    case kRsqrt:
        for (int k = 0; k < n; ++k) v.push_back(std::ldexp(uni(1.0, 2.0), (int)uni(-990, 990)));
        for (int k = 0; k < n; ++k) v.push_back(uni(1e-3, 100.0));
        for (int e = -990; e <= 990; ++e) around(v, std::ldexp(1.0, e));
        if (f == kRcp)
            for (size_t k = 0, m = v.size(); k < m; k += 2) v[k] = -v[k];
        break;
    case kLog:
        for (int k = 0; k < n; ++k) v.push_back(std::ldexp(uni(1.0, 2.0), (int)uni(-990, 990)));
        for (int k = 0; k < n; ++k) v.push_back(uni(1e-3, 4.0));
        for (int e = -3; e <= 3; ++e)
            for (int j = 0; j <= 128; ++j) // the table's intervals: eighths of 2^-4 from 0.6875 on, then of 2^-3
                around(v, std::ldexp(j < 80 ? 0.6875 + j / 256.0 : 1.0 + (j - 80) / 128.0, e));
        for (int e = 1; e <= 52; ++e) {
            v.push_back(1.0 - std::ldexp(1.0, -e));
            v.push_back(1.0 + std::ldexp(1.0, -e));
        }
        around(v, 1.0);
        break;
    case kExp:
    case kExpTab:
        for (int k = 0; k < n; ++k) v.push_back(-uni(0.0, 700.0));
        for (int k = 0; k < n; ++k) v.push_back(-std::exp2(uni(-60.0, 4.0)));
        for (int k = 0; k < 16159; ++k) around(v, -(k + 0.5) * std::log(2.0) / 16); // where the integer changes
        for (double x : {0.0, -0.0, -1e-300, -700.0}) v.push_back(x);
        for (double& x : v) x = std::fmin(x, 0.0);
        for (size_t k = 0; k < v.size(); ++k) v[k] = std::fmax(v[k], -700.0);
        break;
    case kTanh:
        for (int k = 0; k < n; ++k) v.push_back(uni(-25.0, 25.0));
        for (int k = 0; k < n; ++k) v.push_back((k & 1 ? -1 : 1) * std::exp2(uni(-60.0, 9.0)));
        for (double x : {0.0, 1e-300, 18.0, 19.0, 20.0, 349.9, 350.1, 1000.0, 1e300, (double)INFINITY}) {
            v.push_back(x);
            v.push_back(-x);
        }
        break;
    case kSin:
    case kCos:
        for (int k = 0; k < n; ++k) v.push_back(std::floor(uni(0.0, 4294967296.0)));
        for (int q = 0; q < 16; ++q) // quarter turns and the eighths between them
            for (int d = -3; d <= 3; ++d) v.push_back((double)(uint32_t)(q * 0x10000000u + (uint32_t)d));
        break;
    case kFix:
        for (int k = 0; k < n; ++k) v.push_back((float)((k & 1 ? -1 : 1) * std::exp2(uni(-40.0, 40.0))));
        for (int e = -40; e <= 31; ++e)
            for (double x : {1.0, 1.5, 1.0 + std::ldexp(1.0, -23)}) {
                v.push_back((float)std::ldexp(x, e));
                v.push_back(-(float)std::ldexp(x, e));
            }
        v.push_back(0.0);
        break;
    }
    return v;
}

int main() {
    const char* name[] = {"rcp64", "rsqrt64", "log64", "exp64", "exp64_tab", "tanh64", "sin64", "cos64", "fix32"};
    for (int f = 0; f < kFunctions; ++f) {
        const std::vector<double> x = points(f);
        const int n = (int)x.size();
        double *dx, *da, *db;
        OK(cudaMalloc(&dx, n * sizeof(double)));
        OK(cudaMalloc(&da, n * sizeof(double)));
        OK(cudaMalloc(&db, n * sizeof(double)));
        OK(cudaMemcpy(dx, x.data(), n * sizeof(double), cudaMemcpyHostToDevice));
        eval<<<(n + 255) / 256, 256>>>(f, dx, da, db, n);
        OK(cudaGetLastError());
        std::vector<double> a(n), b(n);
        OK(cudaMemcpy(a.data(), da, n * sizeof(double), cudaMemcpyDeviceToHost));
        OK(cudaMemcpy(b.data(), db, n * sizeof(double), cudaMemcpyDeviceToHost));
        double worst = 0.0, rel = 0.0;
        for (int i = 0; i < n; ++i) {
            const double d = std::fabs(a[i] - b[i]);
            const double size = f == kLog ? std::fmax(std::fabs(b[i]), 0.0078125) : std::fabs(b[i]);
            if (!(d <= worst)) worst = d; // (keeps a NaN)
            if (size > 0 && !(d / size <= rel)) rel = d / size;
        }
        std::printf("%s %.3e %.3e\n", name[f], worst, rel);
        OK(cudaFree(dx));
        OK(cudaFree(da));
        OK(cudaFree(db));
    }
}
