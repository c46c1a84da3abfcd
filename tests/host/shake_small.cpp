// Host build of csrc/cph_shake_small.cuh: a cluster's four lanes are four threads,
// a warp exchange is a pass over a barrier.
//   sums N      N random sums over the lanes; prints how many differ between lanes
//   shake N T   N random clusters of 1 to 3 hydrogens after a step, tolerance T:
//               prints unsettled clusters, lanes that disagree on the end, the
//               largest |d^2 / d0^2 - 1| of the settled ones, and the largest
//               displacement off the old bond vectors (A)
#include <atomic>
#include <barrier>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <thread>
#include <vector>

#define __device__
#define __forceinline__ inline
#define __noinline__
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
static float2 make_float2(float x, float y) { return {x, y}; }
static float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fdividef(float a, float b) { return a / b; }

static std::barrier<> gate(4);
static thread_local int lane;
static double slot[4];
static float __shfl_xor_sync(unsigned, float v, int o) {
    slot[lane] = v;
    gate.arrive_and_wait();
    const float r = (float)slot[lane ^ o];
    gate.arrive_and_wait();
    return r;
}
static double __shfl_xor_sync(unsigned, double v, int o) {
    slot[lane] = v;
    gate.arrive_and_wait();
    const double r = slot[lane ^ o];
    gate.arrive_and_wait();
    return r;
}
static bool __all_sync(unsigned, bool p) {
    slot[lane] = p;
    gate.arrive_and_wait();
    const bool r = slot[0] && slot[1] && slot[2] && slot[3];
    gate.arrive_and_wait();
    return r;
}
static std::atomic<int> flags{0};
static void atomicOr(int*, int v) { flags |= v; }

namespace cph {
constexpr int kShakeMaxIter = 1000;
struct View {
    const int *shk_off, *shk_heavy, *shk_h;
    const double* shk_d;
    double shake_tol;
    int* status;
};
} // namespace cph
#include "cph_shake_small.cuh"
using namespace cph;

int main(int argc, char** argv) {
    const bool sums = std::string(argv[1]) == "sums";
    const int n = std::atoi(argv[2]);
    const double tol = argc > 3 ? std::atof(argv[3]) : 0.0;
    std::mt19937_64 rng(7);
    std::normal_distribution<double> g;
    std::uniform_real_distribution<double> uni;
    int differ = 0, unsettled = 0;
    double worst = 0.0, off = 0.0;
    for (int k = 0; k < n; ++k) {
        if (sums) {
            float h[4], l[4], oh[4], ol[4];
            for (int d = 0; d < 4; ++d) {
                const double v = g(rng);
                h[d] = (float)v;
                l[d] = (float)(v - h[d]);
            }
            std::vector<std::thread> t;
            for (int d = 0; d < 4; ++d)
                t.emplace_back([&, d] {
                    lane = d;
                    oh[d] = h[d];
                    ol[d] = l[d];
                    sum4(oh[d], ol[d]);
                });
            for (auto& x : t) x.join();
            for (int d = 1; d < 4; ++d)
                if (std::memcmp(&oh[d], &oh[0], 4) || std::memcmp(&ol[d], &ol[0], 4)) {
                    ++differ;
                    break;
                }
            continue;
        }
        // a heavy atom and its hydrogens, a step of thermal size past a constrained geometry
        const int nh = 1 + k % 3;
        const double m[4] = {12.011, 1.008, 1.008, 1.008}, d0 = 1.09;
        double xo[12], xt[12], dist[3];
        float4 fac[3];
        for (int d = 0; d < 3; ++d) xo[d] = 20.0 * g(rng);
        for (int h = 0; h < nh; ++h) {
            double v[3], r = 0.0;
            for (int d = 0; d < 3; ++d) r += (v[d] = g(rng)) * v[d];
            for (int d = 0; d < 3; ++d) xo[3 + 3 * h + d] = xo[d] + d0 * v[d] / std::sqrt(r);
            dist[h] = d0;
            const double i0 = 1 / m[0], ih = 1 / m[1], f0 = 0.5 * i0 / (i0 + ih), fh = 0.5 * ih / (i0 + ih);
            fac[h] = {(float)f0, (float)(f0 - (float)f0), (float)fh, (float)(fh - (float)fh)};
        }
        for (int a = 0; a <= nh; ++a)
            for (int d = 0; d < 3; ++d) xt[3 * a + d] = xo[3 * a + d] + 0.03 / std::sqrt(m[a]) * g(rng);
        const int off_tab[2] = {0, nh}, heavy = 0, hyd[3] = {1, 2, 3};
        const View V{off_tab, &heavy, hyd, dist, tol, nullptr};
        flags = 0;
        double u[4][4] = {};
        std::vector<std::thread> t;
        for (int d = 0; d < 4; ++d)
            t.emplace_back([&, d] {
                lane = d;
                small_shake<3>(V, fac, 0, true, d, xo, xt, nh, u[d]);
            });
        for (auto& x : t) x.join();
        if (flags) {
            ++unsettled;
            continue;
        }
        for (int h = 0; h < nh; ++h) {
            double r2 = 0.0, cr = 0.0, b[3], w[3];
            for (int d = 0; d < 3; ++d) {
                const double r = (xt[d] + u[d][0]) - (xt[3 + 3 * h + d] + u[d][h + 1]);
                r2 += r * r;
                b[d] = xo[d] - xo[3 + 3 * h + d];
                w[d] = u[d][h + 1]; // a hydrogen moves along its old bond vector
            }
            for (int d = 0; d < 3; ++d) {
                const int e = (d + 1) % 3;
                cr = std::fmax(cr, std::fabs(w[d] * b[e] - w[e] * b[d]) / d0);
            }
            off = std::fmax(off, cr);
            worst = std::fmax(worst, std::fabs(r2 / (d0 * d0) - 1.0));
        }
    }
    if (sums) std::printf("%d\n", differ);
    else std::printf("%d %.3e %.3e\n", unsettled, worst, off);
}
