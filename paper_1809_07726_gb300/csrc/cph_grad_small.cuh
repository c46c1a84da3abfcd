// Differentiable GB energy of small replicas: one thread-block cluster each,
// the whole evaluation in one launch.
//
// For a replica of a few hundred atoms the symmetric kernels (cph_grad_sym.cuh)
// leave most of the chip idle and are a chain of eight to nine launches: 60 us
// for the energy of 1 x 237 atoms and 118 us for its gradient, against 12 and 25
// here.  Here a cluster of eight CTAs holds the
// replica in shared memory; every ordered pair (i, j) is evaluated by a warp of
// i's CTA, and the passes are phases between cluster barriers, as in
// cph_small.cuh (radii and chain weights go to every CTA).  Sums over partners
// are FP32 over a lane's at most 16 partners, then int64 fixed point, so results
// do not depend on launch order.  Twice the pair arithmetic of the symmetric
// form: the rule gsmall in cph_grad.cu says up to where that pays.
#pragma once
#include <cooperative_groups.h>

#include "cph_device.cuh"
#include "cph_grad_sym.cuh"

namespace cph {
namespace grad {

constexpr int kGsRanks = 8;   // CTAs per cluster
constexpr int kGsAtoms = 512; // atoms of a replica at most
constexpr int kGsThreads = 512;

template <bool BACKWARD>
__global__ void __launch_bounds__(kGsThreads) __cluster_dims__(kGsRanks, 1, 1) k_gsmall(SView g) {
    namespace cg = cooperative_groups;
    constexpr int own_max = kGsAtoms / kGsRanks;
    __shared__ float4 xq[kGsAtoms];  // (x, y, z, sqrt(k) q)
    __shared__ float4 st[kGsAtoms];  // (s, rt, 1/rt, c)
    __shared__ float2 rad[kGsAtoms]; // (R, 1/R)
    __shared__ long long sum[own_max][6];
    __shared__ double aR[own_max], aiR[own_max], apsi[own_max], adR[own_max], adq[own_max], aE[own_max], ag[own_max];
    __shared__ long long er[kGsRanks]; // energy sums of the CTAs (rank 0's copy)
    __shared__ long long ew[kGsThreads / 32];
    cg::cluster_group cl = cg::this_cluster();
    auto sync = [&] {
        __syncwarp();
        cl.sync();
    };
    const int rank = (int)cl.block_rank(), rep = (int)blockIdx.x / kGsRanks, n = g.n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int own = (n + kGsRanks - 1) / kGsRanks, a0 = rank * own, nown = min(own, max(0, n - a0));
    const size_t base = (size_t)rep * n;
    const float off = g.off32, sqk = g.sqk32, rc = g.rgbmax32;
    for (int j = tid; j < n; j += kGsThreads) {
        const float* X = g.x + 3 * (base + j);
        xq[j] = make_float4(X[0], X[1], X[2], g.q[base + j] * sqk);
        const float rt = g.rho[base + j] - off;
        st[j] = make_float4(g.screen[j] * rt, rt, 1.f / rt, 0.f);
    }
    sync(); // the operands; and every CTA of the cluster runs, so that others may store into its memory
    // ---- Born radii
    for (int a = warp; a < nown; a += kGsThreads / 32) {
        const int i = a0 + a;
        const float4 xi = xq[i], si = st[i];
        float part = 0.f;
        for (int j = lane; j < n; j += 32) {
            const float4 xj = xq[j];
            const float dx = xi.x - xj.x, dy = xi.y - xj.y, dz = xi.z - xj.z;
            const float r2 = j == i ? 1.f : fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const float rinv = rsqrt_ftz(r2);
            const float h = hct(r2 * rinv, rinv, si.y, si.z, st[j].x, rc);
            part += j == i ? 0.f : h;
        }
        const long long H = warp_sum(fix32(part * 256.f)); // 2^40
        if (lane == 0) sum[a][0] = H;
    }
    __syncthreads();
    for (int a = tid; a < nown; a += kGsThreads) {
        const double rho = g.rho[base + a0 + a], rt = rho - g.offset, irho = rcp64(rho);
        const double psi = rt * ((double)sum[a][0] * (0.5 / kScaleH));
        const double th = tanh64(psi * (g.alpha + psi * (-g.beta + psi * g.gamma)));
        const double iR = rcp64(rt) - th * irho, R = rcp64_radius(iR);
        aR[a] = R;
        aiR[a] = iR;
        apsi[a] = psi;
        adR[a] = R * R * (1.0 - th * th) * (g.alpha + psi * (-2.0 * g.beta + 3.0 * g.gamma * psi)) * irho;
        const float2 o = make_float2(pair_radius32(R), (float)iR);
#pragma unroll
        for (int r = 0; r < kGsRanks; ++r) cl.map_shared_rank(rad, r)[a0 + a] = o;
    }
    sync();
    // ---- GB pair sums
    for (int a = warp; a < nown; a += kGsThreads / 32) {
        const int i = a0 + a;
        const float4 xi = xq[i];
        const float2 Ri = rad[i];
        const float dk = (0.25f * kLog2e) * Ri.y;
        KSum<float> eg;
        float dr = 0.f, dq = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
        auto sweep = [&](auto with_salt) {
            constexpr bool SALT = decltype(with_salt)::value;
            for (int j = lane; j < n; j += 32) {
                const float4 xj = xq[j];
                const float2 Rj = rad[j];
                const float dx = xi.x - xj.x, dy = xi.y - xj.y, dz = xi.z - xj.z;
                const float r2 = j == i ? 1.f : fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                const float D2 = r2 * (dk * Rj.y), e = exp2_ftz(-D2); // D log2(e)
                const float fa = fmaf(Ri.x * Rj.x, e, r2);
                const float fi = j == i ? 0.f : rsqrt_ftz(fa);
                const float qq = xi.w * xj.w;
                float tf = 1.f, td = 1.f;
                if (SALT) {
                    const float f = fa * fi, es = g.ieo32 * exp2_ftz(-g.kap32 * kLog2e * f);
                    tf = g.iei32 - es;
                    td = tf - g.kap32 * f * es;
                }
                const float fit = SALT ? fi * tf : fi;
                eg.add(qq * fit);
                if (BACKWARD) {
                    const float qf3 = qq * (fi * fi * fi), qfe = qf3 * e;
                    float t = qfe * fmaf(D2, kLn2, 1.f);
                    if (SALT) t *= td;
                    dr = fmaf(t, Rj.x, dr);
                    dq = fmaf(xj.w, fit, dq);
                    const float g2 = (SALT ? td : g.tau32) * fmaf(-0.25f, qfe, qf3);
                    gx = fmaf(g2, dx, gx);
                    gy = fmaf(g2, dy, gy);
                    gz = fmaf(g2, dz, gz);
                }
            }
        };
        if (g.kappa > 0) sweep(std::true_type{});
        else sweep(std::false_type{});
        long long v[6] = {fix32(eg.value()), fix32(dr), fix32(dq), fix32(gx), fix32(gy), fix32(gz)};
#pragma unroll
        for (int k = 0; k < (BACKWARD ? 6 : 1); ++k) {
            v[k] = warp_sum(v[k]);
            if (lane == 0) sum[a][k] = v[k];
        }
    }
    __syncthreads();
    // ---- self terms, energy; chain weights to every CTA
    long long ea = 0;
    for (int a = tid; a < nown; a += kGsThreads) {
        const int i = a0 + a;
        const double q = (double)g.q[base + i] * g.sqrt_k, R = aR[a], iR = aiR[a], rho = g.rho[base + i];
        const double esa = sa_ace(g.sa_gamma, g.sa_probe, rho, R);
        const double ts = salt_tau(R, g.inv_eps_in, g.inv_eps_out, g.kappa);
        ea += __double2ll_rn((-0.5 * (g.tau_pair * ((double)sum[a][0] * (1.0 / kScaleE)) + ts * q * q * iR) + esa) * kScaleE);
        if (BACKWARD) {
            const double dEdR = 0.5 * (g.tau_pair * ((double)sum[a][1] * (1.0 / kScaleE)) +
                                       salt_taud(R, g.inv_eps_in, g.inv_eps_out, g.kappa) * q * q * iR * iR) -
                                (g.sa_gamma != 0.0 ? 6.0 * esa * iR : 0.0);
            const double gpsi = dEdR * adR[a];
            adq[a] = -g.sqrt_k * (g.tau_pair * ((double)sum[a][2] * (1.0 / kScaleE)) + ts * q * iR);
            aE[a] = dEdR;
            ag[a] = gpsi;
            const float c = (float)(gpsi * 0.5 * (rho - g.offset));
#pragma unroll
            for (int r = 0; r < kGsRanks; ++r) cl.map_shared_rank(st, r)[i].w = c;
        }
    }
    if (!BACKWARD) {
        ea = warp_sum(ea);
        if (lane == 0) ew[warp] = ea;
        __syncthreads();
        if (tid == 0) {
            long long t = 0;
            for (int k = 0; k < kGsThreads / 32; ++k) t += ew[k];
            cl.map_shared_rank(er, 0)[rank] = t;
        }
        sync();
        if (rank == 0 && tid == 0) {
            long long t = 0;
            for (int r = 0; r < kGsRanks; ++r) t += er[r];
            g.E[rep] = (double)t / kScaleE;
        }
        return;
    }
    sync();
    // ---- chain rule through the radii, and the rho derivatives of the integrals
    for (int a = warp; a < nown; a += kGsThreads / 32) {
        const int i = a0 + a;
        const float4 xi = xq[i], si = st[i];
        float gx = 0.f, gy = 0.f, gz = 0.f, art = 0.f, as = 0.f;
        for (int j = lane; j < n; j += 32) {
            if (j == i) continue;
            const float4 xj = xq[j], sj = st[j];
            const float dx = xi.x - xj.x, dy = xi.y - xj.y, dz = xi.z - xj.z;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const float rinv = rsqrt_ftz(r2), r = r2 * rinv;
            const float t = (si.w * hct_dr_fastlog(r, rinv, si.y, sj.x, rc) + sj.w * hct_dr_fastlog(r, rinv, sj.y, si.x, rc)) * rinv;
            gx = fmaf(t, dx, gx);
            gy = fmaf(t, dy, gy);
            gz = fmaf(t, dz, gz);
            art += hct_drt(r, si.y, si.z, sj.x, rc);
            as = fmaf(sj.w, hct_ds(r, rinv, sj.y, si.x, rc), as);
        }
        long long v[5] = {fix32(gx), fix32(gy), fix32(gz), fix32(art), fix32(as)};
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            v[k] = warp_sum(v[k]);
            // the pair gradient of the pass before is in sum[a][3..5]
            if (lane == 0) sum[a][k < 3 ? 3 + k : k - 3] = k < 3 ? sum[a][3 + k] + v[k] : v[k];
        }
    }
    __syncthreads();
    const double up = g.dE[rep];
    for (int a = tid; a < nown; a += kGsThreads) {
        const size_t k = base + a0 + a;
        const double rho = g.rho[k], rt = rho - g.offset, irt = rcp64(rt), R = aR[a], psi = apsi[a];
        const double th = (irt - aiR[a]) * rho; // 1/R = 1/rt - th / rho
        const double irho = rcp64(rho), esa = sa_ace(g.sa_gamma, g.sa_probe, rho, R);
        const double dr = aE[a] * R * R * (irt * irt - th * irho * irho) + ag[a] * psi * irt +
                          (ag[a] * 0.5 * rt) * ((double)sum[a][0] * (1.0 / kScaleE)) +
                          (double)g.screen[a0 + a] * ((double)sum[a][1] * (1.0 / kScaleE)) +
                          (esa != 0.0 ? esa * (2.0 / (rho + g.sa_probe) + 6.0 * irho) : 0.0);
        for (int c = 0; c < 3; ++c) g.dx[3 * k + c] = (float)(up * ((double)sum[a][3 + c] * (1.0 / kScaleE)));
        g.dqo[k] = (float)(up * adq[a]);
        g.drho[k] = (float)(up * dr);
    }
}

} // namespace grad
} // namespace cph
