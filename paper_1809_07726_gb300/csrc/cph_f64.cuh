// The ordered pair passes in FP64 (the decomposition of cph_kernels.cuh: every
// ordered pair, one warp or four per atom i, tiles of 128 partners).
//
// GB300 issues an FP64 warp instruction every 64 clocks per sub-partition, so a
// pass costs its FP64 instructions and nothing else: 152 x 4 sub-partitions, a
// 160-atom walker's 25,600 ordered pairs are 800 warp evaluations on 608 of
// them.  Per pair, before and now (FP64 instructions): Born radii ~85 -> 41, GB +
// Coulomb + LJ ~100 -> 63, chain rule ~145 -> 76, by third-order reciprocals and
// reciprocal square roots from the approximate ones, one reciprocal for 1/L and
// 1/U, a table logarithm and exponential, coordinates subtracted once, selects
// in place of factors 0 and 1.  Warps whose partners are all padding skip them,
// and the warp that takes a tile's remainder differs from CTA to CTA, so that two
// CTAs on one SM do not load the same sub-partition.  Sums over a warp exchange
// halves (K values in K + 4 - log2 K additions or so, not 5 K).
#pragma once
#include "cph_device.cuh"
#include "cph_internal.h"
#include "cph_kernels.cuh"

namespace cph {

// Sums of K = 4 or 8 values over the warp; lane l returns that of value l / (32 / K).
template <int K>
__device__ __forceinline__ double warp_sums(double (&v)[K]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = K / 2, o = 16; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double keep = up ? v[k + n] : v[k], send = up ? v[k] : v[k + n];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 16 / K; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// ... over the WPA warps of an atom; value k is then in out[k] for the group's
// first warp (WPA = 4: every thread of the CTA calls it; red: [4][K]).
template <int WPA, int K>
__device__ __forceinline__ void group_sums(double (&v)[K], double* red, double (&out)[K]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double t = warp_sums<K>(v);
    if (WPA == 4) {
        constexpr int seg = 32 / K;
        if (lane % seg == 0) red[warp * K + lane / seg] = t;
        __syncthreads();
        if (warp == 0) {
            const int k = lane / seg;
            t = (red[k] + red[K + k]) + (red[2 * K + k] + red[3 * K + k]);
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = __shfl_sync(0xffffffffu, t, k * (32 / K));
}

// The thread's place in its atom's group: entries k of a tile with k % (32 WPA) = sub.
template <int WPA>
__device__ __forceinline__ int place64() {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    return WPA == 1 ? lane : ((warp + (int)blockIdx.x) & 3) * 32 + lane;
}

template <int WPA>
__global__ void __launch_bounds__(kTile) k_born64(const Item* __restrict__ items, View V, int zero_energy) {
    pdl_sync();
    __shared__ J4<double> sj[kTile];
    __shared__ double2 tab[kTab64];
    __shared__ double red[16];
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = place64<WPA>();
    const int i = it.i0 + warp / WPA;
    const bool vi = i < N;
    load_tab64(tab, tid, kTile);
    if (it.i0 == 0) {
        if (zero_energy && tid < kEAcc) V.eacc[w * kEAcc + tid] = 0;
        if (tid == kEAcc) V.vscale[w] = 1.0;
    }
    const int ic = vi ? i : it.i0;
    const double xi = V.x[3 * (A + ic)], yi = V.x[3 * (A + ic) + 1], zi = V.x[3 * (A + ic) + 2];
    const double rti = V.rt[P + ic], irti = V.irt[P + ic], rc = V.rgbmax;
    double acc = 0.0;
    for (int j0 = 0; j0 < N; j0 += kTile) {
        __syncthreads();
        if (j0 + tid < N) {
            const int j = j0 + tid;
            sj[tid] = {V.x[3 * (A + j)], V.x[3 * (A + j) + 1], V.x[3 * (A + j) + 2], V.sc[P + j]};
        }
        __syncthreads();
#pragma unroll 1
        for (int k = sub; k < kTile; k += 32 * WPA) {
            if (j0 + (k & ~31) >= N) break; // no partner in this warp's entries, nor in later ones
            const bool self = j0 + k == i || j0 + k >= N;
            const J4<double> b = sj[min(k, N - 1 - j0)];
            const double dx = xi - b.x, dy = yi - b.y, dz = zi - b.z;
            double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            r2 = self ? 1.0 : r2;
            const double rinv = rsqrt64(r2);
            const double h = hct64(r2 * rinv, r2, rinv, rti, irti, b.w, rc, tab);
            acc += self ? 0.0 : h;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (WPA == 4) {
        if (lane == 0) red[warp] = acc;
        __syncthreads();
        acc = (red[0] + red[1]) + (red[2] + red[3]);
    }
    if (vi && lane == 0 && (WPA == 1 || warp == 0)) {
        const double irho = V.irho[P + i], psi = 0.5 * rti * acc;
        const double th0 = psi * (V.alpha + psi * (-V.beta + psi * V.gamma));
        const double e = exp64(-2.0 * fabs(th0), tab); // tanh = (1 - e) / (1 + e)
        const double th = copysign(fma(-2.0 * e, rcp64(1.0 + e), 1.0), th0);
        const double R = rcp64_radius(irti - th * irho);
        V.psi[A + i] = psi;
        V.R[A + i] = R;
        V.dRdpsi[A + i] = R * R * (1.0 - th * th) * (V.alpha + psi * (-2.0 * V.beta + 3.0 * V.gamma * psi)) * irho;
    }
}

template <bool ENERGY, int WPA>
__global__ void __launch_bounds__(kTile) k_gb64(const Item* __restrict__ items, View V) {
    pdl_sync();
    constexpr int K = ENERGY ? 8 : 4;
    __shared__ J4<double> sa[kTile], sb[kTile];
    __shared__ double2 tab[kTab64];
    __shared__ double red[4 * K];
    __shared__ long long redl[4];
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = place64<WPA>();
    const int i = it.i0 + warp / WPA;
    const bool vi = i < N;
    load_tab64(tab, tid, kTile);
    const int ic = vi ? i : it.i0;
    const double xi = V.x[3 * (A + ic)], yi = V.x[3 * (A + ic) + 1], zi = V.x[3 * (A + ic) + 2];
    const double Ri = pair_radius64(V.R[A + ic]), iRi = rcp64(Ri), mq = -0.25 * iRi;
    const double qi = V.q[A + ic] * V.sqrt_k, sgi = V.sigh[P + ic], sei = V.sqe[P + ic];
    const double tau = V.tau, iei = V.inv_eps_in, kap = V.kappa, ieo = V.inv_eps_out;
    double fx = 0, fy = 0, fz = 0, adr = 0, egb = 0, ec = 0, elj = 0;
    int mp = V.mt_off[it.st];
    const int me = V.mt_off[it.st + 1];
    auto sweep = [&](auto with_salt) {
        constexpr bool SALT = decltype(with_salt)::value;
        int next = mp < me ? V.mt_list[mp] : 0x7fffffff;
        for (int j0 = 0, jt = 0; j0 < N; j0 += kTile, ++jt) {
            __syncthreads();
            if (j0 + tid < N) {
                const int j = j0 + tid;
                const double R = pair_radius64(V.R[A + j]);
                sa[tid] = {V.x[3 * (A + j)], V.x[3 * (A + j) + 1], V.x[3 * (A + j) + 2], V.q[A + j] * V.sqrt_k};
                sb[tid] = {R, rcp64(R), V.sigh[P + j], V.sqe[P + j]};
            }
            __syncthreads();
            uint32_t mex[4] = {0u, 0u, 0u, 0u}, mself[4];
            if (jt == next) {
                ++mp;
                next = mp < me ? V.mt_list[mp] : 0x7fffffff;
                tile_masks(V, P, i, vi, j0, mex, mself);
            }
#pragma unroll 1
            for (int k = sub; k < kTile; k += 32 * WPA) {
                if (j0 + (k & ~31) >= N) break;
                const int q4 = k >> 5;
                const bool self = j0 + k == i || j0 + k >= N;
                const uint32_t m = q4 == 0 ? mex[0] : (q4 == 1 ? mex[1] : (q4 == 2 ? mex[2] : mex[3]));
                const bool ex = self || ((m >> (k & 31)) & 1u);
                const int kc = min(k, N - 1 - j0);
                const J4<double> a = sa[kc], b = sb[kc];
                const double dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
                double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                r2 = self ? 1.0 : r2;
                const double rinv = rsqrt64(r2), rinv2 = rinv * rinv;
                const double q0 = qi * a.w, qq = self ? 0.0 : q0;
                const double mD = r2 * (mq * b.y), e = exp64(mD, tab); // -D
                const double fi = rsqrt64(fma(Ri * b.x, e, r2));
                const double qf3 = qq * fi * (fi * fi), qfe = qf3 * e;
                double tf = 1.0, td = 1.0;
                if (SALT) {
                    const double f = rcp64(fi), es = ieo * exp64(-kap * f, tab);
                    tf = iei - es;
                    td = fma(-kap * es, f, tf);
                }
                double t = qfe * (1.0 - mD);
                if (SALT) t *= td;
                adr = fma(t, b.x, adr);
                const double sig = sgi + b.z, sr2 = (sig * sig) * rinv2, sr6 = sr2 * (sr2 * sr2);
                const double ep = ex ? 0.0 : sei * b.w, cq = ex ? 0.0 : iei * q0;
                const double l6 = ep * sr6, cr = cq * rinv;
                const double lj = fma(48.0 * l6, sr6, fma(-24.0, l6, cr)) * rinv2; // with Coulomb
                const double fs = fma(SALT ? -td : -tau, fma(-0.25, qfe, qf3), lj);
                fx = fma(fs, dx, fx);
                fy = fma(fs, dy, fy);
                fz = fma(fs, dz, fz);
                if (ENERGY) {
                    egb = fma(SALT ? tf * qq : qq, fi, egb);
                    ec += cr;
                    elj = fma(l6, sr6 - 1.0, elj);
                }
            }
        }
    };
    if (V.kappa > 0) sweep(std::true_type{});
    else sweep(std::false_type{});
    double v[K], o[K];
    v[0] = fx;
    v[1] = fy;
    v[2] = fz;
    v[3] = adr;
    if constexpr (ENERGY) {
        v[4] = egb;
        v[5] = ec;
        v[6] = elj;
        v[7] = 0.0;
    }
    group_sums<WPA, K>(v, red, o);
    const bool owner = vi && lane == 0 && (WPA == 1 || warp == 0);
    if (owner) {
        const double taud = salt_taud(Ri, V.inv_eps_in, V.inv_eps_out, V.kappa), qR = qi * iRi;
        const double dEdR = 0.5 * fma(V.tau_pair, o[3], taud * qR * qR) -
                            (V.sa_gamma != 0.0 ? 6.0 * sa_ace(V.sa_gamma, V.sa_probe, V.rho[P + i], Ri) * iRi : 0.0);
        V.c[A + i] = dEdR * V.dRdpsi[A + i] * (0.5 * V.rt[P + i]);
        V.Fd[3 * (A + i)] = o[0];
        V.Fd[3 * (A + i) + 1] = o[1];
        V.Fd[3 * (A + i) + 2] = o[2];
    }
    if constexpr (ENERGY) {
        long long e0 = 0, e1 = 0, e2 = 0;
        if (owner) {
            const double ts = salt_tau(Ri, V.inv_eps_in, V.inv_eps_out, V.kappa);
            e0 = __double2ll_rn((-0.5 * (V.tau_pair * o[4] + ts * qi * qi * iRi) + sa_ace(V.sa_gamma, V.sa_probe, V.rho[P + i], Ri)) * kScaleE);
            e1 = __double2ll_rn(0.5 * o[5] * kScaleE);
            e2 = __double2ll_rn(2.0 * o[6] * kScaleE);
        }
        const long long t0 = block_sum_128(e0, redl), t1 = block_sum_128(e1, redl), t2 = block_sum_128(e2, redl);
        if (tid == 0) {
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 0], (unsigned long long)t0);
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 1], (unsigned long long)t1);
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 2], (unsigned long long)t2);
        }
    }
}

template <bool ENERGY, int WPA>
__global__ void __launch_bounds__(kTile) k_chain64(const Item* __restrict__ items, View V) {
    pdl_sync();
    constexpr int K = ENERGY ? 8 : 4;
    __shared__ J4<double> sa[kTile];
    __shared__ J2<double> sb[kTile];
    __shared__ double2 tab[kTab64];
    __shared__ double red[4 * K];
    __shared__ long long redl[4];
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, sub = place64<WPA>();
    const int i = it.i0 + warp / WPA;
    const bool vi = i < N;
    load_tab64(tab, tid, kTile);
    const int ic = vi ? i : it.i0;
    const double xi = V.x[3 * (A + ic)], yi = V.x[3 * (A + ic) + 1], zi = V.x[3 * (A + ic) + 2];
    const double ci = V.c[A + ic], si = V.sc[P + ic], rti = V.rt[P + ic], rc = V.rgbmax;
    double fx = 0, fy = 0, fz = 0;
    for (int j0 = 0; j0 < N; j0 += kTile) {
        __syncthreads();
        if (j0 + tid < N) {
            const int j = j0 + tid;
            sa[tid] = {V.x[3 * (A + j)], V.x[3 * (A + j) + 1], V.x[3 * (A + j) + 2], V.c[A + j]};
            sb[tid] = {V.sc[P + j], V.rt[P + j]};
        }
        __syncthreads();
#pragma unroll 1
        for (int k = sub; k < kTile; k += 32 * WPA) {
            if (j0 + (k & ~31) >= N) break;
            const bool self = j0 + k == i || j0 + k >= N;
            const int kc = min(k, N - 1 - j0);
            const J4<double> a = sa[kc];
            const J2<double> b = sb[kc];
            const double dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
            double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            r2 = self ? 1.0 : r2;
            const double rinv = rsqrt64(r2), r = r2 * rinv, rinv2 = rinv * rinv;
            const double g = fma(ci, hct_mdr64(r, rinv2, rti, b.x, rc, tab), a.w * hct_mdr64(r, rinv2, b.y, si, rc, tab));
            const double t = self ? 0.0 : g * rinv;
            fx = fma(t, dx, fx);
            fy = fma(t, dy, fy);
            fz = fma(t, dz, fz);
        }
    }
    // the atom's bonded terms: on the warp whose share of the last tile is the least
    double Fb[3] = {0.0, 0.0, 0.0}, eb = 0.0, ea = 0.0;
    const int bl = WPA == 1 ? lane : ((sub + 32) & 127); // 0..31 on the warp of entries 96..127
    if (vi) bonded_atom(V, A, P, i, bl, 32 * WPA, Fb, eb, ea);
    double v[K], o[K];
    v[0] = fx + Fb[0];
    v[1] = fy + Fb[1];
    v[2] = fz + Fb[2];
    v[3] = 0.0;
    if constexpr (ENERGY) {
        v[4] = eb;
        v[5] = ea;
        v[6] = v[7] = 0.0;
    }
    group_sums<WPA, K>(v, red, o);
    const bool owner = vi && lane == 0 && (WPA == 1 || warp == 0);
    if (owner) {
        bool ok = true;
        for (int c = 0; c < 3; ++c) {
            const double F = V.Fd[3 * (A + i) + c] + o[c];
            V.F[3 * (A + i) + c] = F;
            ok = ok && isfinite(F);
        }
        if (!ok) atomicOr(V.status, 1);
    }
    if constexpr (ENERGY) {
        const long long t0 = block_sum_128(owner ? __double2ll_rn(o[4] * kScaleE) : 0ll, redl);
        const long long t1 = block_sum_128(owner ? __double2ll_rn(o[5] * kScaleE) : 0ll, redl);
        if (tid == 0) {
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 3], (unsigned long long)t0);
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 4], (unsigned long long)t1);
        }
    }
}

} // namespace cph
