// Engine kernels: the per-step pair passes over every walker of the replica
// grid, bonded terms, Langevin integration, Monte-Carlo titration sweeps and
// replica exchanges.  Host code lives in cph_engine.cu.
//
// Work decomposition of the ordered pair passes (here, and in FP64 in
// cph_f64.cuh).  One CTA of kTile threads owns kWarpAtoms consecutive atoms i, one
// warp each; the CTA sweeps all j of its walker in tiles of kTile staged in
// shared memory, lane l of a warp taking entries l, l + 32, l + 64, l + 96 of
// every tile, so every ordered pair (i, j) is evaluated by the warp of i.  A
// lane's partial sums are added per tile into its int64 fixed-point accumulator
// (scales 2^32 and 2^40) and reduced by a fixed shuffle tree at the end, so the
// result of an atom does not depend on the launch shape (batched and per-replica
// launches agree bit for bit) and no atomics are needed.
//
// k_born, k_gb and k_chain below are those of FP32 engines with constraints, over
// the FP64 master arrays; other FP32 engines run cph_ordered.cuh over staged
// operands, and whole steps of walkers of up to 512 atoms run in cph_small.cuh.
//
// Tiles in which some atom i of the CTA meets itself or an excluded partner
// are listed per (system, i-tile) at set-up; only those run the masked loop.
#pragma once
#include "cph_device.cuh"
#include "cph_internal.h"

namespace cph {

constexpr int kTile = 128;
constexpr int kWarpAtoms = kTile / 32; // atoms i per CTA of the ordered passes, one warp each
constexpr float kFarF = 1.0e4f;

// Sum of a lane accumulator over the warp by a fixed shuffle tree; lane 0
// receives the total (the same order every time: deterministic).
template <class T>
__device__ __forceinline__ T warp_total(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// The ordered FP32 passes give each atom one warp; what follows the pair loop is
// FP64, and an FP64 instruction holds its sub-partition for 64 clocks however
// few lanes take part.  So the CTA's four atoms finish together in one warp:
// collect() hands atom w's sums to lane w of warp 0.  (8 x 1203 atoms with salt,
// energies: Born radii 47 -> 37 us, pair pass 100 -> 60, chain rule 78 -> 61
// against an epilogue in each warp.)
template <int K>
struct AtomSums {
    long long v[K][kWarpAtoms];
    // every thread of the CTA calls it, with its warp's K lane accumulators;
    // warp 0 may read v after it
    __device__ __forceinline__ void collect(const long long (&acc)[K]) {
        const int warp = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const long long s = warp_total(acc[k]);
            if ((threadIdx.x & 31) == 0 && warp < kWarpAtoms) v[k][warp] = s;
        }
        __syncthreads();
    }
};

// Sum of lanes 0 .. 3 (fixed point: the order does not matter), in lane 0.
__device__ __forceinline__ long long quad_total(long long v) {
    v += __shfl_xor_sync(0xfu, v, 2);
    v += __shfl_xor_sync(0xfu, v, 1);
    return v;
}

template <class Real>
struct alignas(sizeof(Real) * 4) J4 {
    Real x, y, z, w;
};

template <class Real>
struct alignas(sizeof(Real) * 2) J2 {
    Real x, y;
};

// The (sqrt(k) q, R, 1/R, log2(e) / (4 R)) operand of the FP32 pair kernels.
__device__ __forceinline__ float4 gb_operand(double q, double sqrt_k, double R) {
    const float r = pair_radius32(R), ir = __frcp_rn(r);
    return make_float4((float)(q * sqrt_k), r, ir, (0.25f * kLog2e) * ir);
}

// A constant of the engine in the kernel's precision: FP32 kernels take the
// copy that the host rounded.
template <class Real>
__device__ __forceinline__ Real host_const(double d, float f) {
    if constexpr (sizeof(Real) == 4) return f;
    else return d;
}

// An atom's operands from the master arrays, positions relative to the CTA's
// first atom (the passes of engines with constraints, see cph_engine::staged).
struct Masters {
    const View& V;
    int A, P;
    double cx, cy, cz;
    __device__ __forceinline__ Masters(const View& v, int a, int p, int i0) : V(v), A(a), P(p) {
        cx = V.x[3 * (A + i0)];
        cy = V.x[3 * (A + i0) + 1];
        cz = V.x[3 * (A + i0) + 2];
    }
    __device__ __forceinline__ J4<float> position(int i) const {
        return {float(V.x[3 * (A + i)] - cx), float(V.x[3 * (A + i) + 1] - cy), float(V.x[3 * (A + i) + 2] - cz), 0.f};
    }
    __device__ __forceinline__ J4<float> gb(int i) const { // sqrt(k) q, R, 1/R
        const double R = V.R[A + i];
        return {float(V.q[A + i]) * float(V.sqrt_k), pair_radius32(R), float(1.0 / R), 0.f};
    }
    __device__ __forceinline__ J2<float> lj(int i) const { // sigma / 2, sqrt(eps)
        return {float(V.sigh[P + i]), float(V.sqe[P + i])};
    }
    __device__ __forceinline__ J2<float> radii(int i) const { return {float(V.sc[P + i]), float(V.rt[P + i])}; } // s, rt
    __device__ __forceinline__ float weight(int i) const { return float(V.c[A + i]); }
};

// Per-walker energy accumulators (fixed point 2^32): GB, Coulomb, LJ, bond, angle.
constexpr int kEAcc = 5;

template <class T>
__device__ inline T block_sum_128(T v, T* red) {
    // deterministic fixed-order reduction over 128 threads
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[wid] = v;
    __syncthreads();
    T s = 0;
    if (threadIdx.x == 0) s = red[0] + red[1] + red[2] + red[3];
    return s;
}

// Build the exclusion / self masks of atom i for the j-tile starting at j0.
__device__ inline void tile_masks(const View& V, int P, int i, bool vi, int j0, uint32_t ex[4],
                                  uint32_t self[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) ex[q] = self[q] = 0u;
    if (!vi) return;
    int d = i - j0;
    if (d >= 0 && d < kTile) {
        self[d >> 5] |= 1u << (d & 31);
        ex[d >> 5] |= 1u << (d & 31);
    }
    for (int e = V.excl_off[P + i]; e < V.excl_off[P + i + 1]; ++e) {
        int dj = V.excl_j[e] - j0;
        if (dj >= 0 && dj < kTile) ex[dj >> 5] |= 1u << (dj & 31);
    }
}

// ------------------------------------------------ ends of the ordered passes
// What an atom's end of pass reads, to be loaded before the CTA's barrier.
struct BornIn {
    double rt, irho, irt, q;
    BornIn() = default;
    __device__ __forceinline__ BornIn(const View& V, int A, int P, int i)
        : rt(V.rt[P + i]), irho(V.irho[P + i]), irt(V.irt[P + i]), q(V.q[A + i]) {} // 1/rho, 1/rt from set-up
};

__device__ __forceinline__ void born_epilogue(const View& V, int A, int P, int i, long long sum, const BornIn& in) {
    const double psi = 0.5 * in.rt * Prec<float>::value(sum, kScaleH);
    const double th = tanh64(psi * (V.alpha + psi * (-V.beta + psi * V.gamma)));
    const double R = rcp64_radius(in.irt - th * in.irho);
    V.psi[A + i] = psi;
    V.R[A + i] = R;
    V.gq[A + i] = gb_operand(in.q, V.sqrt_k, R);
    V.Ffix[3 * (A + i)] = 0;
    V.Ffix[3 * (A + i) + 1] = 0;
    V.Ffix[3 * (A + i) + 2] = 0;
    V.dRfix[A + i] = 0;
    V.dRdpsi[A + i] = R * R * (1.0 - th * th) * (V.alpha + psi * (-2.0 * V.beta + 3.0 * V.gamma * psi)) * in.irho;
}

struct GbIn {
    double q, R, dRdpsi, rt, rho;
    GbIn() = default;
    __device__ __forceinline__ GbIn(const View& V, int A, int P, int i)
        : q(V.q[A + i]), R(V.R[A + i]), dRdpsi(V.dRdpsi[A + i]), rt(V.rt[P + i]), rho(V.rho[P + i]) {}
};

// lanes 0 .. 3 of warp 0; own: the lane's atom exists
template <bool ENERGY, class Sums>
__device__ __forceinline__ void gb_epilogue(const View& V, int A, int P, int w, int i, bool own, const Sums& sums,
                                            const GbIn& in) {
    using Pr = Prec<float>;
    const int l = threadIdx.x;
    long long e0 = 0, e1 = 0, e2 = 0;
    if (own) {
        const double q = in.q * V.sqrt_k;
        const double R = in.R, iR = rcp64_radius(R);
        const double qqR = q * q * iR;
        // tau(R) and its derivative form share one exponential
        double tau = V.inv_eps_in - V.inv_eps_out, taud = tau;
        if (V.kappa > 0.0) {
            const double es = V.inv_eps_out * exp64(-V.kappa * R);
            tau = V.inv_eps_in - es;
            taud = tau - V.kappa * R * es;
        }
        const double sa = V.sa_gamma != 0.0 ? sa_ace(V.sa_gamma, V.sa_probe, in.rho, R) : 0.0;
        const double dEdR = 0.5 * (V.tau_pair * Pr::value(sums.v[3][l], kScaleE) + taud * qqR * iR) - 6.0 * sa * iR;
        const double c = dEdR * in.dRdpsi * 0.5 * in.rt;
        V.c[A + i] = c;
        V.c32[A + i] = (float)c;
        for (int k = 0; k < 3; ++k) V.Fd[3 * (A + i) + k] = Pr::value(sums.v[k][l], kScaleE);
        if constexpr (ENERGY) {
            e0 = __double2ll_rn((-0.5 * (V.tau_pair * Pr::value(sums.v[4][l], kScaleE) + tau * qqR) + sa) * kScaleE);
            e1 = __double2ll_rn(0.5 * V.inv_eps_in * Pr::value(sums.v[5][l], kScaleE) * kScaleE);
            e2 = __double2ll_rn(2.0 * Pr::value(sums.v[6][l], kScaleE) * kScaleE);
        }
    }
    if constexpr (ENERGY) {
        e0 = quad_total(e0);
        e1 = quad_total(e1);
        e2 = quad_total(e2);
        if (l == 0) {
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 0], (unsigned long long)e0);
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 1], (unsigned long long)e1);
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 2], (unsigned long long)e2);
        }
    }
}

// ------------------------------------------------------------- pass 1: Born radii
// psi_i = rt_i/2 sum_{j != i} H(r_ij, rt_i, s_j); R_i = 1/(1/rt_i - tanh(theta)/rho_i)
// with theta = alpha psi - beta psi^2 + gamma psi^3, finalised in FP64.
__global__ void __launch_bounds__(kTile) k_born(const Item* __restrict__ items, View V,
                                                int zero_energy) {
    pdl_sync();
    using Real = float;
    using Pr = Prec<Real>;
    __shared__ J4<Real> sj[kTile];
    __shared__ AtomSums<1> sums;
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31;
    const int i = it.i0 + (tid >> 5); // one warp per atom
    const bool vi = i < N;
    if (it.i0 == 0) {
        if (zero_energy && tid < kEAcc) V.eacc[w * kEAcc + tid] = 0;
        if (tid == kEAcc) V.vscale[w] = 1.0;
    }
    const Masters stage(V, A, P, it.i0);
    Real xi = Real(-kFarF), yi = Real(-kFarF), zi = Real(-kFarF), rti = Real(1);
    if (vi) {
        const J4<Real> p = stage.position(i);
        xi = p.x;
        yi = p.y;
        zi = p.z;
        rti = stage.radii(i).y;
    }
    const Real irti = Real(1) / rti;
    const Real rc = Real(V.rgbmax); // Born-radius cutoff (INFINITY = none)
    typename Pr::Acc acc = 0;
    Real part = 0;
    int mp = V.mt_off[it.st];
    const int me = V.mt_off[it.st + 1];
    int next = mp < me ? V.mt_list[mp] : 0x7fffffff;
    for (int j0 = 0, jt = 0; j0 < N; j0 += kTile, ++jt) {
        __syncthreads();
        {
            const int j = j0 + tid;
            J4<Real> v;
            if (j < N) {
                v = stage.position(j);
                v.w = stage.radii(j).x;
            } else {
                v.x = v.y = v.z = Real(kFarF);
                v.w = Real(0);
            }
            sj[tid] = v;
        }
        __syncthreads();
        if (jt != next) {
#pragma unroll
            for (int k = lane; k < kTile; k += 32) {
                const J4<Real> b = sj[k];
                const Real dx = xi - b.x, dy = yi - b.y, dz = zi - b.z;
                const Real r2 = dx * dx + dy * dy + dz * dz;
                const Real rinv = Pr::rsqrt(r2);
                part += hct(r2 * rinv, rinv, rti, irti, b.w, rc);
            }
        } else {
            ++mp;
            next = mp < me ? V.mt_list[mp] : 0x7fffffff;
            const int dself = i - j0;
#pragma unroll
            for (int k = lane; k < kTile; k += 32) {
                const J4<Real> b = sj[k];
                const bool self = (k == dself);
                const Real dx = xi - b.x, dy = yi - b.y, dz = zi - b.z;
                Real r2 = dx * dx + dy * dy + dz * dz;
                r2 = self ? Real(1) : r2;
                const Real rinv = Pr::rsqrt(r2);
                const Real h = hct(r2 * rinv, rinv, rti, irti, b.w, rc);
                part += self ? Real(0) : h;
            }
        }
        Pr::add(acc, part, Real(kScaleH));
        part = 0;
    }
    sums.collect({acc});
    if (tid < kWarpAtoms && it.i0 + tid < N) {
        born_epilogue(V, A, P, it.i0 + tid, sums.v[0][tid], BornIn(V, A, P, it.i0 + tid));
    }
}

// ------------------------------------------- pass 2: GB + Coulomb + LJ pair pass
// Owner i accumulates the direct force, dE_GB/dR_i and (optionally) its share
// of the energies; the epilogue turns dE/dR_i into c_i = dE/dR_i dR_i/dpsi_i rt_i/2.
template <bool ENERGY>
__global__ void __launch_bounds__(kTile) k_gb(const Item* __restrict__ items, View V) {
    pdl_sync();
    using Real = float;
    using Pr = Prec<Real>;
    using Acc = typename Pr::Acc;
    __shared__ J4<Real> sa[kTile];
    __shared__ J4<Real> sb[kTile];
    __shared__ AtomSums<ENERGY ? 7 : 4> sums;
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31;
    const int i = it.i0 + (tid >> 5); // one warp per atom
    const bool vi = i < N;
    const Masters stage(V, A, P, it.i0);
    Real xi = Real(-kFarF), yi = Real(-kFarF), zi = Real(-kFarF);
    Real qi = 0, Ri = 1, iRi = 1, sgi = 0, sei = 0;
    if (vi) {
        const J4<Real> p = stage.position(i), g = stage.gb(i);
        const J2<Real> l = stage.lj(i);
        xi = p.x;
        yi = p.y;
        zi = p.z;
        qi = g.x;
        Ri = g.y;
        iRi = g.z;
        sgi = l.x;
        sei = l.y;
    }
    // FP32: the host-rounded copies (no double -> float conversion in the loops)
    const Real tau = host_const<Real>(V.tau, V.tau32), iei = host_const<Real>(V.inv_eps_in, V.iei32);
    const Real kap = host_const<Real>(V.kappa, V.kappa32), ieo = host_const<Real>(V.inv_eps_out, V.ieo32);
    const bool salt = V.kappa > 0; // pair sums then carry tau(f) and taud(f) per pair
    Acc fx = 0, fy = 0, fz = 0, adr = 0, egb = 0, ec = 0, elj = 0;
    Real px = 0, py = 0, pz = 0, pdr = 0;
    KSum<Real> pgb, pc, plj;
    int mp = V.mt_off[it.st];
    const int me = V.mt_off[it.st + 1];
    int next = mp < me ? V.mt_list[mp] : 0x7fffffff;
    for (int j0 = 0, jt = 0; j0 < N; j0 += kTile, ++jt) {
        __syncthreads();
        {
            const int j = j0 + tid;
            J4<Real> a, b;
            if (j < N) {
                const J4<Real> g = stage.gb(j);
                const J2<Real> l = stage.lj(j);
                a = stage.position(j);
                a.w = g.x;
                b.x = g.y;
                b.y = g.z;
                b.z = l.x;
                b.w = l.y;
            } else {
                a.x = a.y = a.z = Real(kFarF);
                a.w = 0;
                b.x = b.y = Real(1);
                b.z = b.w = 0;
            }
            sa[tid] = a;
            sb[tid] = b;
        }
        __syncthreads();
        if (jt != next) {
#pragma unroll
            for (int k = lane; k < kTile; k += 32) {
                const J4<Real> a = sa[k];
                const J4<Real> b = sb[k];
                const Real dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
                const Real r2 = dx * dx + dy * dy + dz * dz;
                const Real rinv = Pr::rsqrt(r2);
                const Real rinv2 = rinv * rinv;
                const Real qq = qi * a.w;
                const Real D = Real(0.25) * r2 * (iRi * b.y);
                const Real e = Pr::expm(D);
                const Real f2 = r2 + (Ri * b.x) * e;
                const Real fi = Pr::rsqrt(f2);
                const Real qf3 = qq * fi * fi * fi;
                Real tf = Real(1), td = Real(1);
                if (salt) {
                    const Real kf = kap * (f2 * fi);
                    const Real es = ieo * Pr::expm(kf);
                    tf = iei - es;
                    td = tf - kf * es;
                }
                pdr += td * qf3 * b.x * e * (Real(1) + D);
                const Real sig = sgi + b.z;
                const Real sr2 = sig * sig * rinv2;
                const Real sr6 = sr2 * sr2 * sr2;
                const Real ep = sei * b.w;
                const Real fs = iei * qq * rinv * rinv2 + Real(4) * ep * sr6 * (Real(12) * sr6 - Real(6)) * rinv2
                              - (salt ? td : tau) * qf3 * (Real(1) - Real(0.25) * e);
                px += fs * dx;
                py += fs * dy;
                pz += fs * dz;
                if (ENERGY) {
                    pgb.add(tf * qq * fi);
                    pc.add(qq * rinv);
                    plj.add(ep * sr6 * (sr6 - Real(1)));
                }
            }
        } else {
            ++mp;
            next = mp < me ? V.mt_list[mp] : 0x7fffffff;
            uint32_t mex[4], mself[4];
            tile_masks(V, P, i, vi, j0, mex, mself);
#pragma unroll
            for (int k = lane; k < kTile; k += 32) {
                {
                    const int q4 = k >> 5, kk = k & 31;
                    const bool self = (mself[q4] >> kk) & 1u;
                    const bool ex = (mex[q4] >> kk) & 1u;
                    const J4<Real> a = sa[k];
                    const J4<Real> b = sb[k];
                    const Real dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
                    Real r2 = dx * dx + dy * dy + dz * dz;
                    r2 = self ? Real(1) : r2;
                    const Real g = self ? Real(0) : Real(1);
                    const Real nb = ex ? Real(0) : Real(1);
                    const Real rinv = Pr::rsqrt(r2);
                    const Real rinv2 = rinv * rinv;
                    const Real qq = qi * a.w;
                    const Real D = Real(0.25) * r2 * (iRi * b.y);
                    const Real e = Pr::expm(D);
                    const Real f2 = r2 + (Ri * b.x) * e;
                    const Real fi = Pr::rsqrt(f2);
                    const Real qf3 = g * qq * fi * fi * fi;
                    Real tf = Real(1), td = Real(1);
                    if (salt) {
                        const Real kf = kap * (f2 * fi);
                        const Real es = ieo * Pr::expm(kf);
                        tf = iei - es;
                        td = tf - kf * es;
                    }
                    pdr += td * qf3 * b.x * e * (Real(1) + D);
                    const Real sig = sgi + b.z;
                    const Real sr2 = sig * sig * rinv2;
                    const Real sr6 = sr2 * sr2 * sr2;
                    const Real ep = nb * sei * b.w;
                    const Real fs = nb * iei * qq * rinv * rinv2
                                  + Real(4) * ep * sr6 * (Real(12) * sr6 - Real(6)) * rinv2
                                  - (salt ? td : tau) * qf3 * (Real(1) - Real(0.25) * e);
                    px += fs * dx;
                    py += fs * dy;
                    pz += fs * dz;
                    if (ENERGY) {
                        pgb.add(tf * g * qq * fi);
                        pc.add(nb * qq * rinv);
                        plj.add(ep * sr6 * (sr6 - Real(1)));
                    }
                }
            }
        }
        Pr::add(fx, px, Real(kScaleE));
        Pr::add(fy, py, Real(kScaleE));
        Pr::add(fz, pz, Real(kScaleE));
        Pr::add(adr, pdr, Real(kScaleE));
        px = py = pz = pdr = 0;
        if (ENERGY) {
            Pr::add(egb, pgb.value(), Real(kScaleE));
            Pr::add(ec, pc.value(), Real(kScaleE));
            Pr::add(elj, plj.value(), Real(kScaleE));
            pgb = pc = plj = KSum<Real>();
        }
    }
    if constexpr (ENERGY) sums.collect({fx, fy, fz, adr, egb, ec, elj});
    else sums.collect({fx, fy, fz, adr});
    if (tid >= kWarpAtoms) return;
    const bool own = it.i0 + tid < N;
    gb_epilogue<ENERGY>(V, A, P, w, it.i0 + tid, own, sums, own ? GbIn(V, A, P, it.i0 + tid) : GbIn());
}

// Bonded forces on atom i (system-local index li) and its owned energy
// shares (a bond or angle is owned by its first atom), split over the threads
// of the atom's group: thread l takes the atom's terms l, l + stride, ... of
// each kind (the caller sums the threads in a fixed order).
__device__ inline void bonded_atom(const View& V, int A, int P, int li, int lane, int stride, double F[3],
                                   double& eb, double& ea) {
    const double* x = V.x;
    for (int e = V.bond_off[P + li] + lane; e < V.bond_off[P + li + 1]; e += stride) {
        const int b = V.bond_idx[e];
        const int ia = V.bond_ij[2 * b], ib = V.bond_ij[2 * b + 1];
        const int o = (ia == li) ? ib : ia;
        double d[3];
        for (int c = 0; c < 3; ++c) d[c] = x[3 * (A + li) + c] - x[3 * (A + o) + c];
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2], ir = rsqrt64(r2);
        const double dr = r2 * ir - V.bond_r0[b];
        const double g = 2.0 * V.bond_k[b] * dr * ir;
        for (int c = 0; c < 3; ++c) F[c] -= g * d[c];
        if (ia == li) eb += V.bond_k[b] * dr * dr;
    }
    for (int e = V.ang_off[P + li] + lane; e < V.ang_off[P + li + 1]; e += stride) {
        const int a = V.ang_idx[e];
        const int ia = V.ang_ijk[3 * a], ib = V.ang_ijk[3 * a + 1], ic = V.ang_ijk[3 * a + 2];
        double u[3], v[3];
        for (int c = 0; c < 3; ++c) {
            u[c] = x[3 * (A + ia) + c] - x[3 * (A + ib) + c];
            v[c] = x[3 * (A + ic) + c] - x[3 * (A + ib) + c];
        }
        const double ru2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        const double rv2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        const double iuv = rsqrt64(ru2 * rv2), iru2 = rcp64(ru2), irv2 = rcp64(rv2);
        double cs = (u[0] * v[0] + u[1] * v[1] + u[2] * v[2]) * iuv;
        cs = fmin(1.0, fmax(-1.0, cs));
        const double th = acos(cs);
        const double dth = th - V.ang_t0[a];
        const double k = -2.0 * V.ang_k[a] * dth * rsqrt64(fmax(1e-300, 1.0 - cs * cs)); // dE/dcos
        double gi[3], gk[3];
        for (int c = 0; c < 3; ++c) {
            gi[c] = k * (v[c] * iuv - cs * u[c] * iru2);
            gk[c] = k * (u[c] * iuv - cs * v[c] * irv2);
        }
        for (int c = 0; c < 3; ++c) {
            if (li == ia) F[c] -= gi[c];
            if (li == ic) F[c] -= gk[c];
            if (li == ib) F[c] += gi[c] + gk[c];
        }
        if (ia == li) ea += V.ang_k[a] * dth * dth;
    }
}

// FP32-mode bonded terms (the symmetric bonded kernel and the ordered chain
// kernel share them): FP64 only where a difference of nearly equal numbers
// decides the result (the separations, r^2 - r0^2, the dot and cross products
// behind the sine and cosine of theta - theta0), FP32 elsewhere (atan2f for
// theta - theta0), so that the few FP64 units of the chip are not the bound.
//
// One harmonic bond from its FP64 separation d = x_i - x_j: the force on i is
// -g d, on j +g d; e its energy.
__device__ __forceinline__ void bond_term32(const double (&d)[3], double r0d, double kbd, float& g, float& e) {
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const float r = sqrtf((float)r2);
    const float dr = (float)(r2 - r0d * r0d) / (r + (float)r0d); // r - r0 at FP32 relative precision
    const float kb = (float)kbd;
    g = 2.f * kb * dr / r;
    e = kb * dr * dr;
}

// One harmonic angle i-j-k from u = x_i - x_j, v = x_k - x_j (FP64) and
// (cos theta0, sin theta0): the force on i is -gi, on k -gk, on j gi + gk;
// kz holds the two factors of gk[2], e the energy.
__device__ __forceinline__ void angle_term32(const double (&u)[3], const double (&v)[3], double2 cs0, double kad,
                                             float (&gi)[3], float (&gk)[3], float2& kz, float& e) {
    // |u||v| cos(theta) and |u||v| sin(theta) in FP64 (the norm of the cross
    // product by an FP32 reciprocal square root and one Newton step)
    const double uv = u[0] * v[0] + u[1] * v[1] + u[2] * v[2];
    const double cx = u[1] * v[2] - u[2] * v[1], cy = u[2] * v[0] - u[0] * v[2], cz = u[0] * v[1] - u[1] * v[0];
    const double w2 = cx * cx + cy * cy + cz * cz;
    const double y = (double)rsqrtf(fmaxf((float)w2, 1e-30f));
    double wn = w2 * y;
    wn += 0.5 * (w2 - wn * wn) * y;
    // theta - theta0 = atan2(sin(theta - theta0), cos(theta - theta0))
    const float dth = atan2f((float)(wn * cs0.x - uv * cs0.y), (float)(uv * cs0.x + wn * cs0.y));
    const float ka = (float)kad;
    float uf[3], vf[3];
    for (int c = 0; c < 3; ++c) {
        uf[c] = (float)u[c];
        vf[c] = (float)v[c];
    }
    const float ru2 = uf[0] * uf[0] + uf[1] * uf[1] + uf[2] * uf[2];
    const float rv2 = vf[0] * vf[0] + vf[1] * vf[1] + vf[2] * vf[2];
    const float iuv = rsqrtf(ru2 * rv2);                     // 1 / (|u| |v|)
    const float cs = (float)uv * iuv, sn = fmaxf((float)wn * iuv, 1e-20f);
    const float k = -2.f * ka * dth / sn;                     // dE/dcos(theta)
    for (int c = 0; c < 3; ++c) {
        gi[c] = k * (vf[c] * iuv - cs * uf[c] / ru2);
        const float wk = uf[c] * iuv - cs * vf[c] / rv2;
        gk[c] = k * wk;
        if (c == 2) kz = make_float2(k, wk);
    }
    e = ka * dth * dth;
}

// The FP32-mode terms of one atom (the ordered chain kernel: each atom takes
// the terms it is part of), its forces and energies summed in FP32.
__device__ inline void bonded_atom32(const View& V, int A, int P, int li, int lane, int stride, float F[3],
                                     float& eb, float& ea) {
    const double* x = V.x;
    for (int e = V.bond_off[P + li] + lane; e < V.bond_off[P + li + 1]; e += stride) {
        const int b = V.bond_idx[e];
        const int ia = V.bond_ij[2 * b], ib = V.bond_ij[2 * b + 1];
        const int o = (ia == li) ? ib : ia;
        double d[3];
        for (int c = 0; c < 3; ++c) d[c] = x[3 * (A + li) + c] - x[3 * (A + o) + c];
        float g, en;
        bond_term32(d, V.bond_r0[b], V.bond_k[b], g, en);
        for (int c = 0; c < 3; ++c) F[c] -= g * (float)d[c];
        if (ia == li) eb += en;
    }
    for (int e = V.ang_off[P + li] + lane; e < V.ang_off[P + li + 1]; e += stride) {
        const int a = V.ang_idx[e];
        const int ia = V.ang_ijk[3 * a], ib = V.ang_ijk[3 * a + 1], ic = V.ang_ijk[3 * a + 2];
        double u[3], v[3];
        for (int c = 0; c < 3; ++c) {
            u[c] = x[3 * (A + ia) + c] - x[3 * (A + ib) + c];
            v[c] = x[3 * (A + ic) + c] - x[3 * (A + ib) + c];
        }
        float gi[3], gk[3], en;
        float2 kz;
        angle_term32(u, v, V.ang_cs0[a], V.ang_k[a], gi, gk, kz, en);
        for (int c = 0; c < 3; ++c) {
            if (li == ia) F[c] -= gi[c];
            if (li == ic) F[c] -= gk[c];
            if (li == ib) F[c] += gi[c] + gk[c];
        }
        if (ia == li) ea += en;
    }
}

// Bonded terms of a CTA's four atoms in one warp, eight lanes to an atom.
struct BondedSums {
    float f[kWarpAtoms][3], eb[kWarpAtoms], ea[kWarpAtoms];
    template <bool ENERGY>
    __device__ __forceinline__ void take(const View& V, int A, int P, int i0, int N, int lane) {
        constexpr int kL = 32 / kWarpAtoms;
        const int a = lane / kL;
        float fb[3] = {0.f, 0.f, 0.f}, ebf = 0.f, eaf = 0.f;
        if (i0 + a < N) bonded_atom32(V, A, P, i0 + a, lane % kL, kL, fb, ebf, eaf);
        __syncwarp();
#pragma unroll
        for (int o = kL / 2; o > 0; o >>= 1) {
            for (int c = 0; c < 3; ++c) fb[c] += __shfl_down_sync(0xffffffffu, fb[c], o, kL);
            if (ENERGY) {
                ebf += __shfl_down_sync(0xffffffffu, ebf, o, kL);
                eaf += __shfl_down_sync(0xffffffffu, eaf, o, kL);
            }
        }
        if (lane % kL == 0) {
            for (int c = 0; c < 3; ++c) f[a][c] = fb[c];
            eb[a] = ebf;
            ea[a] = eaf;
        }
    }
};

// lanes 0 .. 3 of warp 0; own: the lane's atom exists
template <bool ENERGY, class Sums>
__device__ __forceinline__ void chain_epilogue(const View& V, int A, int w, int i, bool own, const Sums& sums,
                                               const BondedSums& bonded) {
    const int l = threadIdx.x;
    if (own) {
        double F[3];
        for (int c = 0; c < 3; ++c) {
            F[c] = V.Fd[3 * (A + i) + c] + Prec<float>::value(sums.v[c][l], kScaleE) + (double)bonded.f[l][c];
            V.F[3 * (A + i) + c] = F[c];
        }
        if (!(isfinite(F[0]) && isfinite(F[1]) && isfinite(F[2]))) atomicOr(V.status, 1);
    }
    if (ENERGY) {
        const long long t0 = quad_total(__double2ll_rn((double)bonded.eb[l] * kScaleE));
        const long long t1 = quad_total(__double2ll_rn((double)bonded.ea[l] * kScaleE));
        if (l == 0) {
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 3], (unsigned long long)t0);
            atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 4], (unsigned long long)t1);
        }
    }
}

// ------------------------------------------ pass 3: chain rule through Born radii
// F_i -= sum_j (c_i dH(r; rt_i, s_j)/dr + c_j dH(r; rt_j, s_i)/dr) (x_i - x_j)/r,
// then the direct pair force and the bonded terms are added: F is the total force.
template <bool ENERGY>
__global__ void __launch_bounds__(kTile) k_chain(const Item* __restrict__ items, View V) {
    pdl_sync();
    using Real = float;
    using Pr = Prec<Real>;
    using Acc = typename Pr::Acc;
    __shared__ J4<Real> sa[kTile];
    __shared__ J2<Real> sb[kTile];
    __shared__ AtomSums<3> sums;
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31;
    const int i = it.i0 + (tid >> 5); // one warp per atom
    const bool vi = i < N;
    const Masters stage(V, A, P, it.i0);
    Real xi = Real(-kFarF), yi = Real(-kFarF), zi = Real(-kFarF), ci = 0, si = 0, rti = 1;
    if (vi) {
        const J4<Real> p = stage.position(i);
        const J2<Real> r = stage.radii(i);
        xi = p.x;
        yi = p.y;
        zi = p.z;
        ci = stage.weight(i);
        si = r.x;
        rti = r.y;
    }
    Acc fx = 0, fy = 0, fz = 0;
    const Real rc = Real(V.rgbmax); // Born-radius cutoff (INFINITY = none)
    Real px = 0, py = 0, pz = 0;
    int mp = V.mt_off[it.st];
    const int me = V.mt_off[it.st + 1];
    int next = mp < me ? V.mt_list[mp] : 0x7fffffff;
    for (int j0 = 0, jt = 0; j0 < N; j0 += kTile, ++jt) {
        __syncthreads();
        {
            const int j = j0 + tid;
            J4<Real> a;
            J2<Real> b;
            if (j < N) {
                a = stage.position(j);
                a.w = stage.weight(j);
                b = stage.radii(j);
            } else {
                a.x = a.y = a.z = Real(kFarF);
                a.w = 0;
                b.x = 0;
                b.y = 1;
            }
            sa[tid] = a;
            sb[tid] = b;
        }
        __syncthreads();
        if (jt != next) {
#pragma unroll
            for (int k = lane; k < kTile; k += 32) {
                const J4<Real> a = sa[k];
                const J2<Real> b = sb[k];
                const Real dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
                const Real r2 = dx * dx + dy * dy + dz * dz;
                const Real rinv = Pr::rsqrt(r2);
                const Real r = r2 * rinv;
                const Real g = ci * hct_dr(r, rinv, rti, b.x, rc) + a.w * hct_dr(r, rinv, b.y, si, rc);
                const Real t = -g * rinv;
                px += t * dx;
                py += t * dy;
                pz += t * dz;
            }
        } else {
            ++mp;
            next = mp < me ? V.mt_list[mp] : 0x7fffffff;
            const int dself = i - j0;
#pragma unroll
            for (int k = lane; k < kTile; k += 32) {
                const J4<Real> a = sa[k];
                const J2<Real> b = sb[k];
                const bool self = (k == dself);
                const Real dx = xi - a.x, dy = yi - a.y, dz = zi - a.z;
                Real r2 = dx * dx + dy * dy + dz * dz;
                r2 = self ? Real(1) : r2;
                const Real rinv = Pr::rsqrt(r2);
                const Real r = r2 * rinv;
                const Real g = ci * hct_dr(r, rinv, rti, b.x, rc) + a.w * hct_dr(r, rinv, b.y, si, rc);
                const Real t = self ? Real(0) : -g * rinv;
                px += t * dx;
                py += t * dy;
                pz += t * dz;
            }
        }
        Pr::add(fx, px, Real(kScaleE));
        Pr::add(fy, py, Real(kScaleE));
        Pr::add(fz, pz, Real(kScaleE));
        px = py = pz = 0;
    }
    __shared__ BondedSums bonded;
    if (tid < 32) bonded.take<ENERGY>(V, A, P, it.i0, N, lane);
    sums.collect({fx, fy, fz});
    if (tid < kWarpAtoms) chain_epilogue<ENERGY>(V, A, w, it.i0 + tid, it.i0 + tid < N, sums, bonded);
}

// ------------------------------------------------------------ Langevin step
// v' = [(1 - g dt/2) v + dt A F/m + sqrt(2 g kB T A dt/m) z] / (1 + g dt/2),
// x' = x + dt v', with T the temperature of the walker's current slot and z
// three normals from one Philox draw (Box-Muller on words (0,1) and (2,3)).
// sin and cos of 2 pi (w + 1/2) / 2^32: the nearest quarter turn from the integer,
// Taylor series on the rest (|t| <= pi/4; remainders 5e-17 and 2e-18).
__device__ __forceinline__ void sincos64(uint32_t w, double& sn, double& cs) {
    const uint32_t k = (w + 0x20000000u) >> 30;
    const double t = fma((double)(int)(w - (k << 30)), 1.4629180792671596e-09, 7.314590396335798e-10);
    const double t2 = t * t;
    double p = fma(t2, -7.647163731819816e-13, 1.6059043836821613e-10);
    p = fma(p, t2, -2.505210838544172e-08);
    p = fma(p, t2, 2.7557319223985893e-06);
    p = fma(p, t2, -0.0001984126984126984);
    p = fma(p, t2, 0.008333333333333333);
    p = fma(p, t2, -0.16666666666666666);
    const double s = fma(p * t2, t, t);
    double q = fma(t2, 4.779477332387385e-14, -1.1470745597729725e-11);
    q = fma(q, t2, 2.08767569878681e-09);
    q = fma(q, t2, -2.755731922398589e-07);
    q = fma(q, t2, 2.48015873015873e-05);
    q = fma(q, t2, -0.001388888888888889);
    q = fma(q, t2, 0.041666666666666664);
    q = fma(q, t2, -0.5);
    const double c = fma(q, t2, 1.0);
    const double a = (k & 1u) ? c : s, b = (k & 1u) ? s : c; // quarter turns
    sn = (k & 2u) ? -a : a;
    cs = ((k + 1u) & 2u) ? -b : b;
}

// The library's sincospi, log and sqrt took ~190 FP64 instructions for an atom's
// three normals, this ~85: one of their two Box-Muller pairs (z0, z1) or (z2, -).
__device__ __forceinline__ void normals64(uint64_t seed, uint32_t idx, uint32_t stream, uint64_t step, int pair,
                                          double z[2], const double2* tab) {
    const U4 u = draw(seed, idx, stream, step, kRngLangevin);
    const double l = -2.0 * log64(unit_open(pair ? u.c : u.a), tab);
    const double r = l * rsqrt64(l);
    double sn, cs;
    sincos64(pair ? u.d : u.b, sn, cs);
    z[0] = r * cs;
    z[1] = r * sn;
}

__device__ inline void normals3(uint64_t seed, uint32_t idx, uint32_t stream,
                                       uint64_t step, float z[3]) {
    U4 u = draw(seed, idx, stream, step, kRngLangevin);
    const float r0 = sqrtf(-2.0f * logf((float)unit_open(u.a)));
    const float r1 = sqrtf(-2.0f * logf((float)unit_open(u.c)));
    float sn, cs;
    sincospif(2.0f * (float)unit_open(u.b), &sn, &cs);
    z[0] = r0 * cs;
    z[1] = r0 * sn;
    z[2] = r1 * cospif(2.0f * (float)unit_open(u.d));
}

// One sample of the observables for walker w (a warp or more; n threads).
__device__ inline void observe_walker(const View& V, int w, int tid, int n) {
    if (!V.w_local[w]) return; // a sharded grid's counts are summed over its engines
    const int s = V.slot_of[w];
    if (tid == 0) {
        V.visits[(long long)w * V.W + s] += 1;
        if (w == V.first_local) *V.n_obs += 1;
    }
    // the walker at slot s belongs to the system of the walker that started
    // there, so slot s's rows are laid out like walker s's sites
    const int ws0 = V.w_site_off[w], ns = V.w_site_off[w + 1] - ws0;
    const long long row0 = V.w_site_off[s];
    for (int k = tid; k < ns; k += n) V.occ[(row0 + k) * CPH_MAX_STATES + V.site_state[ws0 + k]] += 1;
}

// Threads to an atom: in FP64 one for each Box-Muller pair, whose FP64 chain is
// most of the kernel for a small walker (100 steps of 160 atoms 4.92 -> 4.74 ms).
template <class Real>
constexpr int kLangevinThreads = sizeof(Real) == 8 ? 2 : 1;

// Blocks past the atoms' own (obs of them, one per walker) take the step's sample
// of the observables, which depends on nothing the step moves: a launch of 5 us
// less a step.
template <class Real>
__global__ void k_langevin(View V, int s_off, int a0, int n, int obs) {
    pdl_sync();
    const int nb = gridDim.x - obs;
    if ((int)blockIdx.x >= nb) {
        observe_walker(V, (int)blockIdx.x - nb, threadIdx.x, blockDim.x);
        return;
    }
    __shared__ double2 tab[sizeof(Real) == 8 ? kTab64 : 1];
    if constexpr (sizeof(Real) == 8) {
        load_tab64(tab, threadIdx.x, blockDim.x);
        __syncthreads();
    }
    constexpr int kT = kLangevinThreads<Real>;
    const int thread = blockIdx.x * blockDim.x + threadIdx.x, l = thread / kT;
    if (l >= n) return;
    const int a = a0 + l;
    const int w = V.a_walker[a];
    if (!V.w_local[w]) return;
    const int li = a - V.w_off[w];
    const int P = V.sys_poff[V.w_sys[w]];
    const uint64_t t = (uint64_t)(*V.step + s_off);
    const int slot = V.slot_of[w];
    const int first = kT == 1 ? 0 : 2 * (thread % kT), nc = kT == 1 ? 3 : 2 - thread % kT; // the thread's components
    Real z[3];
    if constexpr (sizeof(Real) == 8) normals64(V.seed, (uint32_t)li, (uint32_t)w, t, thread % kT, z, tab);
    else normals3(V.seed, (uint32_t)li, (uint32_t)w, t, z);
    // per-atom factors dt A / m and sqrt(2 g kB A dt / m), and sqrt(T) per
    // slot, are set up once: no FP64 division or square root per step
    const double sd = V.lg_sqT[slot / (V.nE * V.npH)] * V.lg_sf[P + li];
    const double im = V.lg_im[P + li], c1 = V.lg_c1, c2 = V.lg_c2;
    const double vs = V.vscale[w];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < (kT == 1 ? 3 : 2); ++k) {
        if (k >= nc) break;
        const int c = first + k;
        const double vn = (c1 * (V.v[3 * a + c] * vs) + im * V.F[3 * a + c] + sd * (double)z[k]) * c2;
        V.v[3 * a + c] = vn;
        if (V.xprev) V.xprev[3 * a + c] = V.x[3 * a + c]; // SHAKE's reference bond vectors
        const double xn = V.x[3 * a + c] + V.dt * vn;
        V.x[3 * a + c] = xn;
        ok = ok && isfinite(xn);
    }
    if (!ok) atomicOr(V.status, 2);
}

// SHAKE (Ryckaert, Ciccotti & Berendsen 1977) after the leapfrog step, one
// thread per (walker, cluster of one heavy atom and its hydrogens): each
// constraint in turn moves its two atoms along the bond vector before the
// step, in inverse proportion to their masses, until none of the cluster's
// constraints moves (|d0^2 - d^2| <= 2 tol d0^2); velocities take the
// displacement / dt.  The sweeps are bounded; a cluster that does not settle
// raises status flag 8.
constexpr int kShakeMaxH = 8, kShakeMaxIter = 1000;

__global__ void k_shake(View V, int i0, int n) {
    pdl_sync();
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const int it = i0 + l;
    const int w = V.shk_item_w[it], c = V.shk_item_c[it];
    if (!V.w_local[w]) return;
    const int A = V.w_off[w], P = V.sys_poff[V.w_sys[w]];
    const int h0 = V.shk_off[c], nh = V.shk_off[c + 1] - h0;
    int at[kShakeMaxH + 1];
    double xo[kShakeMaxH + 1][3], xn[kShakeMaxH + 1][3], x0[kShakeMaxH + 1][3], im[kShakeMaxH + 1];
    at[0] = V.shk_heavy[c];
    for (int k = 0; k < nh; ++k) at[k + 1] = V.shk_h[h0 + k];
    for (int k = 0; k <= nh; ++k) {
        const int a = A + at[k];
        im[k] = 1.0 / V.mass[P + at[k]];
        for (int d = 0; d < 3; ++d) {
            xo[k][d] = V.xprev[3 * a + d];
            xn[k][d] = x0[k][d] = V.x[3 * a + d];
        }
    }
    const double tol2 = 2.0 * V.shake_tol;
    bool done = false;
    for (int iter = 0; iter < kShakeMaxIter && !done; ++iter) {
        done = true;
        for (int k = 1; k <= nh; ++k) {
            const double d0 = V.shk_d[h0 + k - 1];
            double rij[3], rold[3], r2 = 0.0, dot = 0.0;
            for (int d = 0; d < 3; ++d) {
                rij[d] = xn[0][d] - xn[k][d];
                rold[d] = xo[0][d] - xo[k][d];
                r2 += rij[d] * rij[d];
                dot += rold[d] * rij[d];
            }
            const double diff = d0 * d0 - r2;
            if (fabs(diff) > tol2 * d0 * d0) {
                done = false;
                const double g = diff / (2.0 * dot * (im[0] + im[k]));
                for (int d = 0; d < 3; ++d) {
                    xn[0][d] += g * rold[d] * im[0];
                    xn[k][d] -= g * rold[d] * im[k];
                }
            }
        }
    }
    if (!done) atomicOr(V.status, 8);
    for (int k = 0; k <= nh; ++k) {
        const int a = A + at[k];
        for (int d = 0; d < 3; ++d) {
            V.x[3 * a + d] = xn[k][d];
            V.v[3 * a + d] += (xn[k][d] - x0[k][d]) / V.dt;
        }
    }
}

// velocities *= vscale[walker] (a stand-alone T exchange)
__global__ void k_vscale(View V) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= V.total_atoms) return;
    const double s = V.vscale[V.a_walker[a]];
    for (int c = 0; c < 3; ++c) V.v[3 * a + c] *= s;
}

__global__ void k_vscale_reset(View V) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < V.W) V.vscale[w] = 1.0;
}

__global__ void k_tick(long long* step, long long n) { pdl_sync(); *step += n; }

} // namespace cph
