// MD steps of small walkers in FP32 mode, whole steps in one launch: one
// thread-block cluster per walker.
//
// What bounds a small walker is not arithmetic (a 160-atom step is 12,720
// pairs) but the chain of dependent launches, each a few microseconds: Born
// radii, GB pass, chain pass, observables, Langevin step (and SHAKE), 55 us a
// step for 8 x 160 atoms.  Here the passes of a step are phases of one kernel,
// separated by hardware cluster barriers (~400 clocks), and a launch runs
// steps until the schedule needs something of another kernel (a titration
// sweep, an exchange attempt).  Measured, with sweeps every 10 steps: 8 x 160
// atoms 58.5 -> 20 us a step (15 in this kernel), 4 x 246 atoms with constraints
// 91 -> 39 us.  Which walkers come here: small_setup in cph_engine.cu and
// small_pays below.
//
// Work split.  A cluster of eight CTAs (portable; of sixteen-CTA clusters only
// seven fit the chip) holds the walker.  A warp owns GA consecutive atoms i, its
// lanes the partners j = lane + 32 m; the positions relative to the first atom of
// each group of four are formed once a step, in shared memory, for all three
// passes.  Extra warps evaluate the bonded terms that touch the CTA's
// atoms, gather them and draw the random numbers meanwhile.  Each CTA holds the
// whole walker's operands in shared memory (130 bytes an atom); what changes in
// a phase (positions, radii, chain weights) its owner writes into every CTA of
// the cluster.
//
// FP64 is what a step of this size must count: a warp instruction of it holds
// the sub-partition for 64 clocks, whatever the number of active lanes.  So the
// relative positions come from pairs of floats (x = h + l to 48 bits; the
// difference rounds as the FP64 one does but for ties), fixed-point conversions go through
// 32-bit ones, and per-atom FP64 arithmetic is gathered into full warps and
// spends reciprocals and one short exponential in place of divisions and tanh.
// Operands, orders and sums of the pair passes are those of the ordered kernels
// with operands from the master arrays (k_born, k_gb, k_chain), and so are their
// roundings but for the argument of the salt factor (kappa / (1/f) here, kappa f^2 (1/f)
// there).
#pragma once
#include <cooperative_groups.h>

#include <algorithm>

#include "cph_device.cuh"
#include "cph_internal.h"
#include "cph_kernels.cuh"
#include "cph_shake_small.cuh"

namespace cph {

constexpr int kSmallAtoms = 512;  // atoms of a walker at most
constexpr int kSmallTerms = 1024; // bonded terms that touch a CTA's atoms at most
constexpr int kSmallAux = 2;      // extra warps per CTA
constexpr int kSmallRanks = 8;    // CTAs per cluster
// SHAKE tolerances from here on: the pairs of floats of small_shake leave up to
// 3e-14 of d0^2 (measured at a tolerance of 1e-14), so below that they settle late,
// never, or elsewhere.  Tighter ones take the separate launches (k_shake, FP64).
constexpr double kSmallShakeTol = 1e-12;
constexpr int kSmallUnroll = 2;   // of the partner loops (1 to 4: within 3 %)

// Whether walkers of at most n atoms (`atoms` in all) that fit the kernel also run
// in it, by the whole grid's numbers, so that every engine of a sharded grid decides
// alike.  A cluster holds eight SMs, so `resident` of them (15, of 40-atom walkers
// 32 and more) run at once and the others wait for the next wave; the separate
// launches take a walker's atoms four to a CTA over the whole chip, 2432 atoms at
// a time.  us a step of 100 with sweeps every 10, this kernel / separate launches:
//   atoms  1 walker   8 walkers  15         16         30         45         64
//     80   15 / 22    16 / 23    16 / 23    28 / 24    29 / 25    42 / 34    67 / 47
//    120   16 / 22    17 / 23    17 / 24    31 / 25    31 / 35    45 / 47    73 / 56
//    160   19 / 24    19 / 25    19 / 27    36 / 35    36 / 43    53 / 55    86 / 76
//    237   27 / 24    27 / 26    27 / 38    50 / 38    51 / 55    75 / 78    123 / 102
//    360   50 / 25    51 / 39    51 / 56    97 / 57    99 / 85    146 / 114  240 / 154
//    480   64 / 26    65 / 43    65 / 64    125 / 71   127 / 111  188 / 156  310 / 211
// The tiles of cph_sym.cuh never come near where this form pays (68 to 420).  With
// constraints, whose separate launches are slower (operands from the master arrays,
// SHAKE in a launch of its own):
//    121   27 / 57    28 / 63    28 / 68    52 / 68    53 / 79    77 / 97    126 / 115
//    205   36 / 63    36 / 71    37 / 83    70 / 83    70 / 114   104 / 142  170 / 175
//    246   37 / 64    37 / 74    37 / 89    70 / 89    71 / 132   106 / 160  173 / 201
//    351   59 / 68    59 / 84    60 / 119   114 / 127  116 / 177  172 / 235  284 / 310
//    452   75 / 70    76 / 100   76 / 154   147 / 157  149 / 244  221 / 334  364 / 450
// Over 595 points (1 to 200 walkers of 40 to 460 atoms) what runs is within 5 % of the
// best form but at six, most with a part-filled last wave, where it is 6 to 13 % behind.
inline bool small_pays(int n, long long atoms, int walkers, int resident, bool constrained) {
    const int waves = (walkers + resident - 1) / resident;
    if (constrained) return waves <= (n <= 100 ? 3 : (n <= 200 ? 4 : (n <= 256 ? 8 : (n <= 384 ? 5 : 4))));
    const long long other = (atoms + 2431) / 2432; // waves of the separate launches
    if (n <= 160) return waves <= std::min(other, 3ll);
    if (n <= 256) return waves <= (other >= 5 ? 3 : (other >= 3 ? 2 : (n <= 192 || atoms >= 1600 ? 1 : 0)));
    return n <= 384 && waves == 1 && other >= 3;
}

// phases of a step: where a launch starts its first step and ends its last
enum SmallPhase { kSmallBorn = 0, kSmallForces = 1, kSmallMove = 2 };

// Which bonded terms a CTA evaluates and which of them act on an atom; for
// every (system, rank) the bonds and then the angles among term[], and for every
// system atom its terms in the order of its lists (bonds, then angles) as
// place among its CTA's terms << 2 | the atom's place in the term
struct SmallTab {
    const int *term_off, *term; // [n_sys][ranks] (first bond, first angle, end), and the terms
    const int *ref_off, *ref;   // per system atom
    const int* ref_mid;         // where the atom's angles start
    const int* shk_sys_off;     // SHAKE clusters per system
    const float4* shk_fac;      // per hydrogen: 1/m of its heavy atom and its own over twice their sum, each h + l
    float2* rad;                // [total_atoms] (R, 1/R) as the pair sums read them
};

struct SmallRun {
    int w0;           // first walker of the launch
    int warps;        // pair warps per CTA
    int s_off, steps; // step *V.step + s_off first, this many steps
    int start, end;   // SmallPhase of the first step's start, and of the last step's end (its last phase)
    int zero_energy;
};

// a - b for a, b given as sums h + l of floats (48 bits), rounded to FP32
__device__ __forceinline__ float diff2(const float2& a, const float2& b) {
    const float s = __fsub_rn(a.x, b.x), t = __fsub_rn(s, a.x);
    const float e = __fsub_rn(__fsub_rn(a.x, __fsub_rn(s, t)), __fadd_rn(b.x, t));
    return __fadd_rn(s, __fadd_rn(e, __fsub_rn(a.y, b.y)));
}

// An atom's per-step FP64 state
struct SmallAtom {
    double rt, irt, irho, rho, q, psi, R, iR, dRdpsi;
    double im, sd; // Langevin factors: dt A / m and sqrt(2 g kB T A dt / m)
};

struct SmallSmem {
    float2* xf;    // [2][3N] positions as h + l, this step's and the next one's
    double* x;     // [2][3N] the same in FP64
    float4* gq;    // [N] (sqrt(k) q, R, 1/R, 0)
    float4* st;    // [N] (s, rt, sigma/2, sqrt(eps))
    float* c;      // [N] chain weights
    // of the CTA's own atoms (own = 4 groups per CTA)
    double* v;       // [3 own] velocities
    SmallAtom* at;   // [own]
    long long* sum;  // [own][8] sums over the partners: H | dE/dR, F (direct), energies
    long long* fc;   // [3 own] chain-rule force sums
    float* fb;       // [3 own] bonded forces
    float* z;        // [3 own] normal random numbers
    uint32_t* ex;    // [own][32] excluded partners
    float* rel;      // [own / 4][3][n] positions relative to the first atom of each group of four
    float* tf;       // [terms][8] bonded forces: bond g d; angle gi, gk, the factors of gk's z
    float* te;       // [terms] bonded energies
};

__host__ __device__ inline size_t small_bytes(int n, int own, int terms) {
    return (size_t)n * (2 * 24 + 2 * 24 + 16 + 16 + 4) + (n & 1) * 4 +
           (size_t)own * (24 + sizeof(SmallAtom) + 64 + 24 + 12 + 12 + 128) + (size_t)terms * 36 + (size_t)(own / 4) * 12 * n + 16;
}

__device__ __forceinline__ SmallSmem small_carve(unsigned char* p, int n, int own, int terms) {
    SmallSmem s;
    s.gq = (float4*)p;
    s.st = s.gq + n;
    s.xf = (float2*)(s.st + n);
    s.x = (double*)(s.xf + 6 * n);
    s.v = s.x + 6 * n;
    s.at = (SmallAtom*)(s.v + 3 * own);
    s.sum = (long long*)(s.at + own);
    s.fc = s.sum + 8 * own;
    s.c = (float*)(s.fc + 3 * own);
    s.fb = s.c + n;
    s.z = s.fb + 3 * own;
    s.ex = (uint32_t*)(s.z + 3 * own);
    s.tf = (float*)(s.ex + 32 * own);
    s.te = s.tf + 8 * terms;
    s.rel = s.te + terms;
    return s;
}

// GA: atoms per warp, 1, 2 or 4 for up to 160, 256 or 512 atoms.  The pair warps of a
// CTA then number at most 20, 16 and 16, and the launch bounds leave 80 to 96
// registers.  With one atom a warp up to 224 atoms (28 warps, 64 registers) 176
// atoms took 20.7 us a step for 21.9, 200 atoms 23.4 for 24.3, but 205 with
// constraints 37.2 for 35.8.
template <int GA, bool ENERGY>
__global__ void __launch_bounds__(GA == 1 ? 704 : 576, 1) k_small(View V, SmallTab T, SmallRun run) {
    pdl_sync();
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cl = cg::this_cluster();
    auto sync = [&] {
        __syncwarp();
        cl.sync();
    };
    constexpr int CS = kSmallRanks;
    const int rank = (int)cl.block_rank();
    const int w = run.w0 + (int)blockIdx.x / CS;
    if (!V.w_local[w]) return; // the whole cluster
    const int s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
    const int own = 4 * (((N + 3) / 4 + CS - 1) / CS), a0 = rank * own; // atoms per CTA, its first
    const int nown = min(own, max(0, N - a0));
    const int* toff = T.term_off + 3 * (s * CS + rank);
    const int nterm = toff[2] - toff[0], nbond = toff[1] - toff[0];
    const SmallSmem S = small_carve(smem_raw, N, own, nterm);
    const int npw = run.warps;                                  // pair warps
    const bool pairs = warp < npw && warp * GA < nown;
    const int i0 = a0 + warp * GA;                              // the warp's first atom
    const bool aux = warp >= npw;
    const int atid = tid - 32 * npw;                            // thread among the extra warps

    // ---- the walker's state into every CTA
    for (int k = tid; k < 3 * N; k += nthr) {
        const double x = V.x[3 * A + k];
        S.x[k] = x;
        S.xf[k] = split2(x);
    }
    const float sqk = (float)V.sqrt_k;
    for (int j = tid; j < N; j += nthr) {
        const float4 r = V.pb32[P + j];
        const float2 l = V.plj32[P + j];
        S.st[j] = make_float4(r.x, r.y, l.x, l.y);
        float2 R = make_float2(1.f, 1.f);
        if (run.start > kSmallBorn) R = T.rad[A + j];
        S.gq[j] = make_float4((float)V.q[A + j] * sqk, R.x, R.y, 0.f);
    }
    for (int k = tid; k < 3 * nown; k += nthr) S.v[k] = V.v[3 * (A + a0) + k];
    for (int a = tid; a < nown; a += nthr) {
        const int i = a0 + a;
        SmallAtom& at = S.at[a];
        at.rt = V.rt[P + i];
        at.irt = V.irt[P + i];
        at.irho = V.irho[P + i];
        at.rho = V.rho[P + i];
        at.q = V.q[A + i] * V.sqrt_k;
        at.psi = V.psi[A + i];
        at.R = V.R[A + i];
        at.iR = run.start > kSmallBorn ? rcp64_radius(at.R) : 1.0;
        at.dRdpsi = V.dRdpsi[A + i];
        at.im = V.lg_im[P + i];
        at.sd = V.lg_sqT[V.slot_of[w] / (V.nE * V.npH)] * V.lg_sf[P + i];
    }
    // excluded partners (and itself): bit m of lane j & 31
    for (int a = warp; a < nown; a += nthr / 32) {
        const int i = a0 + a;
        uint32_t ex = (i & 31) == lane ? 1u << (i >> 5) : 0u;
        for (int e = V.excl_off[P + i]; e < V.excl_off[P + i + 1]; ++e) {
            const int j = V.excl_j[e];
            if ((j & 31) == lane) ex |= 1u << (j >> 5);
        }
        S.ex[32 * a + lane] = ex;
    }
    double vs = run.start == kSmallMove ? V.vscale[w] : 1.0;
    if (run.zero_energy && rank == 0 && tid < kEAcc) V.eacc[w * kEAcc + tid] = 0;
    const float rc = (float)V.rgbmax, tau = V.tau32, iei = V.iei32, kap = V.kappa32, ieo = V.ieo32;
    const bool salt = V.kappa > 0;
    const uint64_t t0 = (uint64_t)(*V.step + run.s_off);
    int cur = 0, moved = 0;
    sync();

    for (int st = 0; st < run.steps; ++st) {
        const bool first = st == 0, last = st + 1 == run.steps;
        const bool forces = !(first && run.start == kSmallMove);
        if (forces) {
            // positions relative to the first atom of each group of four
            for (int g = 0; g < (nown + 3) / 4; ++g) {
                const float2 *X = S.xf + 3 * N * cur, *C = X + 3 * (a0 + 4 * g);
                float* rel = S.rel + 3 * N * g;
                for (int j = tid; j < N; j += nthr) {
                    rel[j] = diff2(X[3 * j], C[0]);
                    rel[N + j] = diff2(X[3 * j + 1], C[1]);
                    rel[2 * N + j] = diff2(X[3 * j + 2], C[2]);
                }
            }
            __syncthreads();
            // ---- Born radii; meanwhile the bonded terms and the random numbers
            if (!(first && run.start > kSmallBorn)) {
                if (pairs) {
#pragma unroll 1
                    for (int a = 0; a < GA; ++a) {
                        const int i = min(i0 + a, N - 1);
                        const float* rel = S.rel + 3 * N * ((warp * GA + a) / 4);
                        const float qx = rel[i], qy = rel[N + i], qz = rel[2 * N + i];
                        const float rti = S.st[i].y, irti = 1.f / rti;
                        long long acc = 0;
                        for (int j0 = lane; j0 < N; j0 += 128) { // a tile of 128 partners, four a lane
                            float part = 0.f;
#pragma unroll kSmallUnroll
                            for (int k = 0; k < 4; ++k) {
                                const int j = j0 + 32 * k;
                                if (j >= N) break;
                                const bool self = j == i;
                                const float dx = qx - rel[j], dy = qy - rel[N + j], dz = qz - rel[2 * N + j];
                                float r2 = dx * dx + dy * dy + dz * dz;
                                r2 = self ? 1.f : r2;
                                const float rinv = rsqrtf(r2);
                                const float h = hct(r2 * rinv, rinv, rti, irti, S.st[j].x, rc);
                                part += self ? 0.f : h;
                            }
                            acc += fix32(part * 256.f); // 2^40
                        }
                        acc = warp_sum(acc);
                        if (lane == 0 && i0 + a < N) S.sum[8 * (warp * GA + a)] = acc;
                    }
                }
            }
            if (aux) {
                const double* x = (S.x + 3 * N * cur);
                for (int t = atid; t < nterm; t += 32 * kSmallAux) {
                    const int k = T.term[toff[0] + t];
                    float* f = S.tf + 8 * t;
                    if (t < nbond) {
                        const int i = V.bond_ij[2 * k], j = V.bond_ij[2 * k + 1];
                        double d[3];
                        for (int c = 0; c < 3; ++c) d[c] = x[3 * i + c] - x[3 * j + c];
                        float g, en;
                        bond_term32(d, V.bond_r0[k], V.bond_k[k], g, en);
                        for (int c = 0; c < 3; ++c) f[c] = g * (float)d[c];
                        S.te[t] = en;
                    } else {
                        const int i = V.ang_ijk[3 * k], j = V.ang_ijk[3 * k + 1], l = V.ang_ijk[3 * k + 2];
                        double u[3], v[3];
                        for (int c = 0; c < 3; ++c) {
                            u[c] = x[3 * i + c] - x[3 * j + c];
                            v[c] = x[3 * l + c] - x[3 * j + c];
                        }
                        float gi[3], gk[3], en;
                        float2 kz;
                        angle_term32(u, v, V.ang_cs0[k], V.ang_k[k], gi, gk, kz, en);
                        f[6] = kz.x;
                        f[7] = kz.y;
                        for (int c = 0; c < 3; ++c) {
                            f[c] = gi[c];
                            f[3 + c] = gk[c];
                        }
                        S.te[t] = en;
                    }
                }
            }
            __syncthreads();
            if (!(first && run.start > kSmallBorn)) {
                for (int a = tid; a < nown; a += nthr) { // R and dR/dpsi, to every CTA
                    SmallAtom& at = S.at[a];
                    const double psi = at.rt * ((double)S.sum[8 * a] * (0.5 / kScaleH));
                    const double th = tanh64(psi * (V.alpha + psi * (-V.beta + psi * V.gamma)));
                    const double iR = at.irt - th * at.irho, R = rcp64_radius(iR);
                    at.psi = psi;
                    at.R = R;
                    at.iR = iR;
                    at.dRdpsi = R * R * (1.0 - th * th) *
                                (V.alpha + psi * (-2.0 * V.beta + 3.0 * V.gamma * psi)) * at.irho;
                    const float Rf = pair_radius32(R), iRf = (float)iR;
#pragma unroll
                    for (int r = 0; r < CS; ++r) {
                        float4* o = cl.map_shared_rank(S.gq, r) + a0 + a;
                        o->y = Rf;
                        o->z = iRf;
                    }
                }
            }
            if (last && run.end == kSmallBorn) break;
            sync(); // radii
            // ---- GB + Coulomb + LJ; meanwhile each atom's bonded forces
            if (pairs) {
#pragma unroll 1
                for (int a = 0; a < GA; ++a) {
                    const int i = min(i0 + a, N - 1);
                    const float* rel = S.rel + 3 * N * ((warp * GA + a) / 4);
                    const float qx = rel[i], qy = rel[N + i], qz = rel[2 * N + i];
                    const uint32_t ex = S.ex[32 * min(warp * GA + a, own - 1) + lane];
                    const float4 gi = S.gq[i], si = S.st[i];
                    const float qi = gi.x, Ri = gi.y, iRi = gi.z, sgi = si.z, sei = si.w;
                    long long fx = 0, fy = 0, fz = 0, ar = 0, e0 = 0, e1 = 0, e2 = 0;
                    auto sweep = [&](auto with_salt) {
                        constexpr bool SALT = decltype(with_salt)::value;
                        for (int j0 = lane, m = 0; j0 < N; j0 += 128, m += 4) {
                            float ax = 0.f, ay = 0.f, az = 0.f, adx = 0.f;
                            KSum<float> pgb, pc, plj;
#pragma unroll kSmallUnroll
                            for (int k = 0; k < 4; ++k) {
                                const int j = j0 + 32 * k;
                                if (j >= N) break;
                                const bool self = j == i;
                                const float4 b = S.gq[j], sj = S.st[j];
                                const float dx = qx - rel[j], dy = qy - rel[N + j], dz = qz - rel[2 * N + j];
                                float r2 = dx * dx + dy * dy + dz * dz;
                                r2 = self ? 1.f : r2;
                                const float g = self ? 0.f : 1.f, nb = (ex >> (m + k)) & 1u ? 0.f : 1.f;
                                const float rinv = rsqrtf(r2), rinv2 = rinv * rinv;
                                const float qq = qi * b.x;
                                const float D = 0.25f * r2 * (iRi * b.z);
                                const float e = __expf(-D);
                                const float fi = rsqrtf(r2 + (Ri * b.y) * e);
                                const float qf3 = g * qq * fi * fi * fi;
                                float tf = 1.f, td = 1.f;
                                if (SALT) {
                                    const float es = ieo * __expf(-(kap / fi));
                                    tf = iei - es;
                                    td = tf - kap * es / fi;
                                }
                                adx += td * qf3 * b.y * e * (1.f + D);
                                const float sig = sgi + sj.z;
                                const float sr2 = sig * sig * rinv2;
                                const float sr6 = sr2 * sr2 * sr2;
                                const float ep = nb * sei * sj.w;
                                const float fs = nb * iei * qq * rinv * rinv2 + 4.f * ep * sr6 * (12.f * sr6 - 6.f) * rinv2 -
                                                 (SALT ? td : tau) * qf3 * (1.f - 0.25f * e);
                                ax += fs * dx;
                                ay += fs * dy;
                                az += fs * dz;
                                if (ENERGY) {
                                    pgb.add(tf * g * qq * fi);
                                    pc.add(nb * qq * rinv);
                                    plj.add(ep * sr6 * (sr6 - 1.f));
                                }
                            }
                            fx += fix32(ax);
                            fy += fix32(ay);
                            fz += fix32(az);
                            ar += fix32(adx);
                            if (ENERGY) {
                                e0 += fix32(pgb.value());
                                e1 += fix32(pc.value());
                                e2 += fix32(plj.value());
                            }
                        }
                    };
                    if (salt) sweep(std::true_type{});
                    else sweep(std::false_type{});
                    fx = warp_sum(fx);
                    fy = warp_sum(fy);
                    fz = warp_sum(fz);
                    ar = warp_sum(ar);
                    if (ENERGY) {
                        e0 = warp_sum(e0);
                        e1 = warp_sum(e1);
                        e2 = warp_sum(e2);
                    }
                    if (lane == 0 && i0 + a < N) {
                        long long* o = S.sum + 8 * (warp * GA + a);
                        o[0] = ar;
                        o[1] = fx;
                        o[2] = fy;
                        o[3] = fz;
                        if (ENERGY) {
                            o[4] = e0;
                            o[5] = e1;
                            o[6] = e2;
                        }
                    }
                }
            }
            if (aux) {
                // an atom's bonded terms over eight lanes, in the order of its lists
                long long s0 = 0, s1 = 0;
                for (int a8 = atid; a8 < 8 * ((nown + 3) & ~3); a8 += 32 * kSmallAux) { // whole warps
                    const int a = a8 >> 3, l8 = a8 & 7;
                    float fb[3] = {0.f, 0.f, 0.f}, eb = 0.f, ea = 0.f;
                    if (a < nown) {
                        const int p = P + a0 + a, r0 = T.ref_off[p], rm = T.ref_mid[p], r1 = T.ref_off[p + 1];
                        for (int e = r0 + l8; e < rm; e += 8) {
                            const int k = T.ref[e], t = k >> 2;
                            const float sg = (k & 3) ? 1.f : -1.f;
                            for (int c = 0; c < 3; ++c) fb[c] += sg * S.tf[8 * t + c];
                            if ((k & 3) == 0) eb += S.te[t];
                        }
                        for (int e = rm + l8; e < r1; e += 8) {
                            const int k = T.ref[e], t = k >> 2, role = k & 3;
                            const float* f = S.tf + 8 * t;
                            // (z rounds gk's product and its sum at once, as the one-lane-a-term
                            // sums of the ordered kernel do: constrained trajectories follow
                            // every rounding, see cph_engine::staged)
                            for (int c = 0; c < 3; ++c) {
                                if (role == 0) fb[c] -= f[c];
                                else if (role == 2) fb[c] = c == 2 && e < rm + 8 ? fmaf(-f[6], f[7], fb[2]) : fb[c] - f[3 + c];
                                else fb[c] += c == 2 ? fmaf(f[6], f[7], f[2]) : f[c] + f[3 + c];
                            }
                            if (role == 0) ea += S.te[t];
                        }
                    }
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) fb[c] += __shfl_down_sync(0xffffffffu, fb[c], o, 8);
                        if (ENERGY) {
                            eb += __shfl_down_sync(0xffffffffu, eb, o, 8);
                            ea += __shfl_down_sync(0xffffffffu, ea, o, 8);
                        }
                    }
                    if (l8 == 0 && a < nown) {
                        for (int c = 0; c < 3; ++c) S.fb[3 * a + c] = fb[c];
                        if (ENERGY) {
                            s0 += __double2ll_rn((double)eb * kScaleE);
                            s1 += __double2ll_rn((double)ea * kScaleE);
                        }
                    }
                }
                if (ENERGY) {
                    s0 = warp_sum(s0);
                    s1 = warp_sum(s1);
                    if (lane < 2) atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 3 + lane], (unsigned long long)(lane ? s1 : s0));
                }
            }
            __syncthreads();
            for (int a = tid; a < nown; a += nthr) { // chain weights, to every CTA
                const SmallAtom& at = S.at[a];
                const long long* o = S.sum + 8 * a;
                const double qR = at.q * at.iR;
                double taud = V.inv_eps_in - V.inv_eps_out, ts = taud;
                if (salt) {
                    taud = salt_taud(at.R, V.inv_eps_in, V.inv_eps_out, V.kappa);
                    ts = salt_tau(at.R, V.inv_eps_in, V.inv_eps_out, V.kappa);
                }
                double dEdR = 0.5 * (V.tau_pair * ((double)o[0] * (1.0 / kScaleE)) + taud * qR * qR);
                double esa = 0.0;
                if (V.sa_gamma != 0.0) {
                    esa = sa_ace(V.sa_gamma, V.sa_probe, at.rho, at.R);
                    dEdR -= 6.0 * esa * at.iR;
                }
                const double c = dEdR * at.dRdpsi * (0.5 * at.rt);
                const float cf = (float)c;
#pragma unroll
                for (int r = 0; r < CS; ++r) cl.map_shared_rank(S.c, r)[a0 + a] = cf;
                if (last) V.c[A + a0 + a] = c;
                if (ENERGY) {
                    const long long b0 = __double2ll_rn((-0.5 * (V.tau_pair * ((double)o[4] / kScaleE) + ts * at.q * qR) + esa) * kScaleE);
                    const long long b1 = __double2ll_rn(0.5 * V.inv_eps_in * ((double)o[5] / kScaleE) * kScaleE);
                    const long long b2 = __double2ll_rn(2.0 * ((double)o[6] / kScaleE) * kScaleE);
                    atomicAdd((unsigned long long*)&V.eacc[w * kEAcc], (unsigned long long)b0);
                    atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 1], (unsigned long long)b1);
                    atomicAdd((unsigned long long*)&V.eacc[w * kEAcc + 2], (unsigned long long)b2);
                }
            }
            sync(); // chain weights
            // ---- chain rule; meanwhile the random numbers of the move
            if (pairs) {
#pragma unroll 1
                for (int a = 0; a < GA; ++a) {
                    const int i = min(i0 + a, N - 1);
                    const float* rel = S.rel + 3 * N * ((warp * GA + a) / 4);
                    const float qx = rel[i], qy = rel[N + i], qz = rel[2 * N + i];
                    const float ci = S.c[i], si = S.st[i].x, rti = S.st[i].y;
                    long long fx = 0, fy = 0, fz = 0;
                    for (int j0 = lane; j0 < N; j0 += 128) {
                        float ax = 0.f, ay = 0.f, az = 0.f;
#pragma unroll kSmallUnroll
                        for (int k = 0; k < 4; ++k) {
                            const int j = j0 + 32 * k;
                            if (j >= N) break;
                            const bool self = j == i;
                            const float4 sj = S.st[j];
                            const float dx = qx - rel[j], dy = qy - rel[N + j], dz = qz - rel[2 * N + j];
                            float r2 = dx * dx + dy * dy + dz * dz;
                            r2 = self ? 1.f : r2;
                            const float rinv = rsqrtf(r2), r = r2 * rinv;
                            const float g = ci * hct_dr(r, rinv, rti, sj.x, rc) + S.c[j] * hct_dr(r, rinv, sj.y, si, rc);
                            const float t = self ? 0.f : -g * rinv;
                            ax += t * dx;
                            ay += t * dy;
                            az += t * dz;
                        }
                        fx += fix32(ax);
                        fy += fix32(ay);
                        fz += fix32(az);
                    }
                    fx = warp_sum(fx);
                    fy = warp_sum(fy);
                    fz = warp_sum(fz);
                    if (lane == 0 && i0 + a < N) {
                        long long* o = S.fc + 3 * (warp * GA + a);
                        o[0] = fx;
                        o[1] = fy;
                        o[2] = fz;
                    }
                }
            }
        }
        if (aux) {
            for (int a = atid; a < nown; a += 32 * kSmallAux) {
                float z[3];
                normals3(V.seed, (uint32_t)(a0 + a), (uint32_t)w, t0 + (uint64_t)st, z);
                for (int c = 0; c < 3; ++c) S.z[3 * a + c] = z[c];
            }
        }
        __syncthreads();
        // ---- total force; Langevin step (k_langevin), a component per thread
        const int nxt = cur ^ 1;
        const bool move = !(last && run.end == kSmallForces);
        for (int k = tid; k < 3 * nown; k += nthr) {
            const int a = k / 3, g = 3 * (A + a0) + k;
            double F;
            if (forces) {
                F = fma((double)(S.sum[8 * a + 1 + (k - 3 * a)] + S.fc[k]), 1.0 / kScaleE, (double)S.fb[k]);
                if (!isfinite(F)) atomicOr(V.status, 1);
            } else F = V.F[g];
            if (last && forces) V.F[g] = F;
            if (!move) continue;
            const double vn = (V.lg_c1 * (S.v[k] * vs) + S.at[a].im * F + S.at[a].sd * (double)S.z[k]) * V.lg_c2;
            S.v[k] = vn;
            const double xn = (S.x + 3 * N * cur)[3 * a0 + k] + V.dt * vn;
            if (!isfinite(xn)) atomicOr(V.status, 2);
            const float2 xf = split2(xn);
#pragma unroll
            for (int r = 0; r < CS; ++r) {
                cl.map_shared_rank(S.x + 3 * N * nxt, r)[3 * a0 + k] = xn;
                cl.map_shared_rank(S.xf + 3 * N * nxt, r)[3 * a0 + k] = xf;
            }
        }
        if (!move) break;
        vs = 1.0;
        ++moved;
        sync(); // positions
        if (V.xprev) {
            const double idt = 1.0 / V.dt;
            const int c0 = T.shk_sys_off[s], nc = T.shk_sys_off[s + 1] - c0;
            // this CTA's share of the clusters, eight to a warp
            const int ncl = rank < nc ? (nc - rank + CS - 1) / CS : 0, d = lane & 3;
            double* xt = S.x + 3 * N * nxt;
            auto shake = [&](auto nh_max, int c, bool on, int nh) {
                constexpr int NH = decltype(nh_max)::value;
                double u[NH + 1];
                small_shake<NH>(V, T.shk_fac, c, on, d, S.x + 3 * N * cur, xt, nh, u);
                if (!on || d == 3) return;
                const int h0 = V.shk_off[c];
#pragma unroll
                for (int h = 0; h <= NH; ++h) {
                    if (h > nh) break;
                    const int at = h == 0 ? V.shk_heavy[c] : V.shk_h[h0 + h - 1], owner = at / own;
                    const double x1 = xt[3 * at + d] + u[h];
                    cl.map_shared_rank(S.v, owner)[3 * (at - owner * own) + d] += u[h] * idt;
                    const float2 xf = split2(x1);
#pragma unroll
                    for (int r = 0; r < CS; ++r) {
                        cl.map_shared_rank(S.x + 3 * N * nxt, r)[3 * at + d] = x1;
                        cl.map_shared_rank(S.xf + 3 * N * nxt, r)[3 * at + d] = xf;
                    }
                }
            };
            for (int k0 = 8 * warp; k0 < ncl; k0 += nthr / 4) { // whole warps
                const int k = k0 + (lane >> 2);
                const bool on = k < ncl;
                const int c = c0 + rank + CS * min(k, ncl - 1), nh = on ? V.shk_off[c + 1] - V.shk_off[c] : 0;
                if (__reduce_max_sync(0xffffffffu, nh) <= 3) shake(std::integral_constant<int, 3>{}, c, on, nh);
                else shake(std::integral_constant<int, kShakeMaxH>{}, c, on, nh);
            }
            sync();
        }
        cur = nxt;
    }

    // ---- state out
    __syncthreads();
    for (int a = tid; a < nown; a += nthr) {
        const SmallAtom& at = S.at[a];
        const int g = A + a0 + a;
        V.psi[g] = at.psi;
        V.R[g] = at.R;
        V.dRdpsi[g] = at.dRdpsi;
        V.gq[g] = gb_operand(V.q[g], V.sqrt_k, at.R);
        T.rad[g] = make_float2(pair_radius32(at.R), (float)at.iR);
    }
    for (int k = tid; k < 3 * nown; k += nthr) {
        const int g = 3 * (A + a0) + k, a = k / 3, d = k - 3 * a;
        const double x = (S.x + 3 * N * cur)[3 * a0 + k];
        if (moved) {
            V.x[g] = x;
            V.v[g] = S.v[k];
        }
        // a sweep reads them after the Born phase
        reinterpret_cast<float*>(&V.xs[A + a0 + a])[d] = (float)(x - (S.x + 3 * N * cur)[d]);
    }
    if (moved && rank == 0) { // observables: slots and states do not change within a launch
        const int slot = V.slot_of[w];
        if (tid == 0) {
            V.visits[(long long)w * V.W + slot] += moved;
            if (w == V.first_local) *V.n_obs += moved;
        }
        const int ws0 = V.w_site_off[w], nst = V.w_site_off[w + 1] - ws0;
        const long long row0 = V.w_site_off[slot];
        for (int k = tid; k < nst; k += nthr) V.occ[(row0 + k) * CPH_MAX_STATES + V.site_state[ws0 + k]] += moved;
    }
    // the pending velocity scale ends with the next Born phase, as in k_born
    if (rank == 0 && tid == 0 && (run.start != kSmallMove || run.steps > 1)) V.vscale[w] = 1.0;
    sync(); // no CTA leaves while another may still write to it
}

} // namespace cph
