// The FP32 pair passes over every ordered pair: one warp per atom, four atoms per
// CTA, operands from the arrays staged once per step (FP64 differences, divisions
// and conversions hold a sub-partition's FP64 pipe for 64 clocks each).  They
// serve systems with too few atoms in flight for the tile passes of cph_sym.cuh.
//
// One walker of 2003 atoms gives a sub-partition three warps, so instructions and
// latency are what they take.  A lane meets a partner once, so nothing is staged in
// shared memory: 128 partners at a time (four a lane) come straight into registers,
// the L1 cache serving the CTA's other warps and the SM's other CTAs, and no
// barrier stands in the loop; two partners' values make the halves of the float2
// instructions; near pairs wait in a queue.  The Born pass reads a batch ahead
// (21.7 -> 17.4 us); for the chain rule that costs more registers than it hides
// (20.5 -> 24.2).  Against tiles of partners in shared memory, scalar arithmetic and
// closed forms inside the loop: 1 x 2003 atoms 25.9 -> 17.4, 22.8 -> 18.7 and
// 28.7 -> 20.5 us (Born radii, pair pass, chain rule); 8 x 1203 atoms with salt and a
// cutoff of 12 A, energies, 41.8 -> 37.5, 49.7 -> 43.2 and 59.5 -> 55.2 us (half of
// their pairs within reach lie in the cutoff's band of closed forms).  These without
// the positions' low words (Place), which cost 8 %: 20 steps of 1 x 2003 atoms
// 1.13 -> 1.21 ms, 8 x 1203 atoms 212 -> 227 us.
#pragma once
#include "cph_kernels.cuh"
#include "cph_pair_tiles.cuh"

namespace cph {

constexpr int kBatch = 4;            // partners of a lane at a time, in float2 pairs
// partners summed in FP32 before a conversion to fixed point (with 128: forces of 2003
// atoms 4.70e-7 instead of 4.72e-7 from FP64's, radii the same, 20 steps 1.21 -> 1.30 ms)
constexpr int kOrdFlush = 8 * kTile;

// Near pairs.  A warp step that meets one would run
// the closed forms for all its lanes, in the middle of the pair loop, and 20 to
// 50 % of the steps do.  So the loop runs the far form for every pair and queues
// what a near pair needs; the warp evaluates 32 of them at once, one a lane, while
// it holds that many.  All pairs of a warp belong to its atom: nothing is scattered.
constexpr int kOrdQueue = 32 + 32 * kBatch; // fewer than 32 wait, a batch adds at most 128

template <class Entry>
struct NearQueue {
    Entry* q; // kOrdQueue per warp
    int n = 0;
    __device__ __forceinline__ explicit NearQueue(Entry* warp_queue) : q(warp_queue) {}
    __device__ __forceinline__ void push(bool near, const Entry& e, int lane) {
        const uint32_t bal = __ballot_sync(0xffffffffu, near);
        if (near) q[n + __popc(bal & ((1u << lane) - 1u))] = e;
        n += __popc(bal);
    }
    template <class F>
    __device__ __forceinline__ void drain(int lane, F&& eval) {
        __syncwarp();
        while (n >= 32) {
            n -= 32;
            eval(q[n + lane]);
        }
        __syncwarp();
    }
    template <class F>
    __device__ __forceinline__ void finish(int lane, F&& eval) {
        if (lane < n) eval(q[lane]);
    }
};

__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// An atom's place: its position relative to the walker's first atom as h + l, and
// its s and rt.  The separation of two atoms is then rounded to FP32 once, however
// far from that first atom they are; h alone leaves 4e-6 A of error at 40 A in the
// separation of neighbours (extended chains of 600 to 3000 atoms: Born radii off by
// 4e-6 to 2e-5 relative, with l 2e-7).
struct Place {
    float4 h, l; // (x, y, z, s), (x, y, z, rt)
};
__device__ __forceinline__ Place place(const View& V, int a) { return {V.xs[a], V.xl[a]}; }
// in place of an atom i, and of a partner, that does not exist: no pair of theirs counts
__device__ __forceinline__ Place far_place() {
    return {make_float4(-kFarF, -kFarF, -kFarF, 0.f), make_float4(0.f, 0.f, 0.f, 1.f)};
}
__device__ __forceinline__ Place no_place() {
    return {make_float4(kFarF, kFarF, kFarF, 0.f), make_float4(0.f, 0.f, 0.f, 1.f)};
}
__device__ __forceinline__ void separation(const Place& i, const Place& a, const Place& b, float2& dx, float2& dy,
                                           float2& dz) {
    auto one = [](float hi, float li, float ha, float la, float hb, float lb) {
        return __fadd2_rn(sub2(splat<float2>(hi), make_float2(ha, hb)), sub2(splat<float2>(li), make_float2(la, lb)));
    };
    dx = one(i.h.x, i.l.x, a.h.x, a.l.x, b.h.x, b.l.x);
    dy = one(i.h.y, i.l.y, a.h.y, a.l.y, b.h.y, b.l.y);
    dz = one(i.h.z, i.l.z, a.h.z, a.l.z, b.h.z, b.l.z);
}

// ------------------------------------------------------------- pass 1: Born radii
// CUT: with a Born-radius cutoff
template <bool CUT>
__global__ void __launch_bounds__(kTile) k_born32(const Item* __restrict__ items, View V, int zero_energy) {
    pdl_sync();
    using Pr = Prec<float>;
    __shared__ AtomSums<1> sums;
    __shared__ float2 sq[kWarpAtoms][kOrdQueue];
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31;
    const int i = it.i0 + (tid >> 5);
    if (it.i0 == 0) {
        if (zero_energy && tid < kEAcc) V.eacc[w * kEAcc + tid] = 0;
        if (tid == kEAcc) V.vscale[w] = 1.0;
    }
    Place me = far_place();
    if (i < N) me = place(V, A + i);
    const float rti = me.l.w;
    const PairBand band = pair_band(V.rfar2, V.smax32, (float)V.rgbmax);
    const float irti = 1.f / rti;
    long long acc = 0;
    float2 far = splat<float2>(0.f);
    float part = 0.f;
    NearQueue<float2> near_q(sq[tid >> 5]); // (r^2, s_j)
    auto closed = [&](float2 e) {
        const float rinv = Pr::rsqrt(e.x);
        part += hct(e.x * rinv, rinv, rti, irti, e.y, band.rc);
    };
    auto load = [&](Place (&p)[kBatch], int j0) {
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int j = j0 + 32 * u + lane;
            p[u] = no_place();
            if (j < N) p[u] = place(V, A + j);
        }
    };
    auto work = [&](const Place (&p)[kBatch], int j0) {
        float2 e[kBatch];
        bool near[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; u += 2) {
            float2 dx, dy, dz;
            separation(me, p[u], p[u + 1], dx, dy, dz);
            const float2 sj = make_float2(p[u].h.w, p[u + 1].h.w), s2 = __fmul2_rn(sj, sj);
            float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            e[u] = make_float2(r2.x, sj.x);
            e[u + 1] = make_float2(r2.y, sj.y);
            near[u] = band_near<CUT>(r2.x, band);
            near[u + 1] = band_near<CUT>(r2.y, band);
            r2.x = near[u] ? INFINITY : r2.x; // where the far form is 0
            r2.y = near[u + 1] ? INFINITY : r2.y;
            near[u] = near[u] && j0 + 32 * u + lane != i;
            near[u + 1] = near[u + 1] && j0 + 32 * u + 32 + lane != i;
            const float2 rinv = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)), rinv2 = __fmul2_rn(rinv, rinv);
            float2 wt = __fmul2_rn(rinv2, rinv2);
            if (CUT) { // beyond rc + s_max nothing descreens
                wt.x = r2.x >= band.rout2 ? 0.f : wt.x;
                wt.y = r2.y >= band.rout2 ? 0.f : wt.y;
            }
            const float2 h = __fmul2_rn(hct_series_h(__fmul2_rn(s2, rinv2)), __fmul2_rn(s2, sj));
            far = __ffma2_rn(h, wt, far);
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) near_q.push(near[u], e[u], lane);
        near_q.drain(lane, closed);
        if ((j0 & (kOrdFlush - 1)) == kOrdFlush - kTile) {
            Pr::add(acc, part + (far.x + far.y), (float)kScaleH);
            part = 0.f;
            far = splat<float2>(0.f);
        }
    };
    Place pa[kBatch], pb[kBatch];
    load(pa, 0);
    for (int j0 = 0; j0 < N; j0 += 2 * kTile) {
        load(pb, j0 + kTile);
        work(pa, j0);
        if (j0 + kTile >= N) break;
        load(pa, j0 + 2 * kTile);
        work(pb, j0 + kTile);
    }
    near_q.finish(lane, closed);
    Pr::add(acc, part + (far.x + far.y), (float)kScaleH);
    const bool own = tid < kWarpAtoms && it.i0 + tid < N;
    const BornIn in = own ? BornIn(V, A, P, it.i0 + tid) : BornIn();
    sums.collect({acc});
    if (own) born_epilogue(V, A, P, it.i0 + tid, sums.v[0][tid], in);
}

// ------------------------------------------- pass 2: GB + Coulomb + LJ pair pass
template <bool ENERGY, bool SALT>
__global__ void __launch_bounds__(kTile) k_gb32(const Item* __restrict__ items, View V) {
    pdl_sync();
    using Pr = Prec<float>;
    __shared__ AtomSums<ENERGY ? 7 : 4> sums;
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31;
    const int i = it.i0 + (tid >> 5);
    Place me = far_place();
    float4 gi = make_float4(0.f, 1.f, 1.f, 0.f);
    float2 li = make_float2(0.f, 0.f);
    if (i < N) {
        me = place(V, A + i);
        gi = V.gq[A + i];
        li = V.plj32[P + i];
    }
    const float tau = V.tau32, iei = V.iei32, kap = V.kappa32, ieo = V.ieo32;
    long long fx = 0, fy = 0, fz = 0, adr = 0, egb = 0, ec = 0, elj = 0;
    const float2 one = splat<float2>(1.f), zero = splat<float2>(0.f);
    float2 px = zero, py = zero, pz = zero, pdr = zero;
    KSum<float2> pgb, pc, plj;
    struct Partner {
        Place x;
        float4 g; // sqrt(k) q, R, 1/R, log2(e) / (4 R)
        float2 l; // sigma / 2, sqrt(eps)
    };
    // two partners; bits 0, 1 of self: no pair, of ex: GB only
    auto pair = [&](const Partner& a, const Partner& b, uint32_t self, uint32_t ex) {
        float2 dx, dy, dz;
        separation(me, a.x, b.x, dx, dy, dz);
        float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        float2 qq = __fmul2_rn(splat<float2>(gi.x), make_float2(a.g.x, b.g.x));
        float2 ep = __fmul2_rn(splat<float2>(li.y), make_float2(a.l.y, b.l.y));
        if (self) {
            if (self & 1u) r2.x = 1.f, qq.x = 0.f;
            if (self & 2u) r2.y = 1.f, qq.y = 0.f;
        }
        float2 qc = qq;
        if (ex) {
            if (ex & 1u) ep.x = qc.x = 0.f;
            if (ex & 2u) ep.y = qc.y = 0.f;
        }
        const float2 Rj = make_float2(a.g.y, b.g.y);
        const float2 rinv = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y)), rinv2 = __fmul2_rn(rinv, rinv);
        const float2 D2 = __fmul2_rn(r2, __fmul2_rn(splat<float2>(gi.w), make_float2(a.g.z, b.g.z))); // D log2(e)
        const float2 e = make_float2(exp2_ftz(-D2.x), exp2_ftz(-D2.y));
        const float2 f2 = __ffma2_rn(__fmul2_rn(splat<float2>(gi.y), Rj), e, r2);
        const float2 fi = make_float2(rsqrt_ftz(f2.x), rsqrt_ftz(f2.y));
        const float2 qf3 = __fmul2_rn(qq, __fmul2_rn(__fmul2_rn(fi, fi), fi)), qfe = __fmul2_rn(qf3, e);
        float2 tf = one, td = one; // else the pair sums' common factor tau
        if (SALT) {
            const float2 kf = __fmul2_rn(splat<float2>(kap), __fmul2_rn(f2, fi));
            const float2 es = __fmul2_rn(splat<float2>(ieo),
                                         make_float2(exp2_ftz(-kLog2e * kf.x), exp2_ftz(-kLog2e * kf.y)));
            tf = sub2(splat<float2>(iei), es);
            td = sub2(tf, __fmul2_rn(kf, es));
        }
        float2 d = __fmul2_rn(__fmul2_rn(qfe, Rj), __ffma2_rn(D2, splat<float2>(kLn2), one));
        if (SALT) pdr = __ffma2_rn(d, td, pdr);
        else pdr = __fadd2_rn(d, pdr);
        const float2 sig = __fadd2_rn(splat<float2>(li.x), make_float2(a.l.x, b.l.x));
        const float2 sr2 = __fmul2_rn(__fmul2_rn(sig, sig), rinv2);
        const float2 sr6 = __fmul2_rn(__fmul2_rn(sr2, sr2), sr2);
        const float2 l6 = __fmul2_rn(ep, sr6);
        const float2 lj = __fmul2_rn(l6, __ffma2_rn(splat<float2>(48.f), sr6, splat<float2>(-24.f)));
        // -tau qf3 (1 - e/4); with salt taud(f) in place of tau
        const float2 gb = __fmul2_rn(SALT ? td : splat<float2>(tau), __ffma2_rn(splat<float2>(0.25f), qfe, sub2(zero, qf3)));
        const float2 fs = __ffma2_rn(__ffma2_rn(__fmul2_rn(splat<float2>(iei), qc), rinv, lj), rinv2, gb);
        px = __ffma2_rn(fs, dx, px);
        py = __ffma2_rn(fs, dy, py);
        pz = __ffma2_rn(fs, dz, pz);
        if (ENERGY) {
            pgb.add(SALT ? __fmul2_rn(tf, __fmul2_rn(qq, fi)) : __fmul2_rn(qq, fi));
            pc.add(__fmul2_rn(qc, rinv));
            plj.add(__fmul2_rn(l6, __fadd2_rn(sr6, splat<float2>(-1.f))));
        }
    };
    int mp = V.mt_off[it.st];
    const int mend = V.mt_off[it.st + 1];
    int next = mp < mend ? V.mt_list[mp] : 0x7fffffff;
    for (int j0 = 0, jt = 0; j0 < N; j0 += kTile, ++jt) {
        Partner p[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int j = j0 + 32 * u + lane;
            p[u].x = no_place();
            p[u].g = make_float4(0.f, 1.f, 1.f, 0.f);
            p[u].l = make_float2(0.f, 0.f);
            if (j < N) {
                p[u].x = place(V, A + j);
                p[u].g = V.gq[A + j];
                p[u].l = V.plj32[P + j];
            }
        }
        if (jt != next) {
#pragma unroll
            for (int u = 0; u < kBatch; u += 2) pair(p[u], p[u + 1], 0u, 0u);
        } else {
            ++mp;
            next = mp < mend ? V.mt_list[mp] : 0x7fffffff;
            uint32_t m[kBatch] = {}; // bit l of m[u]: partner j0 + 32 u + l is excluded
            if (i < N) {
                const int e1 = V.excl_off[P + i + 1];
                for (int e0 = V.excl_off[P + i]; e0 < e1; e0 += 32) {
                    const int d = e0 + lane < e1 ? V.excl_j[e0 + lane] - j0 : -1;
#pragma unroll
                    for (int u = 0; u < kBatch; ++u)
                        m[u] |= __reduce_or_sync(0xffffffffu, (d >> 5) == u ? 1u << (d & 31) : 0u);
                }
            }
            const int dself = i - j0 - lane; // 32 u where partner u is the atom itself
#pragma unroll
            for (int u = 0; u < kBatch; u += 2) {
                const uint32_t self = (dself == 32 * u ? 1u : 0u) | (dself == 32 * u + 32 ? 2u : 0u);
                pair(p[u], p[u + 1], self, self | ((m[u] >> lane) & 1u) | (((m[u + 1] >> lane) & 1u) << 1));
            }
        }
        if ((j0 & (kOrdFlush - 1)) == kOrdFlush - kTile || j0 + kTile >= N) {
            Pr::add(fx, px.x + px.y, (float)kScaleE);
            Pr::add(fy, py.x + py.y, (float)kScaleE);
            Pr::add(fz, pz.x + pz.y, (float)kScaleE);
            Pr::add(adr, pdr.x + pdr.y, (float)kScaleE);
            px = py = pz = pdr = zero;
            if (ENERGY) {
                Pr::add(egb, pgb.value(), (float)kScaleE);
                Pr::add(ec, pc.value(), (float)kScaleE);
                Pr::add(elj, plj.value(), (float)kScaleE);
                pgb = pc = plj = KSum<float2>();
            }
        }
    }
    const bool own = tid < kWarpAtoms && it.i0 + tid < N;
    const GbIn in = own ? GbIn(V, A, P, it.i0 + tid) : GbIn();
    if constexpr (ENERGY) sums.collect({fx, fy, fz, adr, egb, ec, elj});
    else sums.collect({fx, fy, fz, adr});
    if (tid < kWarpAtoms) gb_epilogue<ENERGY>(V, A, P, w, it.i0 + tid, own, sums, in);
}

// ------------------------------------------ pass 3: chain rule through Born radii
struct ChainNear {
    float4 p; // separation from atom i, c_j
    float2 r; // s_j, rt_j
};

// A fifth warp takes the CTA's bonded terms (FP64 separations behind four
// dependent loads) while the others run their pairs.
constexpr int kChainThreads = kTile + 32;

template <bool ENERGY, bool CUT>
__global__ void __launch_bounds__(kChainThreads) k_chain32(const Item* __restrict__ items, View V) {
    pdl_sync();
    using Pr = Prec<float>;
    __shared__ AtomSums<3> sums;
    __shared__ BondedSums bonded;
    __shared__ ChainNear sq[kWarpAtoms][kOrdQueue];
    const Item it = items[blockIdx.x];
    const int w = it.w, s = V.w_sys[w], N = V.sys_n[s], A = V.w_off[w], P = V.sys_poff[s];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    long long fx = 0, fy = 0, fz = 0;
    if (warp == kWarpAtoms) {
        bonded.take<ENERGY>(V, A, P, it.i0, N, lane);
    } else {
        const int i = it.i0 + warp;
        Place me = far_place();
        float ci = 0.f;
        if (i < N) {
            me = place(V, A + i);
            ci = V.c32[A + i];
        }
        const float si = me.h.w, rti = me.l.w;
        const PairBand band = pair_band(V.rfar2, V.smax32, (float)V.rgbmax);
        const float2 c2 = splat<float2>(ci), s2i = splat<float2>(si * si), s3i = splat<float2>(si * si * si);
        float2 fx2 = splat<float2>(0.f), fy2 = fx2, fz2 = fx2;
        float px = 0.f, py = 0.f, pz = 0.f;
        NearQueue<ChainNear> near_q(sq[warp]);
        auto closed = [&](const ChainNear& e) {
            const float r2 = e.p.x * e.p.x + e.p.y * e.p.y + e.p.z * e.p.z;
            const float rinv = Pr::rsqrt(r2), r = r2 * rinv;
            const float t = -(ci * hct_dr(r, rinv, rti, e.r.x, band.rc) + e.p.w * hct_dr(r, rinv, e.r.y, si, band.rc)) * rinv;
            px += t * e.p.x;
            py += t * e.p.y;
            pz += t * e.p.z;
        };
        auto flush = [&] {
            Pr::add(fx, px + (fx2.x + fx2.y), (float)kScaleE);
            Pr::add(fy, py + (fy2.x + fy2.y), (float)kScaleE);
            Pr::add(fz, pz + (fz2.x + fz2.y), (float)kScaleE);
            px = py = pz = 0.f;
            fx2 = fy2 = fz2 = splat<float2>(0.f);
        };
        for (int j0 = 0; j0 < N; j0 += kTile) {
            Place x[kBatch];
            float c[kBatch];
            ChainNear e[kBatch];
            bool near[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int j = j0 + 32 * u + lane;
                x[u] = no_place();
                c[u] = 0.f;
                if (j < N) {
                    x[u] = place(V, A + j);
                    c[u] = V.c32[A + j];
                }
            }
#pragma unroll
            for (int u = 0; u < kBatch; u += 2) {
                const Place &a = x[u], &b = x[u + 1];
                float2 dx, dy, dz;
                separation(me, a, b, dx, dy, dz);
                const float2 cj = make_float2(c[u], c[u + 1]), sj = make_float2(a.h.w, b.h.w), s2j = __fmul2_rn(sj, sj);
                float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                near[u] = band_near<CUT>(r2.x, band);
                near[u + 1] = band_near<CUT>(r2.y, band);
                r2.x = near[u] ? INFINITY : r2.x; // where the far form is 0
                r2.y = near[u + 1] ? INFINITY : r2.y;
                near[u] = near[u] && j0 + 32 * u + lane != i;
                near[u + 1] = near[u + 1] && j0 + 32 * u + 32 + lane != i;
                const float2 rinv2 = make_float2(rcp_ftz(r2.x), rcp_ftz(r2.y));
                const float2 qj = hct_series_dr(__fmul2_rn(s2j, rinv2)), qi = hct_series_dr(__fmul2_rn(s2i, rinv2));
                const float2 term = __ffma2_rn(__fmul2_rn(c2, __fmul2_rn(s2j, sj)), qj, __fmul2_rn(__fmul2_rn(cj, s3i), qi));
                float2 v = __fmul2_rn(term, __fmul2_rn(__fmul2_rn(rinv2, rinv2), rinv2));
                if (CUT) { // beyond rc + s_max nothing descreens
                    v.x = r2.x >= band.rout2 ? 0.f : v.x;
                    v.y = r2.y >= band.rout2 ? 0.f : v.y;
                }
                fx2 = __ffma2_rn(v, dx, fx2);
                fy2 = __ffma2_rn(v, dy, fy2);
                fz2 = __ffma2_rn(v, dz, fz2);
                e[u] = {make_float4(dx.x, dy.x, dz.x, cj.x), make_float2(a.h.w, a.l.w)};
                e[u + 1] = {make_float4(dx.y, dy.y, dz.y, cj.y), make_float2(b.h.w, b.l.w)};
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) near_q.push(near[u], e[u], lane);
            near_q.drain(lane, closed);
            if ((j0 & (kOrdFlush - 1)) == kOrdFlush - kTile) flush();
        }
        near_q.finish(lane, closed);
        flush();
    }
    sums.collect({fx, fy, fz});
    if (tid < kWarpAtoms) chain_epilogue<ENERGY>(V, A, w, it.i0 + tid, it.i0 + tid < N, sums, bonded);
}

} // namespace cph
