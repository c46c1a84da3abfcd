// Pair-tile arithmetic shared by the engine's FP32 passes and the
// differentiable GB energy: a lane's two i atoms against partner l + k of two
// staged j-tiles (A, B) at step k, every quantity a float2 whose halves belong
// to tile A and tile B, so that fma/add/mul.rn.f32x2 cover both tiles.
#pragma once
#include "cph_device.cuh"

namespace cph {

constexpr int kTileJ = 32; // atoms per j-tile

// Far GB pairs: with D = r^2 / (4 R_i R_j) >= 18, e^-D <= 1.6e-8, so
// 1/f = 1/r to 1e-10 relative, the GB force factor (1 - e^-D / 4) is 1 to
// 4e-9, and the pair's dE/dR term (~ e^-D (1 + D)) is below 3e-7 of its
// q_i q_j / r^3 (and far below the self and near-pair terms of dE/dR).  The
// engine's GB tiles take that form for each i-atom row of a step whose pairs
// all meet the bound (a warp vote per row), the adjoint's tiles for a step
// whose pairs all do (a warp vote per step).
constexpr float kGbFarD2 = 18.f * kLog2e; // the threshold on D log2(e)

// ========================================================= Born radii
// Each unordered pair yields both descreening integrals, H(r, rt_i, s_j) for
// psi_i (i-side sum ah) and H(r, rt_j, s_i) for psi_j (partner sum jh, which
// moves one lane per step).  In the far regime H = P(y) s^3 / r^4 with
// y = s^2 / r^2 (P the fitted series), so s^2 and s^3 are staged and 1/r^4
// serves both directions as the weight of a fused accumulate (1 for the
// closed forms, 0 for pairs that are not counted).  Bit jj of sk[u][h]
// marks a pair of i atom u and partner jj of tile h that is not counted.
struct BoI2 {
    float2 x, y, z, s2, s3; // the i atom's value in both halves
    float s, rt, irt;       // closed-form operands
};

struct BoJs {
    float4 a[2 * kTileJ]; // (-xA, -xB, -yA, -yB)
    float4 b[2 * kTileJ]; // (-zA, -zB, s2A, s2B)
    float4 c[2 * kTileJ]; // (s3A, s3B, sA, sB)
    float4 n[2 * kTileJ]; // (rtA, rtB, 1/rtA, 1/rtB): closed forms
};

// Which pairs a tile sends to the closed forms.  Without a Born-radius
// cutoff: those inside r_far.  With a cutoff rc, also the band
// rc - s_max < r < rc + s_max, where U = min(r + s, rc) may sit at rc; inside
// the band's lower edge r + s <= rc for every s, so the series still holds
// there, and beyond its upper edge every integral and derivative of the pair
// vanishes (L >= r - s_max >= rc >= U), which CUT tiles apply as a select.
// Skipped pairs take r^2 = infinity, where every form is 0.
struct PairBand {
    float rfar2, rin2, rout2, rc;
};

// rfar2 and s_max over every atom; rc = INFINITY for no cutoff.  The band's
// edges are widened by 1e-5 so that rounding can only move a pair towards
// the closed forms.
__host__ __device__ inline PairBand pair_band(float rfar2, float smax, float rc) {
    PairBand b;
    b.rfar2 = rfar2;
    b.rc = rc;
    if (rc < INFINITY) {
        const float rin = fmaxf(rc - smax, 0.f) * (1.f - 1e-5f), rout = (rc + smax) * (1.f + 1e-5f);
        b.rin2 = rin * rin;
        b.rout2 = rout * rout;
    } else {
        b.rin2 = b.rout2 = INFINITY;
    }
    return b;
}

template <bool CUT>
__device__ __forceinline__ bool band_near(float r2, const PairBand& b) {
    return CUT ? (r2 < b.rfar2 || (r2 > b.rin2 && r2 < b.rout2)) : r2 < b.rfar2;
}

// Closed-form integrals of one pair inside r_far (or in the cutoff band), kept
// out of line: one copy, called where a warp's queued near pairs are
// evaluated.  Returns (H(r, rt_i, s_j), H(r, rt_j, s_i)).
static __device__ __noinline__ float2 born_near(float r2, float rinv, float rt_i, float irt_i, float s_i, float s_j,
                                         float rt_j, float irt_j, float rc) {
    const float r = r2 * rinv;
    return make_float2(hct(r, rinv, rt_i, irt_i, s_j, rc), hct(r, rinv, rt_j, irt_j, s_i, rc));
}

// ------------------------------------------------ near pairs, apart from the tile loop
// A pair inside r_far (or in the cutoff band) costs several times a far one,
// and a warp step of 128 pairs that meets one pays the closed forms for every
// lane: 7 % of the steps of an 8000-atom chain, 20 % at 2400 atoms, 50 % at 240.
// So the tile loop gives near pairs weight 0 and only notes them, one bit per
// (i slot u, half h, step k) in four registers a lane; after each tile pair the
// warp moves its bits into a queue, a lane at a time taking its next one, and
// evaluates the queue 32 pairs at a time with every lane busy.  What is left
// waits for the next tile pair of the staged group and is evaluated at the
// group's end, so the order of a group's sums depends on nothing but its atoms.
// Against closed forms behind a warp vote in the tile loop (GB energy and
// gradient kernels): Born radii 121 -> 43 us, chain rule 202 -> 72 us at
// 16 x 1203 (with the smaller work items), 93 -> 35 us at 1 x 237, and
// 21.59 -> 21.4 ms for energy and gradient of 128 x 8000.
// One queue entry: lane | u << 5 | h << 6 | partner << 7 | tile pair << 12.
constexpr int kNearCap = 64; // entries per warp: a round adds <= 32 to < 32

struct NearBits {
    uint32_t m[2][2]; // [u][h], bit k
};

// Calls eval(entry, valid) for the noted pairs; `last`: the group's last tile
// pair.  nq (warp-uniform) carries the entries that wait.
template <class F>
__device__ __forceinline__ void near_drain(NearBits& nb, uint16_t* q, int& nq, int lane, int pr, bool last, F&& eval) {
    const uint32_t lt = (1u << lane) - 1u;
    for (;;) {
        const bool has = (nb.m[0][0] | nb.m[0][1] | nb.m[1][0] | nb.m[1][1]) != 0u;
        const uint32_t bal = __ballot_sync(0xffffffffu, has);
        if (has) {
            const int s = nb.m[0][0] ? 0 : (nb.m[0][1] ? 1 : (nb.m[1][0] ? 2 : 3));
            const uint32_t m = s == 0 ? nb.m[0][0] : (s == 1 ? nb.m[0][1] : (s == 2 ? nb.m[1][0] : nb.m[1][1]));
            const uint32_t r = m & (m - 1u);
            if (s == 0) nb.m[0][0] = r;
            else if (s == 1) nb.m[0][1] = r;
            else if (s == 2) nb.m[1][0] = r;
            else nb.m[1][1] = r;
            const int jj = (lane + __ffs(m) - 1) & (kTileJ - 1);
            q[nq + __popc(bal & lt)] = (uint16_t)(lane | ((s >> 1) << 5) | ((s & 1) << 6) | (jj << 7) | (pr << 12));
        }
        nq += __popc(bal);
        const int n = nq >= 32 ? 32 : ((last && !bal) ? nq : 0);
        if (n) {
            __syncwarp();
            const bool valid = lane < n;
            const uint32_t e = q[nq - n + (valid ? lane : 0)];
            eval(e, valid);
            nq -= n;
            __syncwarp();
        } else if (!bal) {
            break;
        }
    }
}

// Turns of the lanes that hold the same key, so that each adds to the key's
// slot alone: calls add() in turn, lowest lane first.
template <class F>
__device__ __forceinline__ void in_turn(uint32_t key, bool valid, int lane, F&& add) {
    const uint32_t peers = __match_any_sync(0xffffffffu, valid ? key : 0xffffffffu);
    const int turn = valid ? __popc(peers & ((1u << lane) - 1u)) : 0;
    const int turns = __reduce_max_sync(0xffffffffu, turn);
    for (int t = 0; t <= turns; ++t) {
        if (valid && turn == t) add();
        __syncwarp();
    }
}

// Notes the near pairs of one step and moves them to infinity, where every far
// form is 0 (the pairs that a masked tile skips start there).  Behind a vote:
// 21.52 -> 21.37 ms on 128 x 8000 (energy and gradient), where few steps meet a
// near pair; no difference at 16 x 1203.
template <bool CUT>
__device__ __forceinline__ void note_near(float2 (&r2)[2], const PairBand& band, int k, NearBits& nb) {
    bool n[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        n[u][0] = band_near<CUT>(r2[u].x, band);
        n[u][1] = band_near<CUT>(r2[u].y, band);
    }
    if (__any_sync(0xffffffffu, n[0][0] || n[0][1] || n[1][0] || n[1][1])) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            nb.m[u][0] |= n[u][0] ? 1u << k : 0u;
            nb.m[u][1] |= n[u][1] ? 1u << k : 0u;
            r2[u].x = n[u][0] ? INFINITY : r2[u].x;
            r2[u].y = n[u][1] ? INFINITY : r2[u].y;
        }
    }
}

// Tile pairs below the returned index of the group at j-tile g0 hold only
// partners j <= i of the warp's 64 i atoms (i-tiles start at a multiple of 256
// atoms), or, for a warp without atoms, all of them: nothing of them is
// counted, and the warp passes them by.
__device__ __forceinline__ int live_pair(int i0, int warp, int n, int g0, int npair) {
    const int iw = i0 + warp * 2 * kTileJ;
    return iw >= n ? npair : min(npair, max(0, iw / kTileJ - g0) / 2);
}

template <bool MASKED, bool CUT>
__device__ __forceinline__ void born_tile(const BoJs& sj, int lane, const BoI2 (&I)[2], float2 (&ah)[2],
                                          float2& jh, const uint32_t (&sk)[2][2], const PairBand& band, NearBits& nb) {
    const int src = (lane + 1) & 31;
#pragma unroll 2
    for (int k = 0; k < kTileJ; ++k) {
        const float4 A = sj.a[lane + k], B = sj.b[lane + k], C = sj.c[lane + k];
        const float2 s2j = make_float2(B.z, B.w), s3j = make_float2(C.x, C.y);
        float2 r2[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float2 dx = __fadd2_rn(I[u].x, make_float2(A.x, A.y));
            const float2 dy = __fadd2_rn(I[u].y, make_float2(A.z, A.w));
            const float2 dz = __fadd2_rn(I[u].z, make_float2(B.x, B.y));
            r2[u] = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
            if (MASKED) {
                const int jj = (lane + k) & (kTileJ - 1);
                r2[u].x = ((sk[u][0] >> jj) & 1u) ? INFINITY : r2[u].x;
                r2[u].y = ((sk[u][1] >> jj) & 1u) ? INFINITY : r2[u].y;
            }
        }
        note_near<CUT>(r2, band, k, nb);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float2 rinv2 = make_float2(rcp_ftz(r2[u].x), rcp_ftz(r2[u].y));
            float2 wt = __fmul2_rn(rinv2, rinv2); // r^-4, the weight of both far terms
            if (CUT) { // beyond rc + s_max nothing descreens
                wt.x = r2[u].x >= band.rout2 ? 0.f : wt.x;
                wt.y = r2[u].y >= band.rout2 ? 0.f : wt.y;
            }
            const float2 hi = hct_series_h(__fmul2_rn(s2j, rinv2)), hj = hct_series_h(__fmul2_rn(I[u].s2, rinv2));
            ah[u] = __ffma2_rn(__fmul2_rn(hi, s3j), wt, ah[u]);
            jh = __ffma2_rn(__fmul2_rn(hj, I[u].s3), wt, jh);
        }
        jh.x = __shfl_sync(0xffffffffu, jh.x, src);
        jh.y = __shfl_sync(0xffffffffu, jh.y, src);
    }
}

} // namespace cph
