// SHAKE of the small-walker kernel (cph_small.cuh) in pairs of floats.  Nothing is
// included here: the tests compile this file for the host, with stand-ins for
// View and for the device's arithmetic and warp exchanges.
#pragma once

namespace cph {

__device__ __forceinline__ float2 split2(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}

// a + b as an unevaluated sum of two floats added to (h, l)
__device__ __forceinline__ void add2(float& h, float& l, float b) {
    const float s = __fadd_rn(h, b), t = __fsub_rn(s, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(b, t)));
    h = s;
}

// Sum of h + l over the cluster's lanes, the same bits in each: both lanes of an
// exchange add the low words first and then the (exact) rounding error of the
// high ones.  The lanes decide by it, each for its own component, whether a
// constraint is settled.
__device__ __forceinline__ void sum4(float& h, float& l) {
#pragma unroll
    for (int o = 1; o < 3; o <<= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
        l = __fadd_rn(l, ol);
        add2(h, l, oh);
    }
}

// SHAKE (k_shake) of clusters of at most NH hydrogens, cluster c of the lane, four
// lanes to a cluster, one for each component (the fourth idle).  Each
// constraint moves its atoms along the old bond vector, so the unknowns are
// displacements; with R the bond vector before the sweeps and D the difference of
// the two displacements, d0^2 - |R + D|^2 = (d0^2 - R^2) - (2 R + D) . D.  The
// first term is formed once in FP64; displacements and the second term are kept
// as pairs of floats (1e-14 of d0^2, against a tolerance of 1e-8 and less), and
// so is the step along the bond: an FP32 quotient would do for the constraint, but
// leaves the sweeps somewhere else within the tolerance (1e-11 A), which a
// trajectory grows until it shows in the forces' roundings (100 steps of 48 runs:
// velocities off k_shake's by up to 1.4e-5, with the pair by 8e-6 in one system
// and 6e-7 in the others; 1.92 -> 1.96 ms for 50 steps of 4 x 246 atoms).  In FP64 a
// constraint took ~35 instructions of 64 clocks: 39,000 clocks a step there.
template <int NH>
__device__ __noinline__ void small_shake(const View& V, const float4* fac, int c, bool on, int d, const double* xo,
                                         double* xt, int nh, double (&u)[NH + 1]) {
    const bool live = on && d < 3;
    const int h0 = V.shk_off[c], a0 = V.shk_heavy[c];
    float Rh[NH], Rl[NH], old[NH], oldl[NH], d0h[NH], d0l[NH], tol[NH];
    float uh[NH + 1], ul[NH + 1];   // displacements of the heavy atom and the hydrogens
    float2 dir0[NH], dirk[NH];      // their directions: mass factor times old bond vector
    const double x0 = live ? xt[3 * a0 + d] : 0.0, o0 = live ? xo[3 * a0 + d] : 0.0;
#pragma unroll
    for (int k = 0; k < NH; ++k) {
        const bool has = live && k < nh;
        const int a = has ? V.shk_h[h0 + k] : a0;
        const double r = has ? x0 - xt[3 * a + d] : 0.0;
        const float2 R = split2(2.0 * r);
        Rh[k] = R.x;
        Rl[k] = R.y;
        const float2 o = split2(has ? o0 - xo[3 * a + d] : 0.0);
        const float4 f = on && k < nh ? fac[h0 + k] : make_float4(0.f, 0.f, 0.f, 0.f);
        old[k] = o.x;
        oldl[k] = o.y;
        dir0[k].x = f.x * o.x;
        dir0[k].y = fmaf(f.x, o.x, -dir0[k].x) + fmaf(f.x, o.y, f.y * o.x);
        dirk[k].x = f.z * o.x;
        dirk[k].y = fmaf(f.z, o.x, -dirk[k].x) + fmaf(f.z, o.y, f.w * o.x);
        double r2 = r * r;
        r2 += __shfl_xor_sync(0xffffffffu, r2, 1);
        r2 += __shfl_xor_sync(0xffffffffu, r2, 2);
        const double dk = on && k < nh ? V.shk_d[h0 + k] : 0.0;
        const float2 D = split2(dk * dk - r2);
        d0h[k] = D.x;
        d0l[k] = D.y;
        tol[k] = on && k < nh ? 2.f * (float)V.shake_tol * (float)dk * (float)dk : INFINITY;
    }
#pragma unroll
    for (int k = 0; k <= NH; ++k) uh[k] = ul[k] = 0.f;
    bool done = false;
    for (int iter = 0; iter < kShakeMaxIter && !__all_sync(0xffffffffu, done); ++iter) {
        bool moved = false;
#pragma unroll
        for (int k = 0; k < NH; ++k) {
            float dh = uh[0], dl = ul[0] - ul[k + 1]; // D
            add2(dh, dl, -uh[k + 1]);
            float sh = Rh[k], sl = Rl[k] + dl; // 2 R + D
            add2(sh, sl, dh);
            float ph = sh * dh;
            float pl = fmaf(sh, dh, -ph) + fmaf(sh, dl, sl * dh);
            float qh = 0.5f * Rh[k], ql = fmaf(0.5f, Rl[k], dl); // R / 2 + D, here R is twice the bond
            add2(qh, ql, dh);
            float dot = old[k] * qh, dotl = fmaf(old[k], qh, -dot) + fmaf(old[k], ql, oldl[k] * qh);
            sum4(ph, pl);
            sum4(dot, dotl);
            float eh = d0h[k], el = d0l[k] - pl;
            add2(eh, el, -ph);
            const float diff = eh + el;
            if (!done && fabsf(diff) > tol[k]) {
                moved = true;
                // diff / dot and the products to 1e-14
                const float g = __fdividef(diff, dot);
                const float gl = __fdividef(fmaf(-g, dot, eh) + fmaf(-g, dotl, el), dot);
                const float p0 = g * dir0[k].x, pk = -g * dirk[k].x;
                ul[0] += fmaf(g, dir0[k].x, -p0) + fmaf(g, dir0[k].y, gl * dir0[k].x);
                ul[k + 1] += fmaf(-g, dirk[k].x, -pk) - fmaf(g, dirk[k].y, gl * dirk[k].x);
                add2(uh[0], ul[0], p0);
                add2(uh[k + 1], ul[k + 1], pk);
            }
        }
        done = done || !moved;
    }
    if (!done) atomicOr(V.status, 8);
#pragma unroll
    for (int k = 0; k <= NH; ++k) u[k] = (double)uh[k] + (double)ul[k];
}

} // namespace cph
