// Device-side building blocks of the engine: constants, Philox4x32-10,
// fixed-point helpers and the per-pair arithmetic of the OBC generalized-Born
// model ("igb=2", named in the paper's Implicit Solvent Calculations
// section) with Hawkins-Cramer-Truhlar pairwise descreening.
//
// Pair quantities for atom i and a partner j at distance r:
//   H(r, rt, s)  descreening integral of sphere s (partner's scaled radius)
//                outside the ball rt (this atom's offset radius):
//                0 if rt >= r + s; else with L = max(rt, |r - s|), U = r + s
//                H = 1/L - 1/U + (r/4)(1/U^2 - 1/L^2) + ln(L/U)/(2r)
//                    + (s^2/(4r))(1/L^2 - 1/U^2)  [+ 2(1/rt - 1/L) if rt < s - r]
//   When the spheres are disjoint (L = r - s) H depends on r and x = s/r only:
//   H = (1/r) (x/(1 - x^2) - atanh x) = (1/r) sum_{k>=1} 2k/(2k+1) x^(2k+1).
//   The FP32 path evaluates that series (a degree-5 polynomial in x^2, fitted
//   on the interval) whenever x <= 0.35: it needs no transcendental, and it
//   avoids the cancellation of the closed form (whose terms are O(x) while H
//   is O(x^3)).  The fits stay within 2e-8 relative error.
//   Derivatives: in every branch the L- and U-dependence of H cancels (the
//   integrand vanishes on the moving boundary), so
//     dH/dr  = -(1/4)(1/L^2 - 1/U^2)(1 + s^2/r^2) - ln(L/U)/(2 r^2)
//            = -(1/r^2) sum 2k(2k+2)/(2k+1) x^(2k+1)      (disjoint)
//     dH/ds  = (s/(2r))(1/L^2 - 1/U^2) = (1/r^2) sum 2k x^(2k)
//     dH/drt = ((L - r)^2 - s^2)/(2 r L^3) when L = rt, -2/rt^2 when the ball
//              lies inside sphere s, else 0.
#pragma once
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

namespace cph {

// Physical constants (kcal/mol, A, e, amu, ps, K, V).
constexpr double kCoulomb = 332.0522173;   // kcal A / (mol e^2)
constexpr double kBoltzmann = 0.0019872041; // kcal / (mol K)
constexpr double kFaraday = 23.0605;       // kcal / (mol V)
constexpr double kAccel = 418.4;           // (kcal/mol/A)/amu -> A/ps^2
constexpr double kLn10 = 2.302585092994046;

// Fixed-point scales of the int64 accumulators.
constexpr double kScaleE = 4294967296.0;   // energies and forces: 2^32
constexpr double kScaleH = 1099511627776.0; // descreening sums: 2^40

// Random-number purposes (last counter word).
constexpr uint32_t kRngLangevin = 1, kRngMcPh = 2, kRngMcRedox = 3, kRngExchange = 4;

// ------------------------------------------------------------------ Philox
// Philox4x32 with ten rounds (Salmon, Moraes, Dror and Shaw, SC'11).  A round
// multiplies counter words 0 and 2 by 0xD2511F53 and 0xCD9E8D57, XORs the
// high product words with counter words 1 and 3 and the key, and permutes;
// between rounds the key advances by the Weyl increments 0x9E3779B9 and
// 0xBB67AE85.
struct U4 {
    uint32_t a, b, c, d;
};

__host__ __device__ inline U4 philox4x32_10(U4 ctr, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        uint64_t p0 = (uint64_t)0xD2511F53u * ctr.a;
        uint64_t p1 = (uint64_t)0xCD9E8D57u * ctr.c;
        U4 n;
        n.a = (uint32_t)(p1 >> 32) ^ ctr.b ^ k0;
        n.b = (uint32_t)p1;
        n.c = (uint32_t)(p0 >> 32) ^ ctr.d ^ k1;
        n.d = (uint32_t)p0;
        ctr = n;
    }
    return ctr;
}

// Counter (index, stream, step low word, purpose | step high bits << 8),
// key (seed low word, seed high word).
__host__ __device__ inline U4 draw(uint64_t seed, uint32_t index, uint32_t stream,
                                   uint64_t step, uint32_t purpose) {
    U4 c{index, stream, (uint32_t)step, (purpose & 0xffu) | ((uint32_t)(step >> 32) << 8)};
    return philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
}

// u in (0, 1): u32 * 2^-32 + 2^-33, exact in FP64.
__host__ __device__ inline double unit_open(uint32_t u) {
    return (double)u * 2.3283064365386963e-10 + 1.1641532182693481e-10;
}

// ------------------------------------------------------- salt screening
// A GB term of effective distance f (f = R for a self term) carries
// tau(f) = 1/eps_in - exp(-kappa f)/eps_out; d(tau(f)/f)/df = -taud(f)/f^2 with
// taud(f) = tau(f) - kappa f exp(-kappa f)/eps_out.  kappa = 0: both are the
// constant 1/eps_in - 1/eps_out.
// Without salt both are iei - ieo exactly (exp(-0) = 1): the FP64 exponential,
// slow on GB300's narrow FP64 pipe, is skipped.
__host__ __device__ inline double salt_tau(double f, double iei, double ieo, double kappa) {
    if (!(kappa > 0)) return iei - ieo;
    return iei - exp(-kappa * f) * ieo;
}
__host__ __device__ inline double salt_taud(double f, double iei, double ieo, double kappa) {
    if (!(kappa > 0)) return iei - ieo;
    const double es = exp(-kappa * f) * ieo;
    return iei - es - kappa * f * es;
}

// ------------------------------------------------- nonpolar surface term
// ACE approximation (Schaefer & Karplus 1996): E_SA = 4 pi gamma (rho + probe)^2
// (rho / R)^6 per atom; dE_SA/dR = -6 E_SA / R.  gamma = 0: off.
__host__ __device__ inline double sa_ace(double gamma, double probe, double rho, double R) {
    if (gamma == 0.0) return 0.0;
    const double a = rho + probe, t = rho / R, t3 = t * t * t;
    return 4.0 * 3.14159265358979323846 * gamma * a * a * t3 * t3;
}

// ---------------------------------------------- programmatic launches
// First statement of every kernel of a step: the launch is set up while the one
// before it on the stream still runs, and its work starts when that one has
// completed and its writes are visible (a no-op in a plain launch).  No kernel
// lets the next one in before its own end: blocks that come in early settle
// where SMs happen to be free, and the passes that count on an even spread
// suffer (FP64 evaluation of 2 x 1203 atoms 1.16 -> 1.71 ms).
__device__ __forceinline__ void pdl_sync() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// --------------------------------------------------------- fixed point
__device__ inline long long to_fixed(float v, float scale) { return __float2ll_rn(v * scale); }
__device__ inline long long to_fixed(double v, double scale) { return __double2ll_rn(v * scale); }

// __float2ll_rn(v * 2^32) through 32-bit conversions (exact: the integer part,
// then the fraction's 32 bits, rounded half to even as a whole would be)
__device__ __forceinline__ long long fix32(float v) {
    const float a = fabsf(v);
    if (!(a < 1073741824.f)) return to_fixed(v, (float)kScaleE);
    const unsigned hi = __float2uint_rz(a);
    const unsigned lo = __float2uint_rn((a - (float)hi) * 4294967296.f);
    const long long m = (long long)(((unsigned long long)hi << 32) | lo);
    return v < 0.f ? -m : m;
}

// 64-bit addition to shared memory as two 32-bit ones (a 64-bit atomic there is a
// loop of compare-and-swap)
__device__ __forceinline__ void shared_add(long long* p, long long v) {
    unsigned* w = reinterpret_cast<unsigned*>(p);
    const unsigned lo = (unsigned)v, hi = (unsigned)((unsigned long long)v >> 32);
    const unsigned old = atomicAdd(w, lo);
    const unsigned up = hi + (old > ~lo ? 1u : 0u);
    if (up) atomicAdd(w + 1, up);
}

// sum over the warp, in every lane (exact integers: any order)
__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------ FP64 in few instructions
// A warp instruction of FP64 holds a sub-partition of GB300 for 64 clocks, with
// one active lane or with 32.  Against CUDA's own functions over these domains: rcp64
// and rsqrt64 2.2e-16 relative, log64 2.2e-16 of max(|log x|, 2^-7), exp64 2.2e-16
// relative, tanh64 2.2e-16 and sincos64 3.5e-16 absolute.
// 1 / x for normal x: the PTX approximation (20 bits) and one step of Householder's
// third-order iteration (1970), y (1 + e + e^2) with e = 1 - x y
__device__ __forceinline__ double rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// The same with 1/0 = infinity and 1/infinity = 0: a Born radius (1/R = 1/rt - tanh/rho
// is 0 where the tanh has saturated and the offset is 0) and its reciprocal.
__device__ __forceinline__ double rcp64_radius(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const int h = __double2hiint(y) & 0x7fffffff;
    const double e = fma(-x, y, 1.0);
    return h == 0 || h == 0x7ff00000 ? y : fma(y, fma(e, e, e), y);
}

// Born radii as the pair arithmetic takes them: not infinite, and so are their
// products; with these values 1/f is 0 to every digit that counts.  (NaN stays NaN.)
__device__ __forceinline__ float pair_radius32(double R) {
    const float r = (float)R;
    return r > 1e18f ? 1e18f : r;
}
__device__ __forceinline__ double pair_radius64(double R) { return __double2hiint(R) == 0x7ff00000 ? 1e150 : R; }

// 1 / sqrt(x) for normal x > 0: the same (the binomial series after its second
// term) with y (1 + e/2 + 3 e^2/8), e = 1 - x y^2
__device__ __forceinline__ double rsqrt64(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Tables of log64 and exp64, to be copied to shared memory (divergent indices):
// for the j-th of 128 intervals of m in [0.6875, 1.375) an approximate 1/c of its
// middle c and -log of that number; then 2^(j/16), two to an entry.
constexpr int kTab64 = 136;
static __device__ const double2 kTab64Values[kTab64] = {
    {1.4504249291784703, -0.37185656810621104}, {1.4422535211267606, -0.36620683556409206},
    {1.4341736694677871, -0.36058884325986873}, {1.426183844011142, -0.3550022365512289},
    {1.4182825484764543, -0.3494466667066269}, {1.4104683195592287, -0.343921790774657},
    {1.4027397260273973, -0.3384272714570163}, {1.3950953678474114, -0.3329627769849375},
    {1.3875338753387534, -0.3275279809989806}, {1.3800539083557952, -0.3221225624320727},
    {1.3726541554959786, -0.31674620539569226}, {1.3653333333333333, -0.31139859906909695},
    {1.3580901856763925, -0.306079437591497}, {1.3509234828496042, -0.3007884199570814},
    {1.3438320209973753, -0.2955252499128068}, {1.3368146214099217, -0.2902896358588618},
    {1.3298701298701299, -0.28508129075172356}, {1.322997416020672, -0.279899932009726},
    {1.3161953727506426, -0.2747452814210614}, {1.3094629156010231, -0.26961706505414207},
    {1.3027989821882953, -0.2645150131702466}, {1.2962025316455696, -0.2594388601383859},
    {1.2896725440806045, -0.25438834435231733}, {1.2832080200501252, -0.24936320814964427},
    {1.2768079800498753, -0.24436319773293858}, {1.2704714640198511, -0.23938806309282482},
    {1.2641975308641975, -0.23443755793296864}, {1.257985257985258, -0.22951143959691278},
    {1.2518337408312958, -0.22460946899670603}, {1.245742092457421, -0.2197314105432732},
    {1.2397094430992737, -0.21487703207847508}, {1.2337349397590363, -0.21004610480880959},
    {1.2278177458033572, -0.20523840324070627}, {1.2219570405727924, -0.2004537051173701},
    {1.2161520190023754, -0.19569179135712642}, {1.210401891252955, -0.1909524459932298},
    {1.204705882352941, -0.18623545611509087}, {1.199063231850117, -0.18154061181088324},
    {1.1934731934731935, -0.1768677061114908}, {1.1879350348027842, -0.17221653493575995},
    {1.1824480369515011, -0.16758689703701793}, {1.1770114942528735, -0.16297859395082367},
    {1.17162471395881, -0.15839142994391764}, {1.1662870159453302, -0.15382521196433638},
    {1.1609977324263039, -0.14927974959266183}, {1.1557562076749435, -0.14475485499437207},
    {1.150561797752809, -0.14025034287326765}, {1.145413870246085, -0.13576603042593893},
    {1.1403118040089086, -0.13130173729725345}, {1.1352549889135255, -0.12685728553682943},
    {1.130242825607064, -0.12243249955647377}, {1.1252747252747253, -0.11802720608855737},
    {1.1203501094091903, -0.11364123414530306}, {1.1154684095860568, -0.10927441497896273},
    {1.1106290672451193, -0.10492658204285929}, {1.1058315334773219, -0.10059757095327378},
    {1.1010752688172043, -0.09628721945215148}, {1.0963597430406853, -0.09199536737061052},
    {1.091684434968017, -0.0877218565932284}, {1.0870488322717622, -0.08346653102309001},
    {1.0824524312896406, -0.07922923654757486}, {1.0778947368421052, -0.07500982100486656},
    {1.0733752620545074, -0.07080813415116662}, {1.068893528183716, -0.06662402762859244},
    {1.0644490644490645, -0.06245735493374666}, {1.060041407867495, -0.05830797138693517},
    {1.0556701030927835, -0.054175734102024614}, {1.051334702258727, -0.05006050195691803},
    {1.047034764826176, -0.04596213556463585}, {1.0427698574338085, -0.04188049724498711},
    {1.0385395537525355, -0.037815450996817664}, {1.0343434343434343, -0.033766862470817484},
    {1.0301810865191148, -0.029734598942879144}, {1.0260521042084167, -0.025718529287989036},
    {1.0219560878243512, -0.021718523954642903}, {1.0178926441351888, -0.017734454939768475},
    {1.0138613861386139, -0.01376619576414797}, {1.009861932938856, -0.00981362144832467},
    {1.005893909626719, -0.005876608488984971}, {1.0019569471624266, -0.001955034835803295},
    {0.9961089494163424, 0.003898640415657309}, {0.9884169884169884, 0.01165061721997525},
    {0.9808429118773946, 0.019342962843130987}, {0.973384030418251, 0.026976587698202083},
    {0.9660377358490566, 0.03455238150665973}, {0.9588014981273408, 0.042071213920687044},
    {0.9516728624535316, 0.049533935122276676}, {0.9446494464944649, 0.05694137640013845},
    {0.9377289377289377, 0.06429435070539725}, {0.9309090909090909, 0.07159365318700882},
    {0.924187725631769, 0.078840061707776}, {0.9175627240143369, 0.08603433734180316},
    {0.9110320284697508, 0.09317722485418334}, {0.9045936395759717, 0.10026945316367517},
    {0.8982456140350877, 0.10731173578908804}, {0.89198606271777, 0.11430477128005863},
    {0.8858131487889274, 0.12124924363286965}, {0.8797250859106529, 0.12814582269193006},
    {0.8737201365187713, 0.13499516453750482}, {0.8677966101694915, 0.1417979118602574},
    {0.8619528619528619, 0.1485546943231372}, {0.8561872909698997, 0.15526612891112396},
    {0.8504983388704319, 0.16193282026931324}, {0.8448844884488449, 0.16855536102980664},
    {0.839344262295082, 0.17513433212784915}, {0.8338762214983714, 0.18167030310763463},
    {0.8284789644012945, 0.18816383241818294}, {0.8231511254019293, 0.19461546769967167},
    {0.8178913738019169, 0.2010257460605908}, {0.8126984126984127, 0.2073951943460706},
    {0.807570977917981, 0.21372432939771818}, {0.8025078369905956, 0.22001365830528213},
    {0.7975077881619937, 0.2262636786504534}, {0.7925696594427245, 0.232474878743094},
    {0.7876923076923077, 0.238647737850175}, {0.7828746177370031, 0.24478272641769092},
    {0.7781155015197568, 0.25088030628580943}, {0.7734138972809668, 0.2569409308975004},
    {0.7687687687687688, 0.26296504550088134}, {0.764179104477612, 0.26895308734550394},
    {0.7596439169139466, 0.2749054858727992}, {0.7551622418879056, 0.2808226629008878},
    {0.750733137829912, 0.2867050328039543}, {0.7463556851311953, 0.29255300268637746},
    {0.7420289855072464, 0.2983669725517973}, {0.7377521613832853, 0.3041473354672968},
    {0.7335243553008596, 0.3098944777228647}, {0.7293447293447294, 0.3156087789863033},
    {1.0, 1.0442737824274138}, {1.0905077326652577, 1.1387886347566916}, {1.189207115002721, 1.241857812073484}, {1.2968395546510096, 1.3542555469368927}, {1.4142135623730951, 1.4768261459394993}, {1.5422108254079407, 1.6104903319492543}, {1.681792830507429, 1.7562521603732995}, {1.8340080864093424, 1.9152065613971474}};

__device__ __forceinline__ void load_tab64(double2* tab, int tid, int n) {
    for (int k = tid; k < kTab64; k += n) tab[k] = kTab64Values[k];
}

// log(x), x normal and positive (Tang, 1990; the split of the argument at 0.6875, with
// index and exponent from one difference, is that of Arm's Optimized Routines): x =
// 2^e m, r = m/c - 1 (|r| < 0.006),
// log x = e ln2 + log c + log1p(r); the series stops at r^7/7 < 1e-16 |r|.
__device__ __forceinline__ double log64(double x, const double2* tab) {
    const int i = __double2hiint(x) - 0x3fe60000;
    const double2 c = tab[(i >> 13) & 127];
    const double m = __hiloint2double(__double2hiint(x) - (i & 0xfff00000), __double2loint(x));
    const double r = fma(m, c.x, -1.0);
    const double e = __hiloint2double(0x43300000, (i >> 20) + 1024) - 4503599627371520.0; // 2^52 + 1024
    double p = fma(r, 1.0 / 7, -1.0 / 6);
    p = fma(p, r, 1.0 / 5);
    p = fma(p, r, -0.25);
    p = fma(p, r, 1.0 / 3);
    p = fma(p, r, -0.5);
    return fma(e, 0.6931471805599453, c.y + fma(r * r, p, r));
}

// e^x for x <= 0 (0 below -700; Tang, 1989): x = k ln2/16 + r, a Taylor series in r (|r| <=
// 0.022, remainder 1e-18) and the table.  T(j) = 2^(j/16).
template <class T>
__device__ __forceinline__ double exp64_with(double x, T&& table) {
    const double big = 6755399441055744.0; // 1.5 2^52: the sum's low word is the integer
    const double t = fma(x, 23.083120654223414, big);
    const double k = t - big;
    double r = fma(k, -0.04332169878499658, x);
    r = fma(k, -1.4494042586539372e-18, r);
    double p = fma(r, 1.0 / 5040, 1.0 / 720);
    p = fma(p, r, 1.0 / 120);
    p = fma(p, r, 1.0 / 24);
    p = fma(p, r, 1.0 / 6);
    p = fma(p, r, 0.5);
    p = fma(p, r, 1.0);
    const int n = __double2loint(t);
    const double b = table(n & 15);
    const double v = fma(b * r, p, b);
    const bool zero = (unsigned)__double2hiint(x) > 0xc085e000u; // x < -700
    return zero ? 0.0 : __hiloint2double(__double2hiint(v) + ((n >> 4) << 20), __double2loint(v));
}

__device__ __forceinline__ double exp64(double x, const double2* tab) {
    return exp64_with(x, [&](int j) { return reinterpret_cast<const double*>(tab + 128)[j]; });
}

// 2^(j/16), for the few evaluations that do not load the tables
static __constant__ double kExp2Tab[16] = {1.0, 1.0442737824274138, 1.0905077326652577, 1.1387886347566916, 1.189207115002721, 1.241857812073484, 1.2968395546510096, 1.3542555469368927, 1.4142135623730951, 1.4768261459394993, 1.5422108254079407, 1.6104903319492543, 1.681792830507429, 1.7562521603732995, 1.8340080864093424, 1.9152065613971474};
__device__ __forceinline__ double exp64(double x) {
    return exp64_with(x, [&](int j) { return kExp2Tab[j]; });
}

// tanh(x) = (1 - e) / (1 + e), e = e^(-2|x|): absolute error 2.2e-16, which is what
// the Born radius 1 / (1/rt - tanh / rho) asks for
__device__ __forceinline__ double tanh64(double x) {
    const double e = exp64(-2.0 * fabs(x));
    return copysign(fma(-2.0 * e, rcp64(1.0 + e), 1.0), x);
}

// ---------------------------------------------- MUFU approximations (FP32)
// The PTX ISA's approximate reciprocal square root and base-2 exponential in
// their flush-to-zero forms (rsqrt.approx.ftz.f32, ex2.approx.ftz.f32), written
// as inline PTX.  No operand of the pair loops comes near the denormal range
// (distances >= ~1 A; exp(-D) underflowing to 0 is harmless), so flushing
// changes no result; accuracy is covered by the parity tests against the
// FP64 oracle.
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The PTX ISA's approximate reciprocal (rcp.approx.ftz.f32): 1/r^2 in one MUFU
// operation where the tile needs no 1/r.
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float exp2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// ------------------------------------------------------------- HCT, FP32
constexpr float kHctXmax = 0.35f;

// Far-pair polynomials in y = (s/r)^2 on [0, 0.35^2]: degree-5 near-minimax
// fits (Chebyshev, relative error) of the series
//   P(y) = sum 2k/(2k+1) y^(k-1),  Q(y) = sum 2k(2k+2)/(2k+1) y^(k-1),
//   S(y) = sum 2k y^(k-1) = 2/(1-y)^2,
// with max relative errors 3.5e-9, 1.4e-8 and 1.8e-8 (gen_hct_poly.py derives
// the coefficients).
// Packed FP32: one float2 carries the same quantity for two pairs, and
// fma.rn.f32x2 / add / mul (sm_100 and later) work on both halves in one
// instruction.  The helpers below take float or float2 alike.
__device__ __forceinline__ float fma_p(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 fma_p(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
template <class T> __device__ __forceinline__ T splat(float v);
template <> __device__ __forceinline__ float splat<float>(float v) { return v; }
template <> __device__ __forceinline__ float2 splat<float2>(float v) { return make_float2(v, v); }

template <class T> __device__ __forceinline__ T hct_series_h(T y) { // P
    T p = splat<T>(1.361160215f);
    p = fma_p(p, y, splat<T>(0.8443080909f));
    p = fma_p(p, y, splat<T>(0.8931260308f));
    p = fma_p(p, y, splat<T>(0.8570198603f));
    p = fma_p(p, y, splat<T>(0.8000012903f));
    p = fma_p(p, y, splat<T>(0.6666666645f));
    return p;
}

template <class T> __device__ __forceinline__ T hct_series_dr(T y) { // Q
    T p = splat<T>(20.1395503f);
    p = fma_p(p, y, splat<T>(9.836372412f));
    p = fma_p(p, y, splat<T>(8.959016539f));
    p = fma_p(p, y, splat<T>(6.855114687f));
    p = fma_p(p, y, splat<T>(4.800021136f));
    p = fma_p(p, y, splat<T>(2.666666631f));
    return p;
}

template <class T> __device__ __forceinline__ T hct_series_ds(T y) { // S
    T p = splat<T>(18.77114444f);
    p = fma_p(p, y, splat<T>(8.994253274f));
    p = fma_p(p, y, splat<T>(8.065659941f));
    p = fma_p(p, y, splat<T>(5.998104684f));
    p = fma_p(p, y, splat<T>(4.0000197f));
    p = fma_p(p, y, splat<T>(1.999999967f));
    return p;
}

// Born-radius cutoff rc (AMBER's rgbmax; infinity = none): only shells
// t <= rc descreen, so U = min(r + s, rc), the covered shells of a ball inside
// sphere s end at min(s - r, rc), and H = 0 once L >= U.  The derivative forms
// below hold for a moving or a fixed U alike (the integrand vanishes on the
// moving boundaries), except that the covered-shell term stops moving with r
// and s once capped.  With the ball inside sphere s (L = s - r) the closed
// part's dependence on L cancels that of the covered shells, so dH/dr and
// dH/ds are the closed part's explicit partials alone; once the covered
// shells are capped at rc the closed part is empty and both vanish.
__device__ __forceinline__ bool hct_far(float r, float rt, float s, float rc = INFINITY) {
    return (r - s >= rt) && (s <= kHctXmax * r) && (r + s <= rc);
}

struct HctClosed {
    float iL, iU, lg;
};

__device__ __forceinline__ HctClosed hct_closed(float r, float rt, float s, float rc) {
    float U = fminf(r + s, rc);
    float L = fmaxf(rt, fabsf(r - s));
    float iLU = __fdividef(1.f, L * U);
    HctClosed h;
    h.iL = U * iLU;
    h.iU = L * iLU;
    h.lg = logf(L * h.iU); // accurate log: near pairs dominate psi, keep them to ~1 ulp
    return h;
}

// whether the closed-form part is empty (L >= U)
__device__ __forceinline__ bool hct_empty(float r, float rt, float s, float rc) {
    return fmaxf(rt, fabsf(r - s)) >= fminf(r + s, rc);
}

__device__ __forceinline__ float hct(float r, float rinv, float rt, float irt, float s, float rc = INFINITY) {
    if (hct_far(r, rt, s, rc)) {
        float x = s * rinv, y = x * x;
        return x * y * hct_series_h(y) * rinv;
    }
    float h = 0.f;
    if (!hct_empty(r, rt, s, rc)) {
        HctClosed c = hct_closed(r, rt, s, rc);
        h = (c.iL - c.iU) * fmaf((c.iL + c.iU) * 0.25f * rinv, (s - r) * (s + r), 1.f) + 0.5f * rinv * c.lg;
    }
    if (rt < s - r) {
        const float top = fminf(s - r, rc);
        if (rt < top) h += 2.f * (irt - __fdividef(1.f, top));
    }
    return h;
}

__device__ __forceinline__ float hct_dr(float r, float rinv, float rt, float s, float rc = INFINITY) {
    float rinv2 = rinv * rinv;
    if (hct_far(r, rt, s, rc)) {
        float x = s * rinv, y = x * x;
        return -x * y * hct_series_dr(y) * rinv2;
    }
    float d = 0.f;
    if (!hct_empty(r, rt, s, rc)) {
        HctClosed c = hct_closed(r, rt, s, rc);
        d = -0.25f * (c.iL - c.iU) * (c.iL + c.iU) * fmaf(s * s, rinv2, 1.f) - 0.5f * c.lg * rinv2;
    }
    return d;
}

// dH/dr with the fast logarithm (__logf) in the closed form: the chain-rule
// force of a near pair, where the log term is O(1) and its ~1e-7 absolute
// error stays far below the force bar.
__device__ __forceinline__ float hct_dr_fastlog(float r, float rinv, float rt, float s, float rc = INFINITY) {
    float rinv2 = rinv * rinv;
    if (hct_far(r, rt, s, rc)) {
        float x = s * rinv, y = x * x;
        return -x * y * hct_series_dr(y) * rinv2;
    }
    float d = 0.f;
    if (!hct_empty(r, rt, s, rc)) {
        const float U = fminf(r + s, rc), L = fmaxf(rt, fabsf(r - s));
        const float iLU = __fdividef(1.f, L * U), iL = U * iLU, iU = L * iLU;
        d = -0.25f * (iL - iU) * (iL + iU) * fmaf(s * s, rinv2, 1.f) - 0.5f * __logf(L * iU) * rinv2;
    }
    return d;
}

__device__ __forceinline__ float hct_ds(float r, float rinv, float rt, float s, float rc = INFINITY) {
    if (hct_far(r, rt, s, rc)) {
        float x = s * rinv, y = x * x;
        return y * hct_series_ds(y) * rinv * rinv;
    }
    float d = 0.f;
    if (!hct_empty(r, rt, s, rc)) {
        HctClosed c = hct_closed(r, rt, s, rc);
        d = 0.5f * s * rinv * (c.iL - c.iU) * (c.iL + c.iU);
    }
    return d;
}

__device__ __forceinline__ float hct_drt(float r, float rt, float irt, float s, float rc = INFINITY) {
    if (hct_far(r, rt, s, rc)) return 0.f;
    float d = 0.f;
    if (rt < s - r) {
        if (rt < fminf(s - r, rc)) d = -2.f * irt * irt;
    } else if (rt > fabsf(r - s) && !hct_empty(r, rt, s, rc)) {
        float a = rt - r;
        d = (a * a - s * s) * 0.5f * __fdividef(1.f, r) * irt * irt * irt;
    }
    return d;
}

// --------------------------------------- HCT, FP64, of the pair kernels
// The closed forms below with one reciprocal and the short logarithm.  r2 = r^2.
__device__ __forceinline__ double hct64(double r, double r2, double rinv, double rt, double irt, double s, double rc,
                                        const double2* tab) {
    const double U = fmin(r + s, rc), L = fmax(rt, fabs(r - s));
    double h = 0.0;
    if (L < U) {
        const double iLU = rcp64(L * U), iL = U * iLU, iU = L * iLU, q = 0.25 * rinv;
        h = fma(iL - iU, fma((iL + iU) * q, fma(s, s, -r2), 1.0), 0.5 * rinv * log64(L * iU, tab));
    }
    if (rt < s - r) {
        const double top = fmin(s - r, rc);
        if (rt < top) h += 2.0 * (irt - rcp64(top));
    }
    return h;
}

// - dH/dr
__device__ __forceinline__ double hct_mdr64(double r, double rinv2, double rt, double s, double rc, const double2* tab) {
    const double U = fmin(r + s, rc), L = fmax(rt, fabs(r - s));
    if (!(L < U)) return 0.0;
    const double iLU = rcp64(L * U), iL = U * iLU, iU = L * iLU;
    return fma(0.25 * ((iL - iU) * (iL + iU)), fma(s * s, rinv2, 1.0), 0.5 * rinv2 * log64(L * iU, tab));
}

// ------------------------------------------------------------- HCT, FP64
// Closed forms throughout (FP64 has no cancellation problem at these sizes);
// rc as above (infinity = no cutoff).
__device__ __forceinline__ double hct(double r, double rinv, double rt, double irt, double s, double rc = INFINITY) {
    const double U = fmin(r + s, rc), L = fmax(rt, fabs(r - s));
    double h = 0.0;
    if (L < U) {
        double iL = 1.0 / L, iU = 1.0 / U;
        h = (iL - iU) * (1.0 + (iL + iU) * 0.25 * rinv * (s - r) * (s + r)) + 0.5 * rinv * log(L * iU);
    }
    if (rt < s - r) {
        const double top = fmin(s - r, rc);
        if (rt < top) h += 2.0 * (irt - 1.0 / top);
    }
    return h;
}

// ------------------------------------------------- compensated summation
// Kahan summation of a tile's partial energies: the energy sums cancel
// strongly (sum |terms| >> |E|), so plain FP32 partials over a 128-atom tile
// would lose ~1e-6 of |E|.  FP64 needs no compensation.
template <class Real>
struct KSum {
    Real s = 0, c = 0;
    __device__ __forceinline__ void add(Real v) {
        const Real y = v - c;
        const Real t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ Real value() const { return s; }
};

template <>
struct KSum<float2> { // two sums, one value
    float2 s = {0.f, 0.f}, c = {0.f, 0.f};
    __device__ __forceinline__ void add(float2 v) {
        const float2 m = {-1.f, -1.f};
        const float2 y = __ffma2_rn(c, m, v);
        const float2 t = __fadd2_rn(s, y);
        c = __ffma2_rn(y, m, __ffma2_rn(s, m, t));
        s = t;
    }
    __device__ __forceinline__ float value() const {
        KSum<float> k;
        k.s = s.x;
        k.c = c.x + c.y;
        k.add(s.y);
        return k.s;
    }
};

template <>
struct KSum<double> {
    double s = 0;
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ double value() const { return s; }
};

// ------------------------------------------------------ precision traits
template <class Real>
struct Prec;

template <>
struct Prec<float> {
    using Acc = long long; // int64 fixed point
    __device__ static float rsqrt(float x) { return rsqrtf(x); }
    __device__ static float expm(float x) { return __expf(-x); } // e^-x
    __device__ static float recip(float x) { return __fdividef(1.f, x); }
    __device__ static void add(Acc& a, float part, float scale) { a += to_fixed(part, scale); }
    __device__ static double value(Acc a, double scale) { return (double)a / scale; }
};

template <>
struct Prec<double> {
    using Acc = double;
    __device__ static double rsqrt(double x) { return 1.0 / sqrt(x); }
    __device__ static double expm(double x) { return exp(-x); }
    __device__ static double recip(double x) { return 1.0 / x; }
    __device__ static void add(Acc& a, double part, double) { a += part; }
    __device__ static double value(Acc a, double) { return a; }
};

} // namespace cph
