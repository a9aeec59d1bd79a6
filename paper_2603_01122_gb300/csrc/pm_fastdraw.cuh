// pm_fastdraw.cuh -- the inverse CDF of Eq. 2 over equally spaced headings in
// closed form (private to the library).
//
// With z - g = r (cos al, sin al), s the step and rho = s / r, the distance
// after heading theta is d = r + s h(theta - al), and the weight of a heading,
// up to a factor common to all of them, is the even function
//   w(E) = exp(-kappa h(E)),  E = theta - al,  kappa = beta w2 s,
//   h = (2 cos E + rho) / (1 + sqrt(1 + 2 rho cos E + rho^2)).
// Its Fourier series sum_n a_n cos nE converges like kappa^n / (2^n n!), and
// the sum of each harmonic over headings 0..k is elementary, so the running
// sums of the K weights are values of ONE smooth function at K points:
//   C_k / C_{K-1} = [F(E_k + pi/K) - F(E_0 - pi/K)] / 2 pi,
//   F(E) = E + sin E P(cos E; rho)
// with P of degree 7 in cos E (the harmonics n <= 8, written as monomials) and
// its coefficients cubic in rho. The heading that holds the threshold u is
// floor(x) with F(2 pi x / K - pi/K - al) = F(-pi/K - al) + 2 pi u: a table of
// F^-1 gives the starting point and one third-order step the solution, about
// 110 instructions whatever K is, where forming the K weights takes 10 K.
//
// The result is used only where x lies clear of a whole number by more than
// the error of this evaluation and of the weight-by-weight draw together
// (`tol` below); the lanes that are closer take the weight-by-weight draw, so
// the chosen heading is always the one that the fixed-point weights give. They
// are 2 K tol of the draws: one in 4600 at K = 36 and small kappa, one in 4000
// at kappa = 2, in 750 at 2.5 and in 45 at 3, where the table starts too far
// off on the improbable side. A goal so far away that those weights lose bits
// keeps the weight-by-weight draw (comp_flags).
#pragma once

#include "pm_internal.cuh"

namespace pm {

constexpr int kFastM = 8;          // harmonics kept (degree of P plus one)
constexpr int kFastD = 4;          // coefficients in rho (cubic)
constexpr int kFastGuess = 64;     // intervals of the F^-1 table
constexpr int kFastQ = 12;         // quadrature intervals on [0, pi]: harmonic n is aliased by 24 - n only
constexpr int kFastMaxB = 16;      // beta values with a row; models with more use the weight-by-weight draw
constexpr int kFastMinK = 20;      // fewer controls: the weights themselves are as cheap
// Beyond it eight harmonics are not enough: at 3 (beta = 100, w2 = 1 and a step
// of 3 cm reach it) they are off by 3e-5 of the CDF. One lane whose beta lies
// beyond keeps its whole warp on the weight-by-weight draw, and the components
// of a warp are drawn independently: where 7 % of the belief is on such beta,
// 0.93^32 = 10 % of the warps still take the closed form.
constexpr float kFastMaxKappa = 3.0f;
constexpr int kFastGroup = 64;     // threads that build one row

// One (beta, speed): what a draw needs of it.
struct __align__(16) FastRow {
    float q[kFastD][kFastM]; // coefficient of rho^d cos^m E in P
    float a0[kFastD];        // mean weight over the headings, times the speed's factor exp(-beta w1 v dt (m - m_0))
    float kappa, tol, tol2, s; // tolerance tol + tol2 rho^2
    float2 guess[kFastGuess];     // F^-1 at 2 pi j / kFastGuess, and the step to the next
    float rho_max;                // largest rho of the fit; -1: the row is not usable
    float pad[3]; // an odd number of 16-byte words: rows of different lanes lie in different banks
};

struct FastPrep {
    const float *beta;
    int B, S;                    // rows b * S + q, b < B <= kFastMaxB, q the rank of a speed among the enabled ones
    int K;
    float w2, w1;                // Q weights
    float sl[PM_MAX_SPEEDS];     // step lengths of the enabled speeds (one speed: sl[0])
    FastRow *rows;
};

// Whether a control set takes the closed-form draw: every heading enabled, at
// least 16 of them (fewer alias the harmonics kept), and enough controls
// (S = 0 or 1: one speed).
__host__ __device__ __forceinline__ bool fast_applies(int K, uint64_t enabled, int S)
{
    const uint64_t all = K >= 64 ? ~0ull : ((1ull << K) - 1ull);
    return K >= 16 && K * (S > 1 ? S : 1) >= kFastMinK && (enabled & all) == all;
}

// Whether one human's call is long enough to repay its rows. Building them is
// one serial chain of some 4 us beside the zeroing and 6 us in a launch of its
// own (own_launch); what a step gives back grows with the weights that it need
// not form, and with the tiles per scheduler once each has one. In units of what
// a step of the fused one-speed draw gives back (K = 36, or one enabled speed of
// several with K = 32 or 36), other draws give three, and four from 64 controls
// of several speeds. Both sides at the line, rows / no rows in us, one human of
// N particles waited for:
//   K = 36, N = 1000: 24 steps 37 / 35, 32 steps 41 / 40, 48 steps 50 / 51
//   K = 36, N = 100,000: 5 steps 33 / 32, 8 steps 36 / 38
//   K = 20, N = 1000: 8 steps 28 / 26, 12 steps 29 / 30, 16 steps 32 / 33
//   3 x 32, N = 1000: 5 steps 36 / 33, 8 steps 39 / 43
__host__ __forceinline__ bool fast_fused(int K, int speeds, int speeds_on)
{
    return speeds_on <= 1 && (K == 36 || (speeds > 1 && K == 32));
}

__host__ __forceinline__ bool fast_pays(int K, int speeds, int speeds_on, int64_t tiles, int sm_count, int steps,
                                        bool own_launch)
{
    const float gain = fast_fused(K, speeds, speeds_on) ? 1.0f : (speeds_on > 1 && K * speeds_on >= 64) ? 4.0f : 3.0f;
    const float per_scheduler = (float)tiles / (4.0f * (float)(sm_count > 0 ? sm_count : 1));
    return (float)steps * gain * fminf(fmaxf(per_scheduler, 1.0f), 4.0f) >= (own_launch ? 48.0f : 32.0f);
}

// The same for a batch, whose rows take a launch of their own and cost the
// rollout its early launch (8 us). From 100 tiles on several warps share a
// scheduler (a CTA takes four tiles at a time), and a step gives back twice as
// much; beyond six tiles per scheduler it grows with them. The line lies half
// above the break-even: where no warp can use the rows (|kappa| > 3, which the
// host does not see) the 8 us are lost. Rows / no rows in us, one call after
// another, humans x particles:
//   K = 36: 1 x 1000, 32 steps 39 / 40, 64 steps 59 / 71; 4 x 1000, 16 steps
//     33 / 35, 24 steps 40 / 48; 16 x 8000, 16 steps 48 / 49, 24 steps 58 / 66
//   K = 20: 4 x 1000, 8 steps 26 / 26, 12 steps 30 / 35; 64 x 8000, 5 steps 63 / 80
//   K = 64: 4 x 1000, 8 steps 27 / 30, 12 steps 31 / 40
//   2 x 16: 4 x 1000, 12 steps 33 / 33, 16 steps 36 / 41; 16 x 8000, 12 steps 63 / 63
//   3 x 32: 1 x 1000, 8 steps 33 / 35, 16 steps 38 / 59; 4 x 8000, 8 steps 40 / 47
__host__ __forceinline__ bool fast_pays_batch(int K, int speeds, int speeds_on, int64_t tiles, int sm_count, int steps)
{
    const float gain = fast_fused(K, speeds, speeds_on) ? 1.0f
                       : speeds_on > 1 ? (float)(K * speeds_on) * (1.0f / 32.0f) + 0.5f
                       : (K <= 24 || K == 64) ? 2.0f
                                              : 4.0f;
    const float per_scheduler = (float)tiles / (4.0f * (float)(sm_count > 0 ? sm_count : 1));
    return (float)steps * gain * fmaxf(tiles >= 100 ? 2.0f : 1.0f, per_scheduler * (1.0f / 3.0f)) >= 48.0f;
}

#ifdef __CUDA_ARCH__
#define PM_FAST_SYNC() __syncthreads()
#else
#define PM_FAST_SYNC() ((void)0)
#endif

__host__ __device__ __forceinline__ float fast_sinf(float x)
{
#ifdef __CUDA_ARCH__
    return __sinf(x);
#else
    return sinf(x);
#endif
}

__host__ __device__ __forceinline__ float fast_cosf(float x)
{
#ifdef __CUDA_ARCH__
    return __cosf(x);
#else
    return cosf(x);
#endif
}

__host__ __device__ __forceinline__ float fast_rcp(float x)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}

__host__ __device__ __forceinline__ float fast_rsqrt(float x)
{
#ifdef __CUDA_ARCH__
    return rsqrt_approx(x);
#else
    return 1.0f / sqrtf(x);
#endif
}

// Coefficient of c^m in the Chebyshev polynomial U_n(c), n < kFastM:
// (-1)^j binomial(n - j, j) 2^(n - 2j) with m = n - 2j.
__host__ __device__ __forceinline__ float fast_u(int n, int m)
{
    const int j2 = n - m;
    if (j2 < 0 || (j2 & 1)) return 0.0f;
    const int j = j2 >> 1;
    float v = (j & 1) ? -1.0f : 1.0f;
    for (int i = 0; i < j; ++i) v = v * (float)(n - j - i) / (float)(i + 1);
    return ldexpf(v, m);
}

// Workspace of one row while it is built.
struct FastWork {
    float w[kFastD][kFastQ + 1];      // weights at the quadrature points, per node in rho
    float c[kFastD][kFastM + 1];      // [0]: mean; [n]: coefficient of sin nE in F
    float P[kFastD][kFastM];          // the same as monomials
    float p[kFastM];                  // P at the table's rho
    float g[kFastGuess / 2 + 1];      // F^-1 on [0, pi]
};

// The largest rho that a row is fitted on: there the eight harmonics and the
// cubic fit are off by 2e-6 of the CDF for kappa <= 1, 7e-6 at 2 and 3e-5 at 3
// (K = 16, against 64-bit running sums), by less and less towards rho = 0.
__host__ __device__ __forceinline__ float fast_rho_max(float kappa)
{
    return fminf(0.35f, 0.3f * fast_rsqrt(fmaxf(fabsf(kappa), 0.1f)));
}

// Builds row `row` of `a` with `nthr` threads (tid < nthr); every thread of
// the block calls it (it synchronises), `live` false for a group without a row.
__host__ __device__ __forceinline__ void fast_row_build(const FastPrep &a, int row, bool live, FastWork &ws, int tid,
                                                        int nthr)
{
    constexpr float kPi = 3.14159265358979f;
    const float t[kFastD] = {0.0380602337f, 0.308658284f, 0.691341716f, 0.961939766f}; // Chebyshev nodes of [0, 1]
    const int b = row / a.S, sp = row - b * a.S;
    const float beta = a.beta[b], s = a.sl[sp];
    const float kappa = beta * a.w2 * s;
    const float spd = -beta * a.w1 * (s - a.sl[0]); // log weight of the speed against the first one
    const bool ok = fabsf(kappa) <= kFastMaxKappa && fabsf(spd) <= 4.0f;
    const float kap = ok ? kappa : 0.0f, rmax = fast_rho_max(kap);
    for (int i = tid; i < kFastD * (kFastQ + 1); i += nthr) {
        const int d = i / (kFastQ + 1), j = i - d * (kFastQ + 1);
        const float rho = t[d] * rmax, c = cospif((float)j * (1.0f / (float)kFastQ));
        const float h = (2.0f * c + rho) / (1.0f + sqrtf(fmaf(rho, 2.0f * c + rho, 1.0f)));
        ws.w[d][j] = expf(-kap * h) * ((j == 0 || j == kFastQ) ? 0.5f : 1.0f);
    }
    PM_FAST_SYNC();
    for (int i = tid; i < kFastD * (kFastM + 1); i += nthr) {
        const int d = i / (kFastM + 1), n = i - d * (kFastM + 1);
        float acc = 0.0f;
        for (int j = 0; j <= kFastQ; ++j) {
            const int ph = (n * j) % (2 * kFastQ);
            acc = fmaf(ws.w[d][j], cospif((float)ph * (1.0f / (float)kFastQ)), acc);
        }
        ws.c[d][n] = acc * ((n == 0 ? 1.0f : 2.0f) / (float)kFastQ);
    }
    PM_FAST_SYNC();
    // sum_n c_n sin nE = sin E sum_n c_n U_{n-1}(cos E)
    for (int i = tid; i < kFastD * kFastM; i += nthr) {
        const int d = i / kFastM, m = i - d * kFastM;
        float acc = 0.0f;
        for (int n = 1; n <= kFastM; ++n) {
            const float hn = (float)n / (float)a.K;
            acc = fmaf(ws.c[d][n] * (kPi / ((float)a.K * sinpif(hn))), fast_u(n - 1, m), acc);
        }
        ws.P[d][m] = acc / ws.c[d][0];
    }
    PM_FAST_SYNC();
    const float rt = 0.25f; // the table's rho, as a share of rho_max
    for (int m = tid; m <= kFastM; m += nthr) { // m == kFastM: the mean
        float f[kFastD];
        for (int d = 0; d < kFastD; ++d) f[d] = m < kFastM ? ws.P[d][m] : ws.c[d][0] * expf(ok ? spd : 0.0f);
        // divided differences, then monomials in t
        const float f01 = (f[1] - f[0]) / (t[1] - t[0]), f12 = (f[2] - f[1]) / (t[2] - t[1]);
        const float f23 = (f[3] - f[2]) / (t[3] - t[2]);
        const float f012 = (f12 - f01) / (t[2] - t[0]), f123 = (f23 - f12) / (t[3] - t[1]);
        const float f3 = (f123 - f012) / (t[3] - t[0]);
        const float c0 = f[0] - t[0] * (f01 - t[1] * (f012 - t[2] * f3));
        const float c1 = f01 - (t[0] + t[1]) * f012 + (t[0] * t[1] + t[0] * t[2] + t[1] * t[2]) * f3;
        const float c2 = f012 - (t[0] + t[1] + t[2]) * f3;
        if (m < kFastM) ws.p[m] = fmaf(fmaf(fmaf(f3, rt, c2), rt, c1), rt, c0);
        if (live) {
            FastRow &o = a.rows[row];
            const float ir = 1.0f / rmax;
            float *dst = m < kFastM ? &o.q[0][m] : &o.a0[0];
            const int st = m < kFastM ? kFastM : 1;
            dst[0] = c0;
            dst[st] = c1 * ir;
            dst[2 * st] = c2 * ir * ir;
            dst[3 * st] = f3 * ir * ir * ir;
            if (m == kFastM) {
                o.kappa = kap;
                o.rho_max = ok ? rmax : -1.0f;
                // the FP32 arithmetic of both draws, the 2^-22 of ex2.approx and
                // the 2^-24 weights, and twice the fit's own error
                const float k3 = fabsf(kap) * (1.0f / 3.0f), k4 = k3 * k3 * k3 * k3;
                o.tol = 3.0e-6f + 8.0e-6f * k4 * k3 * k3;
                o.tol2 = (4.0e-6f + 6.0e-5f * k4 * sqrtf(k3)) / (rmax * rmax);
                o.s = s;
            }
        }
    }
    PM_FAST_SYNC();
    for (int j = tid; j <= kFastGuess / 2; j += nthr) {
        const float m = kPi * (float)j / (float)(kFastGuess / 2);
        float lo = 0.0f, hi = kPi, E = m;
        // Newton's method kept inside a bracket (F is increasing); the table only starts the draw's own step
        for (int it = 0; it < 8; ++it) {
            const float c = fast_cosf(E), sn = fast_sinf(E);
            float p = ws.p[kFastM - 1], dp = 0.0f;
            for (int i = kFastM - 2; i >= 0; --i) {
                dp = fmaf(dp, c, p);
                p = fmaf(p, c, ws.p[i]);
            }
            const float r = E + sn * p - m, fp = 1.0f + c * p - sn * sn * dp;
            if (r > 0.0f) hi = E;
            else lo = E;
            const float e = fmaf(-r, fast_rcp(fp), E);
            E = (e > lo && e < hi) ? e : 0.5f * (lo + hi);
        }
        ws.g[j] = (j == 0) ? 0.0f : (j == kFastGuess / 2) ? kPi : E;
    }
    PM_FAST_SYNC();
    for (int j = tid; live && j < kFastGuess; j += nthr) {
        constexpr int h = kFastGuess / 2;
        const float v0 = j <= h ? ws.g[j] : 2.0f * kPi - ws.g[kFastGuess - j];
        const float v1 = j + 1 <= h ? ws.g[j + 1] : 2.0f * kPi - ws.g[kFastGuess - j - 1];
        a.rows[row].guess[j] = make_float2(v0, v1 - v0);
    }
    PM_FAST_SYNC(); // the workspace may be used again
}

// Two FP32 values side by side (packed arithmetic on the device).
struct F2 {
    float x, y;
};

__host__ __device__ __forceinline__ F2 f2_madd(F2 a, F2 b, F2 c) // a b + c
{
#ifdef __CUDA_ARCH__
    F2 r;
    f2_unpack(f2_fma(f2_pack(a.x, a.y), f2_pack(b.x, b.y), f2_pack(c.x, c.y)), r.x, r.y);
    return r;
#else
    return F2{fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)};
#endif
}

// P at one rho: its coefficients in pairs (c^0, c^1), (c^2, c^3), ...
constexpr int kFastP = kFastM / 2;

__host__ __device__ __forceinline__ void fast_poly(const F2 (&q)[kFastD][kFastP], float rho, F2 (&P)[kFastP])
{
    const F2 r{rho, rho};
#pragma unroll
    for (int m = 0; m < kFastP; ++m) P[m] = f2_madd(f2_madd(f2_madd(q[3][m], r, q[2][m]), r, q[1][m]), r, q[0][m]);
}

__host__ __device__ __forceinline__ void fast_load(const FastRow &row, F2 (&q)[kFastD][kFastP])
{
#pragma unroll
    for (int d = 0; d < kFastD; ++d)
#pragma unroll
        for (int m = 0; m < kFastP; m += 2) {
            const float4 v = *reinterpret_cast<const float4 *>(&row.q[d][2 * m]);
            q[d][m] = F2{v.x, v.y};
            q[d][m + 1] = F2{v.z, v.w};
        }
}

// floor(v) for |v| < 2^22 without the conversion unit: v + 1.5 2^23 rounded
// down holds it in the low bits of the sum. Returns it as an integer, f as a float.
__host__ __device__ __forceinline__ int fast_floor(float v, float &f)
{
#ifdef __CUDA_ARCH__
    const float m = __fadd_rd(v, 12582912.0f);
    f = m - 12582912.0f;
    return __float_as_int(m) - 0x4B400000;
#else
    f = floorf(v);
    return (int)f;
#endif
}

// One draw in progress: F's argument at the first heading's lower boundary and
// the value it must reach.
struct FastDraw {
    float ce, se; // cos, sin of E0 = -pi/K - al
    float tau;    // F(E0) - E0 + 2 pi u
    float phi;    // the solution so far, E - E0
    float dl;     // last correction
};

// Starts the draw of the heading that holds the fraction u in [0, 1) of the
// running sums. (ca, sa) = (z - g) / r; P the polynomial at this rho; guess
// the row's table. P is evaluated as its even and odd part in c^2, side by
// side: half the instructions and half the chain of Horner's rule.
__host__ __device__ __forceinline__ FastDraw fast_begin(const FastConst &fc, const F2 (&P)[kFastP], float ca, float sa,
                                                        float u, const float2 *guess)
{
    constexpr float kPi = 3.14159265358979f, kTwoPi = 6.28318530717959f;
    FastDraw w;
    w.ce = fmaf(fc.cK, ca, -fc.sK * sa);
    w.se = -fmaf(fc.sK, ca, fc.cK * sa);
    const F2 e2{w.ce * w.ce, w.ce * w.ce};
    const F2 p = f2_madd(f2_madd(f2_madd(P[3], e2, P[2]), e2, P[1]), e2, P[0]);
    w.tau = fmaf(w.se, fmaf(w.ce, p.y, p.x), kTwoPi * u);
    // E0 to about 1e-4, for the starting point only: asin of the smaller component by its odd minimax polynomial
    const float ax = fabsf(w.ce), ay = fabsf(w.se), mn = fminf(ax, ay), m2 = mn * mn;
    float e0 = mn * fmaf(m2, fmaf(m2, fmaf(m2, 0.1066f, 0.0535f), 0.1686f), 0.99998f);
    e0 = ax < ay ? 0.5f * kPi - e0 : e0;
    e0 = w.ce < 0.0f ? kPi - e0 : e0;
    e0 = copysignf(e0, w.se);
    float turns, fl;
    const float t = (e0 + w.tau) * (1.0f / kTwoPi);
    fast_floor(t, turns);
    const float tn = (t - turns) * (float)kFastGuess;
    const float2 g = guess[fast_floor(tn, fl) & (kFastGuess - 1)];
    w.phi = fmaf(kTwoPi, turns, fmaf(tn - fl, g.y, g.x) - e0);
    return w;
}

// One third-order step of the draw; the heading, or -1 where the solution is
// too close to a boundary for tolx (K times a fraction of the running total) and
// the step's own error.
__host__ __device__ __forceinline__ int fast_step(const FastConst &fc, const F2 (&P)[kFastP], float rho, float kappa,
                                                  float tolx, FastDraw &w)
{
    const float cp = fast_cosf(w.phi), sp = fast_sinf(w.phi);
    const float c = fmaf(w.ce, cp, -w.se * sp), sn = fmaf(w.se, cp, w.ce * sp);
    const F2 c2{c * c, c * c};
    F2 v = f2_madd(P[3], c2, P[2]);
    F2 d = f2_madd(P[3], c2, v);
    v = f2_madd(v, c2, P[1]);
    d = f2_madd(d, c2, v);
    v = f2_madd(v, c2, P[0]);
    const float q = fmaf(c, v.y, v.x);                    // P(c)
    const float dq = fmaf(c + c, fmaf(c, d.y, d.x), v.y); // P'(c)
    const float f = fmaf(c, q, fmaf(-sn * sn, dq, 1.0f)); // F'
    const float inv = fast_rcp(f);
    w.dl = (fmaf(sn, q, w.phi) - w.tau) * inv;
    const float dl2 = w.dl * w.dl;
    // F''/F' = kappa sin E up to O(rho, 1/K^2)
    w.phi -= fmaf(0.5f * kappa * sn, dl2, w.dl);
    const float x = w.phi * fc.K2pi, ak = fabsf(kappa);
    float kf;
    const int k = fast_floor(x, kf);
    const float fr = x - kf;
    const float e = ak * dl2 * fmaf(ak + 0.5f, fabsf(w.dl), fmaf(2.0f, rho, 0.1f)); // error of the step
    const float band = fmaf(tolx, inv, e * fc.K2pi);
    // inv > 0 holds wherever the fit is good; NaN anywhere fails the test
    const bool ok = fminf(fr, 1.0f - fr) > band && inv > 0.0f && (unsigned)k < (unsigned)fc.K;
    return ok ? k : -1;
}

} // namespace pm
