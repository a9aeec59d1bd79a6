// The closed-form draw's host branches (pm_fastdraw.cuh) against 64-bit running
// sums. Reads lines "K kappa rho_share seed n" (rho = rho_share rho_max) and
// prints, per line, whether a row is usable, how many of n draws with uniform u
// were left open, how many of n draws with u at a boundary were, how many
// answers were not the heading that the sums give, and the tolerance there.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "pm_fastdraw.cuh"

using namespace pm;

int main()
{
    int K, seed, n;
    double kappa, share;
    while (std::scanf("%d %lf %lf %d %d", &K, &kappa, &share, &seed, &n) == 5) {
        const double s = 0.05, pi = 3.14159265358979323846;
        const float beta = (float)(kappa / s);
        FastRow row;
        FastWork ws;
        FastPrep a{};
        a.beta = &beta;
        a.B = a.S = 1;
        a.K = K;
        a.w2 = 1.0f;
        a.sl[0] = (float)s;
        a.rows = &row;
        fast_row_build(a, 0, true, ws, 0, 1);
        if (row.rho_max <= 0.0f) {
            std::printf("0 0 0 0 0\n");
            continue;
        }
        FastConst fc{(float)std::cos(pi / K), (float)std::sin(pi / K), (float)(0.5 * K / pi), K};
        F2 q[kFastD][kFastP], P[kFastP];
        fast_load(row, q);
        std::mt19937_64 rng(seed);
        std::uniform_real_distribution<double> uni(0.0, 1.0);
        long open[2] = {0, 0}, wrong = 0;
        const float rho = (float)(share * row.rho_max);
        const float tolx = K * (row.tol + row.tol2 * rho * rho);
        fast_poly(q, rho, P);
        std::vector<double> C(K);
        for (int i = 0; i < 2 * n; ++i) {
            const double al = 2.0 * pi * uni(rng), r = (double)row.s / rho, ca = std::cos(al), sa = std::sin(al);
            double sum = 0.0;
            for (int k = 0; k < K; ++k) {
                const double c = std::cos(2.0 * pi * k / K - al), ss = row.s;
                const double h = (2.0 * r * c + ss) / (std::sqrt(r * r + 2.0 * r * ss * c + ss * ss) + r);
                C[k] = sum += std::exp(-(double)row.kappa * h);
            }
            double u = uni(rng);
            if (i & 1) { // at a boundary, up to two tolerances off it
                const int k = (int)(uni(rng) * K);
                u = C[k] / sum + (2.0 * uni(rng) - 1.0) * 2.0 * tolx / K;
                if (!(u >= 0.0 && u < 1.0)) continue;
            }
            const float uf = (float)(std::floor(u * 8388608.0) / 8388608.0 + 0x1p-25); // as rollout_lane forms it
            int want = 0;
            while (want < K - 1 && C[want] <= (double)uf * sum) ++want;
            FastDraw w = fast_begin(fc, P, (float)ca, (float)sa, uf, row.guess);
            int k = fast_step(fc, P, rho, row.kappa, tolx, w);
            if (k < 0 && std::fabs(w.dl) > 1e-4f) k = fast_step(fc, P, rho, row.kappa, tolx, w);
            if (k < 0) ++open[i & 1];
            else if (k != want) ++wrong;
        }
        std::printf("1 %ld %ld %ld %.9g\n", open[0], open[1], wrong, tolx / K);
    }
}
