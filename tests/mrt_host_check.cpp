// Host build of the fixed-point moments (lbm_collide_df.cuh), with the compiler's checks for
// undefined arithmetic on: which nodes the MRT collision takes in fixed point, its moments of
// those in long double (which holds them exactly), and sums of values that are refused.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_1611_02445_gb300/csrc/lbm_collide_df.cuh"

using namespace lbm;
typedef long double LD;
static const int CV[19][3] = {{0, 0, 0},  {1, 0, 0},   {0, 1, 0},  {-1, 0, 0}, {0, -1, 0}, {0, 0, 1},  {0, 0, -1},
                              {1, 1, 0},  {-1, 1, 0},  {-1, -1, 0}, {1, -1, 0}, {1, 0, 1},  {1, 0, -1}, {-1, 0, 1},
                              {-1, 0, -1}, {0, 1, 1},  {0, 1, -1}, {0, -1, 1}, {0, -1, -1}};

int main() {
    std::mt19937_64 rng(17);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    long taken = 0, wrong_choice = 0, wrong_moment = 0, wide = 0;
    for (int n = 0; n < 400000; n++) {
        double f[19];
        const int kind = n % 8;
        for (int i = 0; i < 19; i++) {
            const double w = i == 0 ? 1.0 / 3 : i < 7 ? 1.0 / 18 : 1.0 / 36;
            f[i] = kind < 3 ? w * (0.6 + 2.2 * U(rng))          // about the weights
                 : kind == 3 ? 0.1 + 0.1 * U(rng)                // a density about 3
                 : kind == 4 ? 1.5 + 0.5 * U(rng)                // a density of 28 to 38
                 : kind == 5 ? std::nextafter(2.0, 0.0)          // the largest, 38
                 : kind == 6 ? std::ldexp(1.0 + U(rng), (int)(rng() % 12) - 8)
                             : std::ldexp(U(rng) - 0.5, (int)(rng() % 2000) - 1000);
        }
        if (kind == 7) f[rng() % 19] = n & 8 ? INFINITY : NAN;
        bool in = true;
        LD rho = 0, j[3] = {0, 0, 0}, e = 0, eps = 0;
        for (int i = 0; i < 19; i++) {
            in = in && f[i] >= 0x1p-6 && f[i] < 2.0;
            const int cc = CV[i][0] * CV[i][0] + CV[i][1] * CV[i][1] + CV[i][2] * CV[i][2];
            rho += f[i];
            e += (LD)(19 * cc - 30) * f[i];
            eps += (LD)((21 * cc * cc - 53 * cc + 24) / 2) * f[i];
            for (int a = 0; a < 3; a++) j[a] += (LD)CV[i][a] * f[i];
        }
        if (in && rho >= 32) wide++;
        MrtMoments<int64_t> m;
        const bool ok = mrt_fix_moments(f, m);
        if (ok != (in && rho < 3)) wrong_choice++;
        if (ok) {
            taken++;
            const LD u = 0x1p-58L;
            if ((LD)m.rho * u != rho || fabsl((LD)m.n1 * u - (e + 11 * rho) / 19) > 1e-17L ||
                fabsl((LD)m.n2 * u - (eps - 3 * rho)) > 1e-16L)
                wrong_moment++;
            for (int a = 0; a < 3; a++)
                if ((LD)m.j[a] * u != j[a]) wrong_moment++;
        }
        // sums of values that the caller refuses
        int64_t q[19], r, x, y, z;
        bool bad = false;
        for (int i = 0; i < 19; i++) q[i] = fix_from_double_fast(f[i], bad);
        fix_moments(q, r, x, y, z);
        if (!bad && rho < 32 && (LD)r * 0x1p-58L != rho) wrong_moment++;
    }
    std::printf("taken %ld\nwide %ld\nwrong_choice %ld\nwrong_moment %ld\n", taken, wide, wrong_choice, wrong_moment);
    return 0;
}
