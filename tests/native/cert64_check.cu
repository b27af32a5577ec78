// Host-side check of the float32 certificate of the Appendix-A positivity
// factor on float64 data beyond the range of a float, as the kernels pass it:
// cell averages and contributions cut by cgl::cert_float.  Whenever
// cgl::euler_alpha_is_one returns true, cgl::euler_alpha<double> on the float64
// data must return exactly 1.  Arguments: trials, then the decades (log10) of the
// density, of m and of m times the density between which they are drawn.
// Prints one JSON line: {"trials", "certified", "wrong"}.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>

#include "../../paper_2509_04673_gb300/csrc/common.cuh"

static uint64_t s_state = 0x2509046735ULL;
static uint64_t next_u64() {
    uint64_t z = (s_state += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
static double unif() { return (next_u64() >> 11) * 0x1p-53; }
static double logu(double lo, double hi) { return std::pow(10.0, lo + (hi - lo) * unif()); }

int main(int argc, char** argv) {
    const long trials = std::atol(argv[1]);
    const double r0 = std::atof(argv[2]), r1 = std::atof(argv[3]), m0 = std::atof(argv[4]), m1 = std::atof(argv[5]);
    const double eps = 1e-10;
    const float ome = (float)(1.0 - eps);
    long certified = 0, wrong = 0;
    for (long t = 0; t < trials; ++t) {
        const double rho = logu(r0, r1), pr = rho * logu(-6.0, 3.0);
        const double vx = (unif() - 0.5) * logu(-3.0, 1.0), vy = (unif() - 0.5) * logu(-3.0, 1.0);
        const double ub[4] = {rho, rho * vx, rho * vy, pr / 0.4 + 0.5 * rho * (vx * vx + vy * vy)};
        const double m = logu(m0, m1);
        const double scale = m * logu(-4.0, 2.0);
        double f[4];
        for (int c = 0; c < 4; ++c) f[c] = (unif() - 0.5) * scale * (c == 3 ? ub[3] : rho);
        if (t % 2) {
            // onto the edge of a constraint, or a little to either side
            const double a = cgl::euler_alpha<double>(ub, f, m, eps);
            if (a < 1.0 && a > 0.0) {
                const double off = std::pow(10.0, -(double)(next_u64() % 13)) * ((next_u64() & 1) ? 1.0 : -1.0);
                for (int c = 0; c < 4; ++c) f[c] *= a * (1.0 + off);
            }
        }
        if (t % 3 == 0) f[0] = -rho * m * (1.0 + 1e-3 * unif());  // just beyond an empty cell
        float ubf[4], ff[4];
        for (int c = 0; c < 4; ++c) {
            ubf[c] = cgl::cert_float(ub[c]);
            ff[c] = cgl::cert_float(f[c]);
        }
        if (!cgl::euler_alpha_is_one<double>(ubf, ff, t % 5 ? (float)m : cgl::cert_float(m), ome)) continue;
        ++certified;
        if (cgl::euler_alpha<double>(ub, f, m, eps) != 1.0 && ++wrong < 5)
            std::fprintf(stderr, "wrong: ub %.9g %.9g %.9g %.9g f %.9g %.9g %.9g %.9g m %.9g\n", ub[0], ub[1], ub[2],
                         ub[3], f[0], f[1], f[2], f[3], m);
    }
    std::printf("{\"trials\": %ld, \"certified\": %ld, \"wrong\": %ld}\n", trials, certified, wrong);
    return 0;
}
