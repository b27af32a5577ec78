// Device check of the arithmetic routines of common.cuh and modal.cuh that
// stand for hardware or library operations: reciprocals, square roots and the
// conversions between float and float64 in integer arithmetic.  One JSON line:
// per routine the largest error over a sweep of its range, in units of the last
// place of the result (against the correctly rounded operation in float64, or
// in float), and the results at zero, subnormals, the ends of the range and
// infinity as hexadecimal floats.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../paper_2509_04673_gb300/csrc/modal.cuh"

using namespace cgl;

enum { RCP_NR_D, RECIP_D, ROOT_D, RCP_NR_F, RECIP_F, ROOT_F, WIDEN, NARROW, SPLIT_HI, SPLIT_LO, N_OP };
static const char* const NAMES[N_OP] = {"rcp_nr_d", "recip_d", "root_d", "rcp_nr_f", "recip_f",
                                        "root_f",   "widen",   "narrow", "split_hi", "split_lo"};

static DEV double apply(int op, double x) {
    float hi, lo;
    switch (op) {
        case RCP_NR_D: return rcp_nr(x);
        case RECIP_D: return recip(x);
        case ROOT_D: return root(x);
        case RCP_NR_F: return (double)rcp_nr((float)x);
        case RECIP_F: return (double)recip((float)x);
        case ROOT_F: return (double)root((float)x);
        case WIDEN: return widen((float)x);
        case NARROW: return (double)narrow(x);
        default:
            split_ff(x, hi, lo);
            return op == SPLIT_HI ? (double)hi : (double)lo;
    }
}

static __global__ void k_apply(int op, const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = apply(op, x[i]);
}

static uint64_t s_state = 0x2509046733ULL;
static uint64_t next_u64() {
    uint64_t z = (s_state += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

static std::vector<double> run(int op, const std::vector<double>& x) {
    const int n = (int)x.size();
    std::vector<double> y(n);
    double *dx, *dy;
    if (cudaMalloc(&dx, n * 8) != cudaSuccess || cudaMalloc(&dy, n * 8) != cudaSuccess) return {};
    cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice);
    k_apply<<<(n + 255) / 256, 256>>>(op, dx, dy, n);
    const cudaError_t e = cudaMemcpy(y.data(), dy, n * 8, cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dy);
    return e == cudaSuccess ? y : std::vector<double>();
}

// |y - exact| in units of the last place of a float64 or float result
static double ulps(double y, long double exact, bool f32) {
    if (std::isnan(y) || std::isinf(y)) return 1e30;
    int e;
    std::frexp((double)exact, &e);
    return (double)(std::fabs((long double)y - exact) / std::ldexp(1.0L, e - (f32 ? 24 : 53)));
}

int main() {
    const int n = 1 << 20;
    std::string out = "{";
    char buf[256];
    for (int op = 0; op < N_OP; ++op) {
        const bool f32 = op == RCP_NR_F || op == RECIP_F || op == ROOT_F;
        std::vector<double> x(n);
        for (int i = 0; i < n; ++i) {
            // mantissa and exponent uniform over the normal range whose result is normal
            const int lo = f32 || op == WIDEN || op == NARROW ? -125 : op >= SPLIT_HI ? -73 : -1020;
            const int hi = f32 || op == WIDEN || op == NARROW || op >= SPLIT_HI ? 125 : 1020;
            const int ex = lo + (int)(next_u64() % (uint64_t)(hi - lo + 1));
            double m = 1.0 + (next_u64() >> 12) * 0x1p-52;
            if (f32 || op == WIDEN) m = (double)(float)m >= 2.0 ? 1.0 : (double)(float)m;
            x[i] = std::ldexp(m, ex);
            const bool sign = op != ROOT_D && op != ROOT_F && op != RECIP_D && op != RECIP_F;
            if (sign && (next_u64() & 1)) x[i] = -x[i];
        }
        const std::vector<double> y = run(op, x);
        if ((int)y.size() != n) {
            std::fprintf(stderr, "launch failed\n");
            return 1;
        }
        std::vector<double> lo;
        if (op == SPLIT_HI) lo = run(SPLIT_LO, x);
        double worst = 0.0, worst_pair = 0.0;
        for (int i = 0; i < n; ++i) {
            const long double v = x[i];
            double d = 0.0;
            switch (op) {
                case RCP_NR_D: case RECIP_D: case RCP_NR_F: case RECIP_F: d = ulps(y[i], 1.0L / v, f32); break;
                case ROOT_D: case ROOT_F: d = ulps(y[i], std::sqrt(v), f32); break;
                case WIDEN: d = y[i] == x[i] ? 0.0 : 1e30; break;
                case NARROW:
                    // towards zero, to 24 bits
                    d = ulps(y[i], v, true);
                    if (std::fabs(y[i]) > std::fabs(x[i])) d = 1e30;
                    break;
                case SPLIT_HI: {
                    d = ulps(y[i], v, true);
                    int e;
                    std::frexp(x[i], &e);
                    const double pr = (double)(std::fabs((long double)y[i] + lo[i] - v) / std::ldexp(1.0L, e - 53));
                    worst_pair = pr > worst_pair ? pr : worst_pair;
                    break;
                }
                default: break;
            }
            worst = d > worst ? d : worst;
        }
        std::snprintf(buf, sizeof buf, "\"%s\": %.6g, ", NAMES[op], worst);
        out += buf;
        if (op == SPLIT_HI) {
            std::snprintf(buf, sizeof buf, "\"split_pair\": %.6g, ", worst_pair);
            out += buf;
        }
    }
    // points of interest
    const std::vector<double> px = {0.0, 0x1p-1074, 1e-320, 1e-312, 0x1.fffffp-1023, 0x1p-1022, 0x1p-600, 0x1p-149, 0x1p-130,
                                    0x1.8p-127, 0x1p-126, 1.0, 0x1p126, 0x1.fp127, 0x1p1000, 0x1p1022, 0x1.8p1023, INFINITY};
    out += "\"points\": {";
    for (int op = 0; op < SPLIT_HI; ++op) {
        const std::vector<double> y = run(op, px);
        std::snprintf(buf, sizeof buf, "\"%s\": [", NAMES[op]);
        out += buf;
        for (size_t i = 0; i < px.size(); ++i) {
            std::snprintf(buf, sizeof buf, "[\"%a\", \"%a\"]%s", px[i], y[i], i + 1 < px.size() ? ", " : "");
            out += buf;
        }
        out += op + 1 < SPLIT_HI ? "], " : "]";
    }
    out += "}}";
    std::puts(out.c_str());
    return 0;
}
