// Prints the sensor's modal tables (modal_tables.h): lines "name basis p i j value"
// with the value as a hexadecimal float.
#include <cmath>
#include <cstdio>

#include "../../paper_2509_04673_gb300/csrc/modal_tables.h"

int main() {
    for (int basis = 0; basis < 2; ++basis)
        for (int p = 1; p <= cgl::PMAX; ++p) {
            // LGL points on [0, 1]: 0, 1 and (1 -+ z) / 2
            const double z = p == 3 ? 1.0 / std::sqrt(5.0) : std::sqrt(3.0 / 7.0);
            const double x1[] = {0.0, 1.0}, x2[] = {0.0, 0.5, 1.0}, x3[] = {0.0, 0.5 - 0.5 * z, 0.5 + 0.5 * z, 1.0};
            const double x4[] = {0.0, 0.5 - 0.5 * z, 0.5, 0.5 + 0.5 * z, 1.0};
            const double* const x[] = {nullptr, x1, x2, x3, x4};
            static cgl::ModalTables T;
            cgl::modal_tables(p, basis ? x[p] : nullptr, T);
            const int n = p + 1, n2 = n * n;
            for (int k = 0; k < n; ++k)
                for (int j = 0; j < 2; ++j) std::printf("mf %d %d %d %d %a\n", basis, p, k, j, T.mf[k][j]);
            for (int k = 0; k < n; ++k)
                for (int j = 0; j < n; ++j) std::printf("mc %d %d %d %d %a\n", basis, p, k, j, T.mc[k][j]);
            for (int i = 0; i < n2; ++i)
                for (int j = 0; j < n2; ++j) std::printf("m2 %d %d %d %d %a\n", basis, p, i, j, T.m2[i * n2 + j]);
        }
    return 0;
}
