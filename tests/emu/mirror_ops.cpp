// Host check of the mirror symmetry of the translation operators: every
// operator entry against the signed entry of the operator at the mirrored
// (all-positive) position, s_o(chi_i) s_o(chi_j) T_+[i][j], and the triangle of
// the M2M and the L2L.  Prints the largest deviation per operator kind and the
// largest entry outside the triangle.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "fmm_math.cuh"

using namespace gf;

static int degree(int k) {
    int n = 0;
    while ((n + 1) * (n + 1) <= k) ++n;
    return n;
}

static int parity(int k) {
    const int n = degree(k), ro = k - n * n, m = (ro + 1) >> 1, im = (ro > 0 && (ro & 1) == 0) ? 1 : 0;
    return ((m + im) & 1) | (im << 1) | (((n + m) & 1) << 2);
}

int main(int argc, char **argv) {
    const int p = argc > 1 ? atoi(argv[1]) : 6, K = (p + 1) * (p + 1);
    double lf[kLogFactN];
    for (int i = 0; i < kLogFactN; ++i) lf[i] = lgamma(i + 1.0);
    auto op = [&](int kind, double x, double y, double z, std::vector<double> &T) {
        const int H = kind == OP_M2L ? 2 * p : p, nt = (H + 1) * (H + 2) / 2;
        std::vector<double> re(nt), im(nt);
        if (kind == OP_M2L)
            irregular_harmonics<double>(H, x, y, z, re.data(), im.data());
        else
            regular_harmonics<double>(H, x, y, z, re.data(), im.data());
        T.resize((size_t)K * K);
        for (int i = 0; i < K; ++i)
            for (int j = 0; j < K; ++j) T[(size_t)i * K + j] = op_entry(kind, p, i, j, re.data(), im.data(), lf);
    };
    double worst[3] = {0, 0, 0}, outside = 0;
    std::vector<double> A, B;
    const double off[3][3] = {{0.25, 0.25, 0.25}, {1, 2, 3}, {3, 0, 2}};
    for (int kind = 0; kind < 3; ++kind)
        for (int c = 0; c < (kind == OP_M2L ? 3 : 1); ++c) {
            const double *d = kind == OP_M2L ? off[c] : off[0];
            op(kind, d[0], d[1], d[2], B);
            for (int o = 0; o < 8; ++o) {
                op(kind, (o & 1) ? d[0] : -d[0], (o & 2) ? d[1] : -d[1], (o & 4) ? d[2] : -d[2], A);
                for (int i = 0; i < K; ++i)
                    for (int j = 0; j < K; ++j) {
                        const int s = __builtin_popcount((parity(i) ^ parity(j)) & ~o & 7) & 1;
                        const double b = B[(size_t)i * K + j];
                        worst[kind] = std::max(worst[kind], fabs(A[(size_t)i * K + j] - (s ? -b : b)));
                        if (kind == OP_M2M && degree(j) > degree(i)) outside = std::max(outside, fabs(A[(size_t)i * K + j]));
                        if (kind == OP_L2L && degree(j) < degree(i)) outside = std::max(outside, fabs(A[(size_t)i * K + j]));
                    }
            }
        }
    printf("%.3e %.3e %.3e %.3e\n", worst[0], worst[1], worst[2], outside);
    return 0;
}
