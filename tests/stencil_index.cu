// Host check of the stencil's index arithmetic on boxes just below 2^31 unknowns:
// every neighbour inside the box has its exact index, every other one an index in
// range, and the grid-stride loop's step past the last unknown does not wrap.
#include <cstdio>

#include "pcg.cuh"
#include "q1.cuh"

int main() {
    const long long box[][3] = {{2147483647, 1, 1}, {1, 2147483647, 1}, {46340, 46341, 1}, {1290, 1290, 1290},
                                {3, 5, 143165576}, {1000, 1000, 2147}, {2, 2, 536870911}, {1073741823, 2, 1},
                                {7, 5, 3}, {1, 1, 1}};
    int bad = 0;
    for (const auto& s : box)
        for (int dim = 2; dim <= 3; ++dim) {
            if (dim == 2 && s[2] != 1) continue;
            const long long nun = s[0] * s[1] * s[2];
            const unsigned n = (unsigned)nun, sy = (unsigned)s[0], sz = sy * (unsigned)s[1];
            const long long at[] = {0, 1, s[0] - 1, s[0], s[0] * s[1] - 1, nun / 2, nun - s[0], nun - 2, nun - 1};
            for (long long u : at) {
                if (u < 0 || u >= nun) continue;
                const long long x = u % s[0], y = u / s[0] % s[1], z = u / (s[0] * s[1]);
                for (int oi = 0; oi < (dim == 3 ? 27 : 9); ++oi) {
                    const long long a = x + oi % 3 - 1, b = y + oi / 3 % 3 - 1, c = z + (dim == 3 ? oi / 9 - 1 : 0);
                    const long long v = msdd::stencil_neighbour((unsigned)u, msdd::stencil_offset(oi, dim, sy, sz), n);
                    const bool inside = a >= 0 && a < s[0] && b >= 0 && b < s[1] && c >= 0 && c < s[2];
                    if (v < 0 || v >= nun || (inside && v != a + s[0] * (b + s[1] * c))) ++bad;
                }
            }
        }
    msdd::UnknownIndex u = 2147483646;
    u += 152u * 8 * msdd::PCG_NT;
    if (u < (msdd::UnknownIndex)2147483647) ++bad;
    std::printf("%d\n", bad);
    return bad != 0;
}
