// Host check of the index arithmetic of the particle kernels: UDiv against the ordinary division, and the
// Lattice sites against their definition i nm / np.
#include <cstdio>

#include "../paper_1506_03737_gb300/csrc/colapm_internal.h"

int main() {
    long bad = 0;
    for (unsigned d = 2; d <= 1024; ++d) {
        const colapm::UDiv u = colapm::make_udiv((int)d);
        auto check = [&](unsigned n) {
            int x, y, z;
            u.split(n, x, y, z);
            bad += u.div(n) != n / d || x != (int)(n % d) || y != (int)((n / d) % d) || z != (int)((n / d / d) % d);
        };
        const unsigned limit = 1u << 30;
        for (unsigned q = 0; q < limit / d; q += 1 + q / 512)   // both sides of multiples of d over the range
            for (int e = -1; e <= 1; ++e)
                if (q || e >= 0) check(q * d + (unsigned)e);
        for (int c : {0, 1, -1, (int)d - 1, (int)d, -(int)d, -(int)d - 1, 5 * (int)d + 3, -5 * (int)d + 3, 1 << 30, -(1 << 30),
                      2147483647, -2147483647 - 1}) {
            const int want = (int)(((long long)c % (int)d + d) % d);
            bad += u.wrap(c) != want;
        }
        for (unsigned e = 0; e < 3000; ++e) {   // the top of the range, and words beyond it
            check(limit - 1 - e);
            check(limit + e);
            check(0xffffffffu - e);
        }
    }
    const int sizes[] = {16, 32, 64, 96, 128, 160, 192, 256, 320, 384, 512, 1024};
    for (int np : sizes)
        for (int nm : sizes) {
            if (nm % np != 0 && np != 2 * nm && np != 4 * nm) continue;
            const colapm::Lattice l = colapm::make_lattice(np, nm);
            for (int i = 0; i < np; ++i) {
                int base;
                float frac;
                l.at(i, base, frac);
                const int t = i * nm;
                bad += base != t / np || frac != (float)(t % np) / (float)np;
            }
        }
    printf("%ld mismatches\n", bad);
    return bad != 0;
}
