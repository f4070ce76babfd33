// Host check of the index arithmetic of the particle kernels: UDiv against the ordinary division, and the
// Lattice sites against their definition i nm / np, and the P(k) bin thresholds against a search through every |n|^2.
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
    for (int nm : {16, 64, 96, 256})
        for (int nbins : {1, 7, 100, 700})
            for (double box : {100.0, 256.0, 512.7})
                for (int k = 0; k < 4; ++k) {   // default range, edges on modes, a narrow range, edges beyond the mesh
                    const double kf = 2.0 * M_PI / box, ny = M_PI * nm / box;
                    const double kmin = k == 1 ? 2.0 * kf : (k == 2 ? 0.31 * ny : (k == 3 ? 0.01 * kf : kf));
                    const double kmax = k == 1 ? 6.0 * kf : (k == 2 ? 0.33 * ny : (k == 3 ? 100.0 * ny : ny));
                    const int n2max = 3 * (nm / 2) * (nm / 2);
                    static int lo[701];
                    colapm::power_thresholds(nbins, kmin, kmax, kf, n2max, lo);
                    for (int b = 0, n2 = 0; b <= nbins; ++b) {
                        const double edge = kmin * std::pow(kmax / kmin, (double)b / nbins);
                        while (n2 <= n2max && !(kf * std::sqrt((double)n2) >= edge)) ++n2;   // edges grow
                        bad += lo[b] != n2;
                    }
                }
    printf("%ld mismatches\n", bad);
    return bad != 0;
}
