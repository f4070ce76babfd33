// Host check of the index maps of every mesh that uses the blocked layout and is not in host_layout_check.cu (no GPU needed):
// hs_index<L, true> maps (kx < L/2, y < L, z < L) one-to-one onto [0, L/2 L L); and, in both layouts and at every length with
// a y pass, hs_row(j, r) is the distance of row j + r STEP from row 0 for the strides of both stages (mixed lengths
// have strides that are no multiples of 8). Exit status 0 when every check passes.
#include <cstdio>
#include <vector>

#include "fft2.cuh"

using namespace colapm;

template <int L>
static int one_to_one() {
    const size_t n = (size_t)(L / 2) * L * L;
    std::vector<unsigned char> seen(n, 0);
    for (int z = 0; z < L; ++z)
        for (int y = 0; y < L; ++y)
            for (int kx = 0; kx < L / 2; ++kx) {
                const size_t i = hs_index<L, true>(kx, y, z);
                if (i >= n || seen[i]++) {
                    std::printf("L=%d: index %zu of (%d,%d,%d) out of range or repeated\n", L, i, kx, y, z);
                    return 1;
                }
            }
    std::printf("L=%d: one-to-one\n", L);
    return 0;
}

template <int L, bool BLK, int STEP, int COUNT>
static int rows() {
    int bad = 0;
    for (int j = 0; j < STEP; ++j)
        for (int r = 0; r < COUNT; ++r)
            for (int kx : {0, 5, 8, L / 2 - 1})
                for (int z : {0, 3, L - 1})
                    bad += hs_row<L, BLK, STEP>(j, r) != hs_index<L, BLK>(kx, j + r * STEP, z) - hs_index<L, BLK>(kx, 0, z);
    if (bad) std::printf("L=%d BLK=%d step %d: %d wrong rows\n", L, (int)BLK, STEP, bad);
    return bad != 0;
}
template <int L>
static int both() {
    constexpr int RA = F2<L>::R1, RB = F2<L>::R2;
    static_assert(RA * RB == L, "");
    int bad = rows<L, false, L / RA, RA>() | rows<L, false, RA, RB>();
    if constexpr (L >= 64) bad |= rows<L, true, L / RA, RA>() | rows<L, true, RA, RB>();
    if (!bad) std::printf("L=%d: rows consistent\n", L);
    return bad;
}

int main() {
    int bad = one_to_one<64>() | one_to_one<96>() | one_to_one<128>() | one_to_one<160>() | one_to_one<192>() | one_to_one<256>() |
              one_to_one<320>() | one_to_one<384>();
    bad |= both<32>() | both<64>() | both<96>() | both<128>() | both<160>() | both<192>() | both<256>() | both<320>() | both<384>() |
           both<512>() | both<1024>();
    return bad;
}
