// Host emulation (no GPU needed) of the passes whose radix-32 stages run on pairs of lanes 16 apart, thread by thread with the
// kernels' own task numbers and the library's transforms, tables and exchange-buffer code:
//  - the table twiddles of 512 and 1024 points: a root rounded once is within sqrt(2) 2^-25 = 4.22e-8 of the exact one,
//    a product of two within three times that (1.27e-7);
//  - the force z chain of 512 points (16 x 32 forward, 32 x 16 inverse): forward against an FP64 DFT, then L times the input;
//  - the inverse y transform of 512 (16 x 32) and 1024 points (32 x 32) against an FP64 DFT.
// Limits of the transforms: 2^-24 of the rms per radix-2 level. Exit status 0 when every check passes.
#include <cmath>
#include <cstdio>
#include <vector>

#include "fft_pair.cuh"

using namespace colapm;

static unsigned g_s = 99u;
static float rnd() {
    g_s = g_s * 1664525u + 1013904223u;
    return (float)((g_s >> 8) * (1.0 / 16777216.0) - 0.5);
}
template <int L>
static Tw8<32> tables() {
    Tw8<32> t;
    auto w = [](long long i) {
        const double a = 2.0 * M_PI * (double)(i % L) / L;
        return make_float2((float)std::cos(a), (float)-std::sin(a));
    };
    for (int j = 0; j < 32; ++j) {
        for (int k = 0; k < 8; ++k) t.w[k][j] = w(k * j);
        for (int m = 0; m < 4; ++m) t.w8[m][j] = w(8 * m * j);
    }
    return t;
}

template <int L>
static int check_twiddles(const Tw8<32>& t) {
    double once = 0.0, product = 0.0;
    for (int j = 0; j < L / 32; ++j)
        for (int h = 0; h < 2; ++h) {
            float2 v[16];
            for (auto& e : v) e = make_float2(1.0f, 0.0f);
            pair_twiddle<-1>(v, &t, j, h);
            for (int m = 0; m < 16; ++m) {
                const int r = 2 * m + h;
                const double a = 2.0 * M_PI * j * r / L, e = std::hypot(v[m].x - std::cos(a), v[m].y + std::sin(a));
                double& worst = r < 8 || r % 8 == 0 ? once : product;
                worst = std::fmax(worst, e);
            }
        }
    std::printf("L=%d: twiddles %.2e, products of two %.2e off\n", L, once, product);
    return once <= 4.22e-8 && product <= 1.27e-7 ? 0 : 1;
}

// thread t of a 4-column tile: column, task alone, half and task of a pair
struct Who {
    int c, js, h, jp;
    explicit Who(int t) : c(t & 3), js(t >> 2), h((t >> 4) & 1), jp(((t >> 2) & 3) + 4 * (t >> 5)) {}
};
struct Regs {
    float2 v[16];
};
// the exchange with the partner, lane ^ 16, for every thread
template <int S>
static void dit(std::vector<Regs>& r) {
    const std::vector<Regs> in = [&] {
        for (auto& e : r) dft<16, S, true>(e.v);
        return r;
    }();
    for (int t = 0; t < (int)r.size(); ++t)
        for (int i = 0; i < 8; ++i)
            pair_dit_finish<S>(r[t].v, Who(t).h, i, pair_dit_send(in[t ^ 16].v, Who(t ^ 16).h, i));
}
template <int S>
static void dif(std::vector<Regs>& r) {
    std::vector<float2> sent(8 * r.size());
    for (int t = 0; t < (int)r.size(); ++t)
        for (int i = 0; i < 8; ++i) sent[8 * t + i] = pair_dif_send<S>(r[t].v, Who(t).h, i);
    for (int t = 0; t < (int)r.size(); ++t) {
        for (int i = 0; i < 8; ++i) pair_dif_finish(r[t].v, Who(t).h, i, sent[8 * (t ^ 16) + i]);
        pair_dif_dft<S>(r[t].v);
    }
}

static double error(const std::vector<float2>& in, const std::vector<float2>& out, int L, int sign) {   // [z][4]
    double err = 0.0, ref = 0.0;
    for (int c = 0; c < 4; ++c)
        for (int k = 0; k < L; ++k) {
            double re = 0.0, im = 0.0;
            for (int m = 0; m < L; ++m) {
                const double a = sign * 2.0 * M_PI * (double)((long long)m * k % L) / L;
                const float2 v = in[4 * m + c];
                re += v.x * std::cos(a) - v.y * std::sin(a);
                im += v.x * std::sin(a) + v.y * std::cos(a);
            }
            err += std::pow(out[4 * k + c].x - re, 2) + std::pow(out[4 * k + c].y - im, 2);
            ref += re * re + im * im;
        }
    return std::sqrt(err / ref);
}

// R1 alone (or on pairs) and R2 = 32 on pairs; X[k] in out, the registers of stage B in r
template <int L, int S>
static void transform(const std::vector<float2>& in, std::vector<float2>& out, std::vector<Regs>& r, const Tw8<32>& t) {
    constexpr int R1 = F2<L>::R1;
    using X = Xch<L, R1, 4>;
    const int T = (int)r.size();
    std::vector<float2> xb(X::SIZE);
    if constexpr (R1 == 32) {
        for (int i = 0; i < T; ++i)
            for (int m = 0; m < 16; ++m) r[i].v[m] = in[4 * (Who(i).jp + (L / R1) * (2 * m + Who(i).h)) + Who(i).c];
        dit<S>(r);
        for (int i = 0; i < T; ++i)
            for (int q = 0; q < 16; ++q) xb[X::at(Who(i).c, Who(i).jp * R1 + pair_dit_r(q, Who(i).h))] = r[i].v[q];
    } else {
        for (int i = 0; i < T; ++i) {
            float2 v[R1];
            for (int q = 0; q < R1; ++q) v[q] = in[4 * (Who(i).js + q * (L / R1)) + Who(i).c];
            dft<R1, S, true>(v);
            for (int q = 0; q < R1; ++q) xb[X::at(Who(i).c, Who(i).js * R1 + q)] = v[q];
        }
    }
    for (int i = 0; i < T; ++i) {
        for (int m = 0; m < 16; ++m) r[i].v[m] = xb[X::at(Who(i).c, Who(i).jp + R1 * (2 * m + Who(i).h))];
        pair_twiddle<S>(r[i].v, &t, Who(i).jp, Who(i).h);
    }
    dit<S>(r);
    for (int i = 0; i < T; ++i)
        for (int q = 0; q < 16; ++q) out[4 * (Who(i).jp + R1 * pair_dit_r(q, Who(i).h)) + Who(i).c] = r[i].v[q];
}

template <int L>
static int check() {
    const Tw8<32> t = tables<L>();
    const double limit = std::log2((double)L) * std::ldexp(1.0, -24);
    std::vector<float2> in(4 * L), out(4 * L);
    for (auto& e : in) e = make_float2(rnd(), rnd());
    std::vector<Regs> r(L / 4);
    int bad = check_twiddles<L>(t);
    transform<L, +1>(in, out, r, t);
    double e = error(in, out, L, +1);
    std::printf("L=%d inverse: rms rel error %.2e\n", L, e);
    bad |= !(e < limit);
    if constexpr (L == 512) {
        transform<L, -1>(in, out, r, t);
        e = error(in, out, L, -1);
        std::printf("L=%d forward: rms rel error %.2e\n", L, e);
        bad |= !(e < limit);
        using X = Xch<L, 32, 4>;
        std::vector<float2> xb(X::SIZE);
        dif<+1>(r);
        for (int i = 0; i < (int)r.size(); ++i)
            for (int m = 0; m < 16; ++m) xb[X::at(Who(i).c, Who(i).jp * 32 + 2 * m + Who(i).h)] = r[i].v[m];
        double err = 0.0, ref = 0.0;
        for (int i = 0; i < (int)r.size(); ++i) {
            float2 v[16];
            stage_b<L, 32, 16, +1, 4, true>(xb.data(), &t, Who(i).c, Who(i).js, v);
            for (int q = 0; q < 16; ++q) {
                const float2 a = in[4 * (Who(i).js + 32 * q) + Who(i).c];
                err += std::pow(v[q].x / L - a.x, 2) + std::pow(v[q].y / L - a.y, 2);
                ref += (double)a.x * a.x + (double)a.y * a.y;
            }
        }
        e = std::sqrt(err / ref);
        std::printf("L=%d forward then inverse: rms rel error %.2e\n", L, e);
        bad |= !(e < 2 * limit);
    }
    return bad;
}

int main() { return check<512>() | check<1024>(); }
