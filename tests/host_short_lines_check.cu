// Host check of the two-stage plans of 32, 48 and 80 points (no GPU needed), with the library's own DFT, twiddle table and
// exchange-buffer code:
//  - the twiddles, read off by twiddling ones: a root rounded once is within sqrt(2) 2^-25 = 4.22e-8 of the exact one
//    (each component at most 2^-25 off), a product of two within three times that (1.27e-7), whatever the power;
//  - forward and inverse transforms of 8 lines against an FP64 DFT: at most 2^-24 of the rms per radix-2 level;
//  - forward (radices R1, R2), then the outputs of task j unchanged into the inverse with swapped radices: L times the input.
// Exit status 0 when every check passes.
#include <cmath>
#include <cstdio>
#include <vector>

#include "fft2.cuh"

using colapm::Xch;

template <int L>
static float2 root(long long i) {
    const double a = 2.0 * M_PI * (double)(i % L) / L;
    return make_float2((float)std::cos(a), (float)-std::sin(a));
}
template <int L, int JN>
static void fill(colapm::Tw8<JN>& t) {   // as the library's load_tw2 does
    for (int j = 0; j < JN; ++j) {
        for (int k = 0; k < 8; ++k) t.w[k][j] = root<L>(k * j);
        for (int m = 0; m < 4; ++m) t.w8[m][j] = root<L>(8 * m * j);
    }
}
template <int L>
static void fill(colapm::Tw2& t) {
    for (int j = 0; j < 32; ++j) {
        t.w1[j] = root<L>(j);
        for (int m = 0; m < 4; ++m) t.w8[m][j] = root<L>(8 * m * j);
    }
}

// R twiddles of the tasks j < J
template <int L, int R, int J, int S, class TW>
static int check_twiddles(const TW& t) {
    double once = 0.0, product = 0.0;
    for (int j = 0; j < J; ++j) {
        float2 v[R];
        for (auto& e : v) e = make_float2(1.0f, 0.0f);
        colapm::twiddle2<R, S>(v, &t, j);
        for (int r = 0; r < R; ++r) {
            const double a = S * 2.0 * M_PI * j * r / L, e = std::hypot(v[r].x - std::cos(a), v[r].y - std::sin(a));
            double& worst = r <= 8 ? once : product;
            worst = std::fmax(worst, e);
        }
    }
    std::printf("L=%d radix %d sign=%+d: twiddles %.2e, products of two %.2e off\n", L, R, S, once, product);
    return once <= 4.22e-8 && product <= 1.27e-7 ? 0 : 1;
}

template <int L, int RA, int RB, int S, class TW>
static void stage_b(const std::vector<float2>& xb, std::vector<float2>& out, const TW& t) {
    for (int c = 0; c < 8; ++c)
        for (int j = 0; j < RA; ++j) {
            float2 v[RB];
            colapm::stage_b<L, RA, RB, S>(xb.data(), &t, c, j, v);
            for (int r = 0; r < RB; ++r) out[c * L + j + RA * r] = v[r];
        }
}
template <int L, int RA, int S>
static void stage_a(const std::vector<float2>& in, std::vector<float2>& xb) {   // task j: inputs j + r L / RA
    for (int c = 0; c < 8; ++c)
        for (int j = 0; j < L / RA; ++j) {
            float2 v[RA];
            for (int r = 0; r < RA; ++r) v[r] = in[c * L + j + r * (L / RA)];
            colapm::dft<RA, S>(v);
            for (int r = 0; r < RA; ++r) xb[Xch<L, RA>::at(c, j * RA + r)] = v[r];
        }
}

template <int L>
static int check() {
    constexpr int R1 = colapm::F2<L>::R1, R2 = colapm::F2<L>::R2;
    colapm::TwOf<L> t;
    fill<L>(t);
    int bad = check_twiddles<L, R2, R1, -1>(t) | check_twiddles<L, R2, R1, +1>(t) | check_twiddles<L, R1, R2, +1>(t);
    std::vector<float2> x(8 * L), X(8 * L), y(8 * L), xb(Xch<L, R1>::SIZE), xi(Xch<L, R2>::SIZE);
    unsigned s = 4321u + L;
    auto rnd = [&s] { s = s * 1664525u + 1013904223u; return (float)((s >> 8) * (1.0 / 16777216.0) - 0.5); };
    for (auto& e : x) e = make_float2(rnd(), rnd());
    const double limit = std::log2((double)L) * std::ldexp(1.0, -24);
    for (int dir = +1; dir >= -1; dir -= 2) {   // forward last: X feeds the chain below
        if (dir < 0) {
            stage_a<L, R1, -1>(x, xb);
            stage_b<L, R1, R2, -1>(xb, X, t);
        } else {
            stage_a<L, R1, +1>(x, xb);
            stage_b<L, R1, R2, +1>(xb, X, t);
        }
        double err = 0.0, ref = 0.0;
        for (int c = 0; c < 8; ++c)
            for (int k = 0; k < L; ++k) {
                double re = 0.0, im = 0.0;
                for (int m = 0; m < L; ++m) {
                    const double a = dir * 2.0 * M_PI * (double)(m * k % L) / L;
                    const float2 v = x[c * L + m];
                    re += v.x * std::cos(a) - v.y * std::sin(a);
                    im += v.x * std::sin(a) + v.y * std::cos(a);
                }
                err += std::pow(X[c * L + k].x - re, 2) + std::pow(X[c * L + k].y - im, 2);
                ref += re * re + im * im;
            }
        std::printf("L=%d sign=%+d: rms rel error %.2e\n", L, dir, std::sqrt(err / ref));
        bad |= !(std::sqrt(err / ref) < limit);
    }
    stage_a<L, R2, +1>(X, xi);
    stage_b<L, R2, R1, +1>(xi, y, t);
    double err = 0.0, ref = 0.0;
    for (int i = 0; i < 8 * L; ++i) {
        err += std::pow(y[i].x / L - x[i].x, 2) + std::pow(y[i].y / L - x[i].y, 2);
        ref += std::pow(x[i].x, 2) + std::pow(x[i].y, 2);
    }
    std::printf("L=%d forward then swapped-radix inverse: rms rel error %.2e\n", L, std::sqrt(err / ref));
    return bad | !(std::sqrt(err / ref) < 2 * limit);
}

int main() { return check<32>() | check<48>() | check<80>(); }
