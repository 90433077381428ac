// Host check of index and counting rules of the CUDA kernels (csrc/hostdev.h)
// that results on a GPU show only indirectly. Compiled with g++ by
// tests/test_hostdev_layout.py; prints "name value" lines.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "hostdev.h"

using namespace hr;

// One to three rounds of arrivals at one counter, mixed (the units are alike,
// so their order does not matter), then a round by itself: it must have one
// last unit, the last to come, and leave the counter at zero.
static int arrival_violations() {
    int bad = 0;
    for (int units = 2; units <= 6; ++units) {
        unsigned counter = 0;
        auto inc = [&](unsigned most) {
            const unsigned old = counter;
            counter = old >= most ? 0 : old + 1;
            return old;
        };
        for (int mixed = units; mixed <= 3 * units; mixed += units) {      // one to three rounds before
            counter = 0;
            int lasts = 0;
            for (int i = 0; i < mixed; ++i) lasts += last_arrival(units, inc);
            if (lasts != mixed / units) ++bad;
            for (int i = 0; i < units; ++i)
                if (last_arrival(units, inc) != (i == units - 1)) ++bad;
            if (counter != 0) ++bad;
        }
    }
    return bad;
}

// The lengths the kernels take: 2^a <= 4096, 3 2^a <= 6144, 5 2^a <= 5120, 9 2^a <= 2304.
static std::vector<int> lengths() {
    std::vector<int> out;
    int R[kMaxDifPasses], S[kMaxDifPasses];
    for (int n = 2; n <= 6144; ++n)
        if ((n % 3 == 0 ? n <= 6144 : n % 5 == 0 ? n <= 5120 : n <= 4096) && dif_plan(n, R, S) > 0) out.push_back(n);
    return out;
}

// The shared-memory layout of length n: elements below seq_pitch and apart,
// sequences back to back, every pass's address steps, and the positions of
// the frequencies.
static int layout_violations(int n) {
    int R[kMaxDifPasses], S[kMaxDifPasses], lst[kMaxDifPasses] = {}, bad = 0;
    const int s = dif_plan(n, R, S);
    for (int p = 0; p < s; ++p) {
        while ((1 << lst[p]) < S[p]) ++lst[p];
        bad += (1 << lst[p]) != S[p];
    }
    const int pitch = seq_pitch(n, R[0]), ls0 = lst[0];
    const bool by16 = fft_by16(n);
    auto at = [&](int i) { return by16 ? padn(i, ls0) : pad16(i); };
    std::vector<int> seen(pitch, 0);
    for (int i = 0; i < n; ++i) {
        const int a = at(i);
        if (a < 0 || a >= pitch || seen[a]++) ++bad;
    }
    if (!by16) return bad;
    bad += s < 2 || s > 4 || S[s - 1] != 1 || R[s - 1] != 16 || S[0] % 16 != 0 || (s == 4 && R[1] != 4);
    for (int q = 1; q < 6; ++q)
        for (int i = 0; i < n; ++i) bad += padn(q * n + i, ls0) != q * pitch + padn(i, ls0);
    for (int m = 0; m < S[0]; ++m)
        for (int r = 0; r < R[0]; ++r) bad += padn(m + r * S[0], ls0) != pad16(m) + r * first_step(ls0);
    for (int p = 1; p < s; ++p)
        for (int b = 0; b < n / R[p]; ++b) {
            const int base = dif_base(R[p], S[p], b), step = S[p] == 1 ? 1 : S[p] + S[p] / 16;
            bad += S[p] > 1 && S[p] % 16 != 0;
            for (int r = 0; r < R[p]; ++r) bad += padn(base + r * S[p], ls0) != padn(base, ls0) + r * step;
        }
    const FreqDigits pos(s, R[0], lst);
    for (int k = 0; k < n; ++k) bad += pos(k) != padn(dif_pos(s, R, S, k), ls0);
    return bad;
}

// A small DFT whose inputs from NZ on are zero and not read, against its
// definition; the inputs not to be read hold NaN.
template <int R, int NZ>
static double zeros_error(std::mt19937& rng) {
    std::normal_distribution<double> N(0, 1);
    double worst = 0;
    for (int dir : {-1, 1}) {
        cf v[R], x[R];
        for (int r = 0; r < R; ++r) {
            x[r] = r < NZ ? cf{(float)N(rng), (float)N(rng)} : cf{0.f, 0.f};
            v[r] = r < NZ ? x[r] : cf{NAN, NAN};
        }
        dft_zeros<R, NZ>(v, dir);
        double num = 0, den = 0;
        for (int k = 0; k < R; ++k) {
            double re = 0, im = 0;
            for (int r = 0; r < R; ++r) {
                const double c = std::cos(2 * M_PI * (r * k % R) / R), sn = dir * std::sin(2 * M_PI * (r * k % R) / R);
                re += x[r].x * c - x[r].y * sn;
                im += x[r].x * sn + x[r].y * c;
            }
            num += (v[k].x - re) * (v[k].x - re) + (v[k].y - im) * (v[k].y - im);
            den += re * re + im * im;
        }
        const double e = std::sqrt(num / den);
        if (!(e <= worst)) worst = e;            // NaN too
    }
    return worst;
}
template <int R>
static double zeros_errors(std::mt19937& rng) {
    const double a = zeros_error<R, R>(rng), b = zeros_error<R, (R + 1) / 2>(rng);
    return a > b || a != a ? a : b;
}

int main() {
    int bad = 0;
    for (int n : lengths()) bad += layout_violations(n);
    std::printf("fft_lengths %d\n", (int)lengths().size());
    std::printf("layout_violations %d\n", bad);
    std::mt19937 rng(1604);
    double e = 0;
    for (double x : {zeros_errors<2>(rng), zeros_errors<3>(rng), zeros_errors<4>(rng), zeros_errors<5>(rng),
                     zeros_errors<6>(rng), zeros_errors<8>(rng), zeros_errors<9>(rng), zeros_errors<10>(rng),
                     zeros_errors<12>(rng), zeros_errors<16>(rng)})
        if (!(x <= e)) e = x;
    std::printf("dft_zeros_rel_l2 %.3e\n", e);
    std::printf("arrival_violations %d\n", arrival_violations());
    return 0;
}
