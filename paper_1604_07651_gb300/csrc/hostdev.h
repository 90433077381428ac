// Pure arithmetic shared by the device kernels and by the host unit tests of
// those kernels (compiled with g++ for the tests, nvcc for the library):
// * cubic B-spline tap weights (the B3 of Eq. (14)-(17));
// * the in-register DFTs and the in-place FFT passes, with their position
//   maps (the FFTs of Eq. (7), (16)-(17));
// * the packing of a real FFT into a complex FFT of half the length.
#pragma once

#include <math.h>
#include <stdint.h>

#if defined(__CUDACC__)
#define HD __host__ __device__ __forceinline__
#define HD_UNROLL _Pragma("unroll")
#else
#define HD inline
#define HD_UNROLL
#endif

namespace hr {

struct cf { float x, y; };             // complex float

// Cubic B-spline weights of the four taps i0 .. i0+3, i0 = floor(x) - 1,
// at fractional part f = x - floor(x): B3(f+1), B3(f), B3(f-1), B3(f-2).
HD void b3_weights(float f, float w[4]) {
    float g = 1.0f - f;
    float f2 = f * f, f3 = f2 * f;
    w[0] = g * g * g * (1.0f / 6.0f);
    w[1] = (4.0f - 6.0f * f2 + 3.0f * f3) * (1.0f / 6.0f);
    w[2] = (1.0f + 3.0f * f + 3.0f * f2 - 3.0f * f3) * (1.0f / 6.0f);
    w[3] = f3 * (1.0f / 6.0f);
}

// Quintic B-spline weights of the six taps i0 .. i0+5, i0 = floor(x) - 2, at
// fractional part t: B5(t+2), B5(t+1), B5(t), B5(t-1), B5(t-2), B5(t-3), the
// pieces of (3-|x|)^5 - 6 (2-|x|)^5 + 15 (1-|x|)^5 over 120 (terms with a
// positive base only), expanded in t; weights d and 5-d are mirror images
// (t -> 1 - t).
HD void b5_weights(float t, float w[6]) {
    const float s = 1.0f - t;
    const float t2 = t * t, s2 = s * s;
    const float k = 1.0f / 120.0f;
    w[0] = s2 * s2 * s * k;
    w[5] = t2 * t2 * t * k;
    // 5 t^5 - 20 t^4 + 20 t^3 + 20 t^2 - 50 t + 26 and its mirror
    w[1] = ((((5.0f * t - 20.0f) * t + 20.0f) * t + 20.0f) * t - 50.0f) * t * k + 26.0f * k;
    w[4] = ((((5.0f * s - 20.0f) * s + 20.0f) * s + 20.0f) * s - 50.0f) * s * k + 26.0f * k;
    // -10 t^5 + 30 t^4 - 60 t^2 + 66 and its mirror
    w[2] = (((-10.0f * t + 30.0f) * t2 - 60.0f) * t2 + 66.0f) * k;
    w[3] = (((-10.0f * s + 30.0f) * s2 - 60.0f) * s2 + 66.0f) * k;
}

// B-spline weights of NT = order + 1 taps: cubic (4) or quintic (6).
template <int NT>
HD void bspline_weights(float f, float w[NT]);
template <>
HD void bspline_weights<4>(float f, float w[4]) { b3_weights(f, w); }
template <>
HD void bspline_weights<6>(float f, float w[6]) { b5_weights(f, w); }

// Arrival of one of a tile's `units` at its counter; true for the last. `inc`
// counts like CUDA's atomicInc: returns the old value and stores it plus one,
// or zero where it has reached the argument. So the counter holds zero again
// after every full round without a store of its own, also when the rounds of
// calls that wrongly overlap on one plan mix (their results are lost, the
// plan is not: a store of zero by the last unit could fall between the other
// call's arrivals and leave a count behind for good).
template <class Inc>
HD bool last_arrival(int units, Inc&& inc) { return inc((unsigned)units - 1) == (unsigned)units - 1; }

// A layout of 8-byte elements that no kernel uses any more (tests/hostdev_check.cpp
// still checks it): the low four bits XOR-ed with the next four, a permutation
// within each block of 16 (and the identity below 16).
HD int sw(int i) { return i ^ ((i >> 4) & 15); }

HD cf cmul(cf a, cf b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
HD cf cmulc(cf a, cf b) { return {a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y}; }  // a * conj(b)
HD cf cadd(cf a, cf b) { return {a.x + b.x, a.y + b.y}; }
HD cf csub(cf a, cf b) { return {a.x - b.x, a.y - b.y}; }
// The operations of the in-register DFTs, on one complex number (cf) here and
// on the same element of two sequences at once in the kernels (fft2.cuh):
// a + i b, a - i b, the product with a constant, a + s b and s a for real s.
HD cf caddi(cf a, cf b) { return {a.x - b.y, a.y + b.x}; }
HD cf csubi(cf a, cf b) { return {a.x + b.y, a.y - b.x}; }
HD cf cmulk(cf a, float re, float im) { return {a.x * re - a.y * im, a.x * im + a.y * re}; }
HD cf caxpy(cf a, float s, cf b) { return {a.x + s * b.x, a.y + s * b.y}; }
HD cf cscale(float s, cf a) { return {s * a.x, s * a.y}; }

// In-register DFT of size R (2, 3, 4, 5, 6, 8, 9, 10, 12, 16) with sign dir
// (-1 forward, +1 inverse; a compile-time constant after inlining), for any
// element type with the operations above.
template <int R>
struct Dft;
template <int R, class C>
HD void dft_small(C* v, int dir) { Dft<R>::template run<R>(v, dir); }
// The same when the inputs from NZ on are zero (they are not read): the
// zero-padded half of an FFT's first pass.
template <int R, int NZ, class C>
HD void dft_zeros(C* v, int dir) { Dft<R>::template run<NZ>(v, dir); }
template <int R, int NZ, class C>
HD void dft_lead(C* v, int dir);
// Inputs below NZ among the every-F-th ones n2, n2 + F, ... of a size-R DFT.
HD constexpr int lead_count(int NZ, int F, int n2) { return NZ > n2 ? (NZ - n2 + F - 1) / F : 0; }

template <>
struct Dft<2> {
    template <int NZ, class C>
    HD static void run(C* v, int) {
        if (NZ == 1) {
            v[1] = v[0];
            return;
        }
        const C a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};

template <>
struct Dft<4> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        if (NZ < 3) return dft_lead<4, NZ>(v, dir);
        const C a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
        const C b0 = cadd(v[1], v[3]), b1 = csub(v[1], v[3]);
        v[0] = cadd(a0, b0);
        v[2] = csub(a0, b0);
        v[1] = dir < 0 ? csubi(a1, b1) : caddi(a1, b1);
        v[3] = dir < 0 ? caddi(a1, b1) : csubi(a1, b1);
    }
};

template <>
struct Dft<3> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        if (NZ < 3) return dft_lead<3, NZ>(v, dir);
        const float s = 0.86602540378443864676f * (float)dir;  // sin(2 pi/3) * dir
        const C t = cadd(v[1], v[2]);
        const C d = cscale(s, csub(v[1], v[2]));
        const C m = caxpy(v[0], -0.5f, t);
        v[0] = cadd(v[0], t);
        v[1] = caddi(m, d);
        v[2] = csubi(m, d);
    }
};

// DFTs of size 3, 4 and 5 whose inputs from NZ on are zero.
template <int R, int NZ, class C>
HD void dft_lead(C* v, int dir) {
    if (NZ >= R || (R == 4 && NZ == 3) || (R == 5 && NZ == 4)) {
        dft_small<R>(v, dir);
    } else if (NZ == 1) {
HD_UNROLL
        for (int k = 1; k < R; ++k) v[k] = v[0];
    } else if (R == 3) {                                   // two inputs
        const C m = caxpy(v[0], -0.5f, v[1]), d = cscale(0.86602540378443864676f * (float)dir, v[1]);
        v[0] = cadd(v[0], v[1]);
        v[1] = caddi(m, d);
        v[2] = csubi(m, d);
    } else if (R == 4) {
        const C a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[2] = csub(a, b);
        v[1] = dir < 0 ? csubi(a, b) : caddi(a, b);
        v[3] = dir < 0 ? caddi(a, b) : csubi(a, b);
    } else {                                               // R == 5, two or three inputs
        const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
        const float s1 = 0.95105651629515357212f * (float)dir, s2 = 0.58778525229247312917f * (float)dir;
        C a1 = caxpy(v[0], c1, v[1]), a2 = caxpy(v[0], c2, v[1]), b1 = cscale(s1, v[1]), b2 = cscale(s2, v[1]);
        C sum = cadd(v[0], v[1]);
        if (NZ == 3) {
            a1 = caxpy(a1, c2, v[2]);
            a2 = caxpy(a2, c1, v[2]);
            b1 = caxpy(b1, s2, v[2]);
            b2 = caxpy(b2, -s1, v[2]);
            sum = cadd(sum, v[2]);
        }
        v[0] = sum;
        v[1] = caddi(a1, b1);
        v[4] = csubi(a1, b1);
        v[2] = caddi(a2, b2);
        v[3] = csubi(a2, b2);
    }
}

// cos(2 pi i / 16); with i a compile-time constant after unrolling, the
// switch folds to a literal (no table in local memory).
HD float cos16(int i) {
    switch (i & 15) {
        case 0: return 1.0f;
        case 1: case 15: return 0.92387953251128674f;
        case 2: case 14: return 0.70710678118654752f;
        case 3: case 13: return 0.38268343236508977f;
        case 4: case 12: return 0.0f;
        case 5: case 11: return -0.38268343236508977f;
        case 6: case 10: return -0.70710678118654752f;
        case 7: case 9: return -0.92387953251128674f;
        default: return -1.0f;
    }
}
// cos(2 pi m / 12) and cos(2 pi m / 10), as above.
HD float cos12(int i) {
    switch (((i % 12) + 12) % 12) {
        case 0: return 1.0f;
        case 1: case 11: return 0.86602540378443864676f;   // sqrt(3)/2
        case 2: case 10: return 0.5f;
        case 3: case 9: return 0.0f;
        case 4: case 8: return -0.5f;
        case 5: case 7: return -0.86602540378443864676f;
        default: return -1.0f;
    }
}
HD float cos10(int i) {
    switch (((i % 10) + 10) % 10) {
        case 0: return 1.0f;
        case 1: case 9: return 0.80901699437494742410f;    // (sqrt5 + 1)/4
        case 2: case 8: return 0.30901699437494742410f;    // (sqrt5 - 1)/4
        case 3: case 7: return -0.30901699437494742410f;
        case 4: case 6: return -0.80901699437494742410f;
        default: return -1.0f;
    }
}
HD float sin10(int i) {
    switch (((i % 10) + 10) % 10) {
        case 1: case 4: return 0.58778525229247312917f;    // sin 36 deg = sin 144 deg
        case 2: case 3: return 0.95105651629515357212f;    // sin 72 deg = sin 108 deg
        case 6: case 9: return -0.58778525229247312917f;
        case 7: case 8: return -0.95105651629515357212f;
        default: return 0.0f;
    }
}

// v times exp(dir * 2 pi i m / 16) or / 12; a quarter turn (m = N / 4) is a
// swap done by the caller's caddi / csubi where it can be, here by a product
// with (0, dir).
template <class C>
HD C turn16(C v, int m, int dir) { return m ? cmulk(v, cos16(m), dir * cos16(m - 4)) : v; }   // sin(x) = cos(x - pi/2)
template <class C>
HD C turn12(C v, int m, int dir) { return m ? cmulk(v, cos12(m), dir * cos12(m - 3)) : v; }

// Size 6 as 3 x 2 and size 12 as 3 x 4 (Cooley-Tukey with n = F n1 + n2,
// k = k1 + 3 k2): Y[n2][k1] = DFT3 over n1 of x[F n1 + n2], times
// W^(n2 k1), then X[k1 + 3 k2] = DFT-F over n2.
template <int F, int NZ, class C>
HD void dft_3xF(C* v, int dir) {
    C y[F][3];
HD_UNROLL
    for (int n2 = 0; n2 < F; ++n2) {
HD_UNROLL
        for (int n1 = 0; n1 < 3; ++n1)
            if (F * n1 + n2 < NZ) y[n2][n1] = v[F * n1 + n2];
    }
    dft_lead<3, lead_count(NZ, F, 0)>(y[0], dir);
    dft_lead<3, lead_count(NZ, F, 1)>(y[1], dir);
    if (F > 2) {
        dft_lead<3, lead_count(NZ, F, 2)>(y[F > 2 ? 2 : 0], dir);
        dft_lead<3, lead_count(NZ, F, 3)>(y[F > 2 ? 3 : 0], dir);
    }
HD_UNROLL
    for (int k1 = 0; k1 < 3; ++k1) {
        C z[F];
HD_UNROLL
        for (int n2 = 0; n2 < F; ++n2) z[n2] = turn12(y[n2][k1], n2 * k1 * (12 / (3 * F)), dir);
        dft_small<F>(z, dir);
HD_UNROLL
        for (int k2 = 0; k2 < F; ++k2) v[k1 + 3 * k2] = z[k2];
    }
}

template <>
struct Dft<6> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) { dft_3xF<2, NZ>(v, dir); }
};

template <>
struct Dft<12> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) { dft_3xF<4, NZ>(v, dir); }
};

// exp(dir * 2 pi i m / 9) for m = 1, 2, 4, the twiddles of the 3 x 3 split
// (cos and sin of 40, 80 and 160 degrees).
HD cf root9(int m, int dir) {
    switch (m) {
        case 1: return {0.76604444311897803520f, dir * 0.64278760968653932632f};
        case 2: return {0.17364817766693034885f, dir * 0.98480775301220805936f};
        default: return {-0.93969262078590838405f, dir * 0.34202014332566873304f};
    }
}

// Size 9 as 3 x 3 (Cooley-Tukey with n = 3 n1 + n2, k = k1 + 3 k2):
// Y[n2][k1] = DFT3 over n1 of x[3 n1 + n2], times W9^(n2 k1), then
// X[k1 + 3 k2] = DFT3 over n2.
template <>
struct Dft<9> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        C y[3][3];
HD_UNROLL
        for (int n2 = 0; n2 < 3; ++n2) {
HD_UNROLL
            for (int n1 = 0; n1 < 3; ++n1)
                if (3 * n1 + n2 < NZ) y[n2][n1] = v[3 * n1 + n2];
        }
        dft_lead<3, lead_count(NZ, 3, 0)>(y[0], dir);
        dft_lead<3, lead_count(NZ, 3, 1)>(y[1], dir);
        dft_lead<3, lead_count(NZ, 3, 2)>(y[2], dir);
HD_UNROLL
        for (int k1 = 0; k1 < 3; ++k1) {
            C z[3];
HD_UNROLL
            for (int n2 = 0; n2 < 3; ++n2)
                z[n2] = (n2 * k1 != 0) ? cmulk(y[n2][k1], root9(n2 * k1, dir).x, root9(n2 * k1, dir).y) : y[n2][k1];
            dft_small<3>(z, dir);
HD_UNROLL
            for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = z[k2];
        }
    }
};

// Size 5 directly: with t1 = x1 + x4, t2 = x2 + x3, t3 = x1 - x4,
// t4 = x2 - x3 and c_m = cos(2 pi m / 5), s_m = sin(2 pi m / 5):
// X1,4 = x0 + c1 t1 + c2 t2 +- i dir (s1 t3 + s2 t4),
// X2,3 = x0 + c2 t1 + c1 t2 +- i dir (s2 t3 - s1 t4).
template <>
struct Dft<5> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        if (NZ < 4) return dft_lead<5, NZ>(v, dir);
        const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;   // (sqrt5 - 1)/4, -(sqrt5 + 1)/4
        const float s1 = 0.95105651629515357212f * (float)dir, s2 = 0.58778525229247312917f * (float)dir;
        const C t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
        const C t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
        const C a1 = caxpy(caxpy(v[0], c1, t1), c2, t2);
        const C a2 = caxpy(caxpy(v[0], c2, t1), c1, t2);
        const C b1 = caxpy(cscale(s1, t3), s2, t4);
        const C b2 = caxpy(cscale(s2, t3), -s1, t4);
        v[0] = cadd(v[0], cadd(t1, t2));
        v[1] = caddi(a1, b1);
        v[4] = csubi(a1, b1);
        v[2] = caddi(a2, b2);
        v[3] = csubi(a2, b2);
    }
};

// Size 10 as 5 x 2: Y[n2][k1] = DFT5 over n1 of x[2 n1 + n2], times
// W10^(n2 k1), then X[k1 + 5 k2] = DFT2 over n2.
template <>
struct Dft<10> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        C y0[5], y1[5];
HD_UNROLL
        for (int n1 = 0; n1 < 5; ++n1) {
            if (2 * n1 < NZ) y0[n1] = v[2 * n1];
            if (2 * n1 + 1 < NZ) y1[n1] = v[2 * n1 + 1];
        }
        dft_lead<5, lead_count(NZ, 2, 0)>(y0, dir);
        dft_lead<5, lead_count(NZ, 2, 1)>(y1, dir);
HD_UNROLL
        for (int k1 = 0; k1 < 5; ++k1) {
            const C t = k1 ? cmulk(y1[k1], cos10(k1), dir * sin10(k1)) : y1[k1];
            v[k1] = cadd(y0[k1], t);
            v[k1 + 5] = csub(y0[k1], t);
        }
    }
};

// Size 8 as 2 x 4: inputs x[2 n1 + n2], X[k1 + 4 k2]; the quarter turn of
// k1 = 2 is folded into the last butterfly.
template <>
struct Dft<8> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        C e[4], o[4];
HD_UNROLL
        for (int n1 = 0; n1 < 4; ++n1) {
            if (2 * n1 < NZ) e[n1] = v[2 * n1];
            if (2 * n1 + 1 < NZ) o[n1] = v[2 * n1 + 1];
        }
        dft_lead<4, lead_count(NZ, 2, 0)>(e, dir);
        dft_lead<4, lead_count(NZ, 2, 1)>(o, dir);
HD_UNROLL
        for (int k = 0; k < 4; ++k) {
            if (k == 2) {
                v[k] = dir < 0 ? csubi(e[k], o[k]) : caddi(e[k], o[k]);
                v[k + 4] = dir < 0 ? caddi(e[k], o[k]) : csubi(e[k], o[k]);
            } else {
                const C t = turn16(o[k], 2 * k, dir);
                v[k] = cadd(e[k], t);
                v[k + 4] = csub(e[k], t);
            }
        }
    }
};

// Size 16 as 4 x 4: Y[n2][k1] = DFT4 over n1 of x[4 n1 + n2], times
// W16^(n2 k1), then X[k1 + 4 k2] = DFT4 over n2; the quarter turn of
// n2 k1 = 4 (n2 = k1 = 2) is folded into that DFT4's first butterfly.
template <>
struct Dft<16> {
    template <int NZ, class C>
    HD static void run(C* v, int dir) {
        C y[4][4];
HD_UNROLL
        for (int n2 = 0; n2 < 4; ++n2) {
HD_UNROLL
            for (int n1 = 0; n1 < 4; ++n1)
                if (4 * n1 + n2 < NZ) y[n2][n1] = v[4 * n1 + n2];
        }
        dft_lead<4, lead_count(NZ, 4, 0)>(y[0], dir);
        dft_lead<4, lead_count(NZ, 4, 1)>(y[1], dir);
        dft_lead<4, lead_count(NZ, 4, 2)>(y[2], dir);
        dft_lead<4, lead_count(NZ, 4, 3)>(y[3], dir);
HD_UNROLL
        for (int k1 = 0; k1 < 4; ++k1) {
            C z[4];
HD_UNROLL
            for (int n2 = 0; n2 < 4; ++n2)
                z[n2] = n2 * k1 == 4 ? y[n2][k1] : turn16(y[n2][k1], n2 * k1, dir);
            if (k1 == 2) {
                const bool plus = dir > 0;
                const C a0 = plus ? caddi(z[0], z[2]) : csubi(z[0], z[2]);
                const C a1 = plus ? csubi(z[0], z[2]) : caddi(z[0], z[2]);
                const C b0 = cadd(z[1], z[3]), b1 = csub(z[1], z[3]);
                z[0] = cadd(a0, b0);
                z[2] = csub(a0, b0);
                z[1] = plus ? caddi(a1, b1) : csubi(a1, b1);
                z[3] = plus ? csubi(a1, b1) : caddi(a1, b1);
            } else {
                dft_small<4>(z, dir);
            }
HD_UNROLL
            for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = z[k2];
        }
    }
};

// Twiddle table of one FFT pass with Ns butterflies per block and radix R:
// entry (r - 1) Ns + jm is exp(-2 pi i r jm / (Ns R)), r = 1 .. R-1,
// jm < Ns; computed in FP64 and rounded once. A pass with Ns = 1 has none.
HD int stage_table_len(int Ns, int R) { return Ns > 1 ? Ns * (R - 1) : 0; }

inline void stage_twiddles(int Ns, int R, cf* T) {
    if (Ns <= 1) return;
    for (int r = 1; r < R; ++r)
        for (int jm = 0; jm < Ns; ++jm) {
            const double a = -2.0 * 3.14159265358979323846 * (double)((r * jm) % (Ns * R)) / (double)(Ns * R);
            T[(r - 1) * Ns + jm] = {(float)cos(a), (float)sin(a)};
        }
}

// Radix plan of n = 2^a, 3 * 2^a, 5 * 2^a or 9 * 2^a (n <= 2304): radix 16
// while possible, then the rest r = n / 16^k in one stage when r is 2, 3, 4,
// 5, 6, 8, 9, 10 or 12, else radix 4 then 6 (r = 24), radix 4 then 5
// (r = 20), radix 8 then 5 (r = 40) or radix 2, 4, 8 then 9 (r = 18, 36,
// 72); the factor 3, 5 or 9 is always in the last stage, so every stage sees
// a power-of-two Ns. Returns the number of stages, or -1 for any other n.
HD int fft_radices(int n, int rad[32]) {
    int m = n;
    if (m % 9 == 0) {
        if (n > 2304) return -1;   // 9 * 2^a up to 2304 (a larger one would need radix 18)
        m /= 9;
    } else if (m % 3 == 0) m /= 3;
    else if (m % 5 == 0) m /= 5;
    if (m < 1 || (m & (m - 1)) != 0) return -1;
    int k = 0;
    while (n % 16 == 0) {
        rad[k++] = 16;
        n /= 16;
    }
    if (n == 24) {
        rad[k++] = 4;
        rad[k++] = 6;
    } else if (n == 20) {
        rad[k++] = 4;
        rad[k++] = 5;
    } else if (n == 40) {
        rad[k++] = 8;
        rad[k++] = 5;
    } else if (n == 18 || n == 36 || n == 72) {
        rad[k++] = n / 9;
        rad[k++] = 9;
    } else if (n != 1) {
        rad[k++] = n;   // 2, 3, 4, 5, 6, 8, 9, 10 or 12
    }
    return k;
}

// ---------------------------------------------------------------------------
// In-place mixed-radix FFT by decimation in frequency (forward) and in time
// (inverse). The forward transform leaves its output in digit-reversed order
// and the inverse takes digit-reversed input back to natural order, so a
// pointwise product between them needs no reordering, and every pass reads
// and writes the same positions (one barrier between passes in shared
// memory).
//
// Passes p = 0 .. s-1 take the radices of fft_radices in order, with strides
// S_p = n / (R_0 ... R_p) and blocks of L_p = R_p S_p consecutive elements.
// Forward pass p, butterfly b in [0, n / R_p): block q = b div S_p,
// m = b mod S_p; inputs x_r at q L_p + m + r S_p (r < R_p); outputs
//     y_k = W_{L_p}^(m k) sum_r x_r W_{R_p}^(r k),   W_N = exp(-2 pi i / N),
// at the same positions (k in place of r). After the last pass position
// sum_p k_p S_p holds frequency sum_p k_p R_0 ... R_(p-1). Inverse pass p
// (p = s-1 down to 0) undoes forward pass p up to the factor R_p:
//     x_r = sum_k conj(W_{L_p}^(m k)) y_k W_{R_p}^(-r k).
// The twiddles W_{L_p}^(m k) of pass p are stage_twiddles(S_p, R_p); the last
// pass has S = 1 and none.
// ---------------------------------------------------------------------------
constexpr int kMaxDifPasses = 8;

// Radices and strides of the passes of length n: the radices of fft_radices
// in reverse order (the factor 3, 5 or 9 first, radix 16 last, so that the
// last pass, stride 1, is a radix-16 pass whenever 16 divides n); returns s
// (-1 if n is not a supported length).
HD int dif_plan(int n, int R[kMaxDifPasses], int S[kMaxDifPasses]) {
    int rad[32];
    const int s = fft_radices(n, rad);
    if (s < 0 || s > kMaxDifPasses) return -1;
    int L = n;
    for (int p = 0; p < s; ++p) {
        R[p] = rad[s - 1 - p];
        S[p] = L / R[p];
        L = S[p];
    }
    return s;
}

// A layout of 16-byte elements that no kernel uses any more either (padn took
// its place): the low three bits XOR-ed with bits 4..6, a permutation of every
// aligned group of 8 (and the identity below 16).
HD int swc(int i) { return i ^ ((i >> 4) & 7); }

// First position of butterfly b's elements in pass (R, S): q L + m.
HD int dif_base(int R, int S, int b) {
    const int q = b / S;
    return q * S * R + (b - q * S);
}

// Frequency held at position pos after the forward passes.
HD int dif_freq(int s, const int R[kMaxDifPasses], const int S[kMaxDifPasses], int pos) {
    int f = 0, w = 1;
    for (int p = 0; p < s; ++p) {
        const int k = pos / S[p];
        pos -= k * S[p];
        f += k * w;
        w *= R[p];
    }
    return f;
}

// Position holding frequency f after the forward passes (inverse of
// dif_freq): the digits of f in the mixed radix R_0, R_1, ... (least
// significant first) weighted by the strides.
HD int dif_pos(int s, const int R[kMaxDifPasses], const int S[kMaxDifPasses], int f) {
    int pos = 0;
    for (int p = 0; p < s; ++p) {
        const int q = f / R[p];
        pos += (f - q * R[p]) * S[p];
        f = q;
    }
    return pos;
}

// Shared-memory layouts of the kernels' sequences of 16-byte elements (the same
// element of two columns or rows, fft2.cuh). Lengths of 32 and more that are
// multiples of 16: element i at padn(i) = i + i / 16 + i / S0, S0 = 1 << ls0
// the first pass's stride (a multiple of 16). For a pass of stride S < S0, a
// multiple of 16, the addresses of a butterfly advance by the constant S + S /
// 16, those of the first pass by first_step, those of the last pass by one.
// The other lengths (small ones): pad16.
HD int pad16(int i) { return i + (i >> 4); }
HD int padn(int i, int ls0) { return i + (i >> 4) + (i >> ls0); }
HD int first_step(int ls0) { return (1 << ls0) + (1 << ls0 >> 4) + 1; }
HD bool fft_by16(int n) { return n >= 32 && (n & 15) == 0; }
// Elements between sequences of length n, R0 the first pass's radix.
HD int seq_pitch(int n, int R0) { return fft_by16(n) ? n + (n >> 4) + R0 : n + (n >> 4) + 1; }

// padn(dif_pos(k)) of a length fft_by16 serves: the digits of k times padded
// strides. lst: log2 of the strides.
struct FreqDigits {
    unsigned magic;          // ceil(2^20 / R0): k / R0 = (k magic) >> 20, exact while the product fits 32 bits, k < 2^12 R0
    int R0, step0, l1, l2, step1, s;
    HD FreqDigits(int passes, int radix0, const int* lst) {
        R0 = radix0;
        magic = ((1u << 20) + R0 - 1) / R0;
        s = passes;
        step0 = first_step(lst[0]);
        l1 = lst[0] - lst[1];                        // log2 of the second radix
        step1 = (1 << lst[1]) + (1 << lst[1] >> 4);
        l2 = s > 2 ? lst[1] - lst[2] : 0;            // log2 of the third
    }
    HD int operator()(int k) const {
        const int q = (int)(((unsigned)k * magic) >> 20), k0 = k - q * R0;
        if (s == 2) return k0 * step0 + q;
        const int k1 = q & ((1 << l1) - 1), r = q >> l1;
        if (s == 3) return k0 * step0 + k1 * step1 + r;
        return k0 * step0 + k1 * step1 + (r & ((1 << l2) - 1)) * 17 + (r >> l2);
    }
};

// Every pass's twiddle table back to back in pass order (the last pass has
// none); returns the number of entries (T may be null to query it).
inline int fft_dif_tables(int n, cf* T) {
    int R[kMaxDifPasses], S[kMaxDifPasses];
    const int s = dif_plan(n, R, S);
    int len = 0;
    for (int p = 0; p < s; ++p) {
        if (T) stage_twiddles(S[p], R[p], T + len);
        len += stage_table_len(S[p], R[p]);
    }
    return len;
}

// Real FFT of length P = 2M through a complex FFT of length M of the packed
// pairs z[n] = x[2n] + i x[2n+1] with transform Z. Unnormalised, without the
// factors 1/2 (they are folded into the kernel spectrum):
//   X[k] = (Z[k] + conj Z[M-k]) - i W^k (Z[k] - conj Z[M-k]),  W = exp(-2 pi i / P),
// Z[M] = Z[0], twP[k] = W^k. The inverse builds, for the pair (k, M-k),
// 0 < k < M, from the half spectrum X (X[M] = 0), Z[k] = E + i O with
//   E = X[k] + conj X[M-k],  O = W^-k (X[k] - conj X[M-k]),
// and W^-(M-k) = -W^k gives Z[M-k] from the same two values.
// k = 0 of the inverse: X[0] real part only (its imaginary part and X[M]
// are zero for a real signal), Z[0] = X0 + i X0.
HD cf c2r_pre_dc(cf X0) { return {X0.x, X0.x}; }

// a + conj(b), a - conj(b) and conj(a - i b).
HD cf cadd_conj(cf a, cf b) { return {a.x + b.x, a.y - b.y}; }
HD cf csub_conj(cf a, cf b) { return {a.x - b.x, a.y + b.y}; }
HD cf conj_subi(cf a, cf b) { return {a.x + b.y, b.x - a.y}; }

// The forward step from Zk = Z[k], Zmk = Z[M-k] and w = W^k, for any element
// type with these operations (two rows at once in the kernels);
template <class C>
HD C r2c_post(C Zk, C Zmk, C w) { return csubi(cadd_conj(Zk, Zmk), cmul(csub_conj(Zk, Zmk), w)); }
// with Z in digit-reversed order, read at positions pk and pmk;
HD cf r2c_post_at(const cf* Z, int pk, int pmk, int k, const cf* twP) { return r2c_post(Z[pk], Z[pmk], twP[k]); }
// the inverse step takes a = X[k], b = X[M-k] and w = W^k and gives the
// packed inputs Z[k] (zk) and Z[M-k] (zmk), 0 < k < M: with E = a + conj(b)
// and O = conj(w) (a - conj(b)), E + i O and conj(E - i O).
template <class C>
HD void c2r_pre_vals(C a, C b, C w, C& zk, C& zmk) {
    const C e = cadd_conj(a, b), o = cmulc(csub_conj(a, b), w);
    zk = caddi(e, o);
    zmk = conj_subi(e, o);
}

}  // namespace hr
