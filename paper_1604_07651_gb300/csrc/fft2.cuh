// Packed FP32 arithmetic and the shared-memory FFT passes of the column and
// row kernels: two sequences at once, the same element of both in the halves
// of 64-bit register pairs, every operation one add / sub / mul / fma.f32x2.
//
// Why packed: the passes are bound by instruction issue and by fetching
// their straight-line code, not by the FP32 pipe (which takes two cycles for
// a packed operation, so its peak does not change). Packing halves the
// arithmetic, the shared-memory and the address instructions per element:
// an element of two sequences is one 16-byte shared-memory access.
#pragma once

#include "hostdev.h"

namespace hr {

typedef unsigned long long f2;                    // two floats, sequence 0 in the low half

__device__ __forceinline__ f2 pk(float lo, float hi) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 upk(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// One complex element of two sequences: 16 bytes (re0, re1, im0, im1).
struct __align__(16) c2 { f2 re, im; };

// The DFTs' constants as pairs in constant memory: a packed operand cannot be
// an immediate, and building the pair in registers costs two moves per use
// (the column pass at 2048^2: 59 us with built pairs, 55 us with these).
#define HR_PAIR(v) {v, v}, {-(v), -(v)}
__constant__ float2 kPairs[] = {
    HR_PAIR(0.92387953251128674f), HR_PAIR(0.70710678118654752f), HR_PAIR(0.38268343236508977f),
    HR_PAIR(0.86602540378443864676f), HR_PAIR(0.5f), HR_PAIR(0.30901699437494742410f),
    HR_PAIR(0.80901699437494742410f), HR_PAIR(0.95105651629515357212f), HR_PAIR(0.58778525229247312917f),
    HR_PAIR(0.76604444311897803520f), HR_PAIR(0.64278760968653932632f), HR_PAIR(0.17364817766693034885f),
    HR_PAIR(0.98480775301220805936f), HR_PAIR(0.93969262078590838405f), HR_PAIR(0.34202014332566873304f)};
#undef HR_PAIR
// The pair of constant v (a compile-time constant after unrolling: the chain
// folds to one address).
__device__ __forceinline__ f2 pkc(float v) {
    const float a = v < 0.f ? -v : v;
    const int sg = v < 0.f ? 1 : 0;
    const f2* k = reinterpret_cast<const f2*>(kPairs) + sg;
    if (a == 0.92387953251128674f) return k[0];
    if (a == 0.70710678118654752f) return k[2];
    if (a == 0.38268343236508977f) return k[4];
    if (a == 0.86602540378443864676f) return k[6];
    if (a == 0.5f) return k[8];
    if (a == 0.30901699437494742410f) return k[10];
    if (a == 0.80901699437494742410f) return k[12];
    if (a == 0.95105651629515357212f) return k[14];
    if (a == 0.58778525229247312917f) return k[16];
    if (a == 0.76604444311897803520f) return k[18];
    if (a == 0.64278760968653932632f) return k[20];
    if (a == 0.17364817766693034885f) return k[22];
    if (a == 0.98480775301220805936f) return k[24];
    if (a == 0.93969262078590838405f) return k[26];
    if (a == 0.34202014332566873304f) return k[28];
    return pk(v, v);
}

__device__ __forceinline__ c2 cadd(c2 a, c2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ c2 csub(c2 a, c2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ c2 caddi(c2 a, c2 b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }
__device__ __forceinline__ c2 csubi(c2 a, c2 b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }
__device__ __forceinline__ c2 cmulk(c2 a, float re, float im) {
    const f2 r = pkc(re), i = pkc(im), ni = pkc(-im);
    return {fma2(a.im, ni, mul2(a.re, r)), fma2(a.im, r, mul2(a.re, i))};
}
__device__ __forceinline__ c2 caxpy(c2 a, float s, c2 b) {
    const f2 k = pkc(s);
    return {fma2(k, b.re, a.re), fma2(k, b.im, a.im)};
}
__device__ __forceinline__ c2 cscale(float s, c2 a) {
    const f2 k = pkc(s);
    return {mul2(k, a.re), mul2(k, a.im)};
}
// Products with per-sequence factors. A packed operand has no sign modifier
// (negating one costs two more instructions, measured at half the rate), so
// the difference is a multiply and a subtract.
__device__ __forceinline__ c2 cmul(c2 a, c2 w) {
    return {sub2(mul2(a.re, w.re), mul2(a.im, w.im)), fma2(a.im, w.re, mul2(a.re, w.im))};
}
__device__ __forceinline__ c2 cmulc(c2 a, c2 w) {             // a * conj(w)
    return {fma2(a.im, w.im, mul2(a.re, w.re)), sub2(mul2(a.im, w.re), mul2(a.re, w.im))};
}
__device__ __forceinline__ c2 cswap(c2 a) { return {a.im, a.re}; }

__device__ __forceinline__ c2 ld2(const c2* p) {               // shared or global, 16 bytes
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ c2 ldg2(const c2* p) {
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ void st2(c2* p, c2 v) { *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v.re, v.im); }

// Operations of the real-FFT packing (hostdev.h).
__device__ __forceinline__ c2 cadd_conj(c2 a, c2 b) { return {add2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ c2 csub_conj(c2 a, c2 b) { return {sub2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ c2 conj_subi(c2 a, c2 b) { return {add2(a.re, b.im), sub2(b.re, a.im)}; }

// --------------------------------------------------------------------------
// Passes of the in-place FFT pair (dif_plan) on sequences of 16-byte elements
// in shared memory, element i at padn(i) = i + i / 16 + i / S0 (hostdev.h; S0
// the first pass's stride): the quarter warps of every pass (consecutive
// elements, stride 16, and the stride-1 pass's 16 elements per thread) touch
// eight different 16-byte bank groups, and the odd step of the first pass
// spreads the frequencies of neighbouring digits, which the row kernels read
// and write, over the banks. Sequences of n elements (n a multiple of 16) back
// to back are one sequence for every pass but the first and last.
//
// Every stride is a power of two (the factor 3, 5 or 9 is in pass 0), and a
// length that is a multiple of 16 and longer ends with a radix-16 pass of
// stride 1, so the pass before it (radix R1) has stride 16. Both stay within
// blocks of 16 R1 <= 256 elements: a warp takes 512 consecutive elements (32
// stride-1 butterflies) through the two, and only the first pass needs the
// whole CTA (one barrier each way instead of one per pass).
//
// Radix 16 (two sequences: 64 registers of data, 15 warps per SM) against
// radix 8 (30 warps): the column pass at 2048^2 takes 49 us against 62 us,
// radix 8 moving nearly twice the bytes through shared memory.
//
// Swapped form: with s(z) = the exchange of real and imaginary part,
// IDFT(x) = s(DFT(s(x))) and s(x conj(w)) = s(x) w. The inverse passes run
// the forward butterflies and twiddles on exchanged data; the exchange itself
// is a renaming where data enter and leave.
// --------------------------------------------------------------------------
// Twiddle product of a butterfly: x[k] *= T[(k - 1) S] (T at the butterfly's
// m; entries (wr, wr, wi, wi)).
template <int R>
__device__ __forceinline__ void twiddle2(c2* x, const c2* T, int S) {
#pragma unroll
    for (int k = 1; k < R; ++k) x[k] = cmul(x[k], ld2(T + (k - 1) * S));
}

// Pass of radix R and stride S = 1 << ls (a multiple of 16, below the first
// pass's 1 << ls0) over the butterflies b0, b0 + step, ... below nbf. INV:
// twiddles before the butterfly.
template <int R, bool INV>
__device__ __forceinline__ void pass16(c2* A, int b0, int nbf, int step, int ls, int ls0, const c2* __restrict__ T) {
    const int S = 1 << ls, SP = S + (S >> 4);
    for (int b = b0; b < nbf; b += step) {
        const int q = b >> ls, m = b & (S - 1);
        c2* Z = A + padn(q * (S * R) + m, ls0);
        c2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = ld2(Z + r * SP);
        if (INV) twiddle2<R>(x, T + m, S);
        dft_small<R>(x, -1);
        if (!INV) twiddle2<R>(x, T + m, S);
#pragma unroll
        for (int r = 0; r < R; ++r) st2(Z + r * SP, x[r]);
    }
}
// Who shares the last two passes: a warp and 512 elements at a time, or the
// whole CTA where that would leave warps without elements.
struct Team {
    bool whole;
    int me, n, chunk, first, next;       // my index and the team's size; elements per round, mine and the next round's
    __device__ __forceinline__ Team(int nall, int t, int nt) {
        whole = nall < 12 * nt;
        me = whole ? t : t & 31;
        n = whole ? nt : 32;
        chunk = whole ? 16 * nt : 512;
        first = whole ? 0 : (t >> 5) * 512;
        next = 16 * nt;
    }
    __device__ __forceinline__ void sync() const {
        if (whole) __syncthreads();
        else __syncwarp();
    }
};
// The stride-16 pass of a team's elements from e0 on (nall in all).
template <int R, bool INV>
__device__ __forceinline__ void team_mid(c2* A, const Team& w, int e0, int nall, int ls0, const c2* __restrict__ T) {
    pass16<R, INV>(A, e0 / R + w.me, min(nall, e0 + w.chunk) / R, w.n, 4, ls0, T);
}
#define HR_MID_CASES(CALL)        \
    case 16: CALL(16); break;     \
    case 8: CALL(8); break;       \
    case 4: CALL(4); break;       \
    default: CALL(2); break;
// The stride-1 radix-16 butterfly of 16 consecutive elements (no twiddles).
__device__ __forceinline__ void pass16_last(c2* Z) {
    c2 x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = ld2(Z + r);
    dft_small<16>(x, -1);
#pragma unroll
    for (int r = 0; r < 16; ++r) st2(Z + r, x[r]);
}
// Pass of any stride over nseq sequences of nbf butterflies, `pitch` elements
// apart.
template <int R, bool INV>
__device__ __forceinline__ void pass_any(c2* A0, int pitch, int nseq, int nbf, int S, const c2* __restrict__ T, int t, int nt) {
    for (int i = t; i < nseq * nbf; i += nt) {
        const int sq = i / nbf, b = i - sq * nbf;
        const int q = b / S, m = b - q * S, base = q * S * R + m;
        c2* A = A0 + sq * pitch;
        c2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = ld2(A + pad16(base + r * S));
        if (INV && S > 1) twiddle2<R>(x, T + m, S);
        dft_small<R>(x, -1);
        if (!INV && S > 1) twiddle2<R>(x, T + m, S);
#pragma unroll
        for (int r = 0; r < R; ++r) st2(A + pad16(base + r * S), x[r]);
    }
}

}  // namespace hr
