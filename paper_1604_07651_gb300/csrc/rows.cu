// Row transforms: the real FFT of the lattice rows and its inverse (first and
// last part of Eq. (7)/(16)), and the adjoint interpolation's theta spread.
//
// The real FFT of a lattice row of length Prho is a complex FFT of the M =
// Prho / 2 packed pairs z[n] = x[2n] + i x[2n+1], by the in-place passes of
// dif_plan(M). Two neighbouring rows run as one sequence of 16-byte elements
// with packed arithmetic (fft2.cuh); a CTA holds a band of P.Re rows, Re / 2
// such pairs, back to back in shared memory. The forward leaves Z in
// digit-reversed order; the real-FFT post-processing reads Z[k] and Z[M - k]
// at their positions (FreqPos), and the inverse's pre-processing writes the
// packed pairs straight to theirs. The last row's partner beyond an odd
// lattice is a copy of it whose result is not used.
#include "device.cuh"
#include "fft2.cuh"

namespace hr {

constexpr int kRowThreadsMax = 256;   // two such CTAs fill the registers (128 per thread)
constexpr int kBandCols = 64;        // output columns whose theta weights the band kernel holds at once

__host__ __device__ __forceinline__ size_t rows_smem(const PieceDev& P) {
    return (size_t)(P.Re / 2) * seq_pitch(P.Prho / 2, P.fftM.rad[0]) * sizeof(c2);
}

// Forward pass 0 reading np pairs of lattice rows (Nr reals each, row pitch
// lp, nrows of them exist) from global memory. NZ: the inputs from NZ on are
// zero padding and not read.
template <int R, int NZ>
__device__ __forceinline__ void row_first(c2* A, const float* lat, int lp, int Nr, int nrows, int np, int ls,
                                          const c2* __restrict__ T, int t, int nt) {
    const int S = 1 << ls, SP = first_step(ls);
#pragma unroll 2
    for (int i = t; i < np << ls; i += nt) {
        const int pr = i >> ls, m = i & (S - 1);
        const float* s0 = lat + (size_t)(2 * pr) * lp + 2 * m;
        const float* s1 = 2 * pr + 1 < nrows ? s0 + lp : s0;
        c2 x[R];
#pragma unroll
        for (int r = 0; r < NZ; ++r) {
            const int n2 = 2 * (m + r * S);
            float2 a = make_float2(0.f, 0.f), b = a;
            if (n2 < Nr) {
                a = __ldca(reinterpret_cast<const float2*>(s0 + 2 * r * S));
                b = __ldca(reinterpret_cast<const float2*>(s1 + 2 * r * S));
                if (n2 + 1 == Nr) a.y = b.y = 0.f;       // the pitch's padding
            }
            x[r] = {pk(a.x, b.x), pk(a.y, b.y)};
        }
        dft_zeros<R, NZ>(x, -1);
#pragma unroll
        for (int k = 1; k < R; ++k) x[k] = cmul(x[k], ldg2(T + (k - 1) * S + m));
        c2* Z = A + pr * (SP * R) + pad16(m);
#pragma unroll
        for (int r = 0; r < R; ++r) st2(Z + r * SP, x[r]);
    }
}
template <int R>
__device__ __forceinline__ void row_first_any(c2* A, const float* lat, int lp, int Nr, int nrows, int np, int ls,
                                              const c2* T, int t, int nt) {
    constexpr int H = (R + 1) / 2;
    if (Nr > 2 * H << ls) row_first<R, R>(A, lat, lp, Nr, nrows, np, ls, T, t, nt);
    else row_first<R, H>(A, lat, lp, Nr, nrows, np, ls, T, t, nt);
}

// Inverse pass 0 (exchanged data) writing the first Nr reals of the rows.
template <int R, int NZ>
__device__ __forceinline__ void row_last(const c2* A, float* lat, int lp, int Nr, int nrows, int np, int ls,
                                         const c2* __restrict__ T, int t, int nt) {
    const int S = 1 << ls, SP = first_step(ls);
    for (int i = t; i < np << ls; i += nt) {
        const int pr = i >> ls, m = i & (S - 1);
        const c2* Z = A + pr * (SP * R) + pad16(m);
        c2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = ld2(Z + r * SP);
#pragma unroll
        for (int k = 1; k < R; ++k) x[k] = cmul(x[k], ldg2(T + (k - 1) * S + m));
        dft_small<R>(x, -1);
        float* d0 = lat + (size_t)(2 * pr) * lp + 2 * m;
#pragma unroll
        for (int r = 0; r < NZ; ++r) {
            if (2 * (m + r * S) >= Nr) continue;
            const float2 re = upk(x[r].im), im = upk(x[r].re);
            *reinterpret_cast<float2*>(d0 + 2 * r * S) = make_float2(re.x, im.x);
            if (2 * pr + 1 < nrows) *reinterpret_cast<float2*>(d0 + lp + 2 * r * S) = make_float2(re.y, im.y);
        }
    }
}
template <int R>
__device__ __forceinline__ void row_last_any(const c2* A, float* lat, int lp, int Nr, int nrows, int np, int ls, const c2* T,
                                             int t, int nt) {
    constexpr int H = (R + 1) / 2;
    if (Nr > 2 * H << ls) row_last<R, R>(A, lat, lp, Nr, nrows, np, ls, T, t, nt);
    else row_last<R, H>(A, lat, lp, Nr, nrows, np, ls, T, t, nt);
}

// Forward passes 1 .. s-1 of a length fft_by16 serves: the last two per team.
__device__ __forceinline__ void row_passes(c2* A, const FftPlan& fp, int np, const c2* T, int t, int nt) {
    const int nall = np * fp.n, s = fp.nst, ls0 = fp.lst[0];
    if (s == 4) {
        pass16<4, false>(A, t, nall >> 2, nt, fp.lst[1], ls0, T + fp.tw[1]);
        __syncthreads();
    }
    const Team w(nall, t, nt);
    for (int e0 = w.first; e0 < nall; e0 += w.next) {
        if (s >= 3) {
#define HR_RF(RR) team_mid<RR, false>(A, w, e0, nall, ls0, T + fp.tw[s - 2])
            switch (fp.rad[s - 2]) { HR_MID_CASES(HR_RF) }
#undef HR_RF
            w.sync();
        }
        const int b = (e0 >> 4) + w.me;
        if (16 * b < nall) pass16_last(A + padn(16 * b, ls0));
    }
    __syncthreads();
}
// Inverse passes s-1 .. 1.
__device__ __forceinline__ void row_passes_inv(c2* A, const FftPlan& fp, int np, const c2* T, int t, int nt) {
    const int nall = np * fp.n, s = fp.nst, ls0 = fp.lst[0];
    const Team w(nall, t, nt);
    for (int e0 = w.first; e0 < nall; e0 += w.next) {
        const int b = (e0 >> 4) + w.me;
        if (16 * b < nall) pass16_last(A + padn(16 * b, ls0));
        if (s >= 3) {
            w.sync();
#define HR_RF(RR) team_mid<RR, true>(A, w, e0, nall, ls0, T + fp.tw[s - 2])
            switch (fp.rad[s - 2]) { HR_MID_CASES(HR_RF) }
#undef HR_RF
        }
    }
    __syncthreads();
    if (s == 4) {
        pass16<4, true>(A, t, nall >> 2, nt, fp.lst[1], ls0, T + fp.tw[1]);
        __syncthreads();
    }
}
// All passes of any length, in shared memory.
template <bool INV>
__device__ __forceinline__ void row_passes_any(c2* A, int pitch, const FftPlan& fp, int np, const c2* T, int t, int nt) {
    for (int i = 0; i < fp.nst; ++i) {
        const int p = INV ? fp.nst - 1 - i : i;
#define HR_RA(RR) pass_any<RR, INV>(A, pitch, np, fp.n / RR, fp.st[p], T + fp.tw[p], t, nt)
        switch (fp.rad[p]) { HR_RADIX_CASES(HR_RA) }
#undef HR_RA
        __syncthreads();
    }
}

// Where the forward passes leave frequency k (dif_pos): for lengths fft_by16
// serves computed (a table read would put its latency before every access),
// else from the plan's table.
struct FreqPos {
    const int* tab;
    FreqDigits digits;
    __device__ __forceinline__ FreqPos(const PieceDev& P)
        : tab(fft_by16(P.fftM.n) ? nullptr : P.rpos), digits(P.fftM.nst, P.fftM.rad[0], P.fftM.lst) {}
    __device__ __forceinline__ int operator()(int k) const { return tab ? __ldg(tab + k) : digits(k); }
};

// Real-FFT post-processing of the band's transformed rows into the half
// spectrum, bins k <= k2max: a thread takes the two bins of a column block for
// a pair of rows, and writes two neighbouring 16-byte elements.
__device__ __forceinline__ void rows_post(const PieceDev& P, const c2* A, int pitch, int mb, int np, int t, int nt) {
    const int M = P.Prho / 2;
    const FreqPos pos(P);
    const float inv_np = 1.0f / (float)np;
#pragma unroll 2
    for (int i = t; i < P.nkb * np; i += nt) {
        const int kb = (int)(((float)i + 0.5f) * inv_np);       // exact for i < 2^22
        const int pr = i - kb * np;
        const c2* Z = A + pr * pitch;
        c2 X[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int k = min(2 * kb + c, M - 1);
            const float2 w = __ldg(reinterpret_cast<const float2*>(P.twP) + k);
            X[c] = r2c_post(ld2(Z + pos(k)), ld2(Z + pos(k == 0 ? 0 : M - k)), c2{pk(w.x, w.x), pk(w.y, w.y)});
        }
        const float2 a = upk(X[0].re), b = upk(X[1].re), c = upk(X[0].im), d = upk(X[1].im);
        float4* e = P.spec + (size_t)kb * P.sp + mb + 2 * pr;   // the partner beyond the last row is padding
        e[0] = make_float4(a.x, b.x, c.x, d.x);
        e[1] = make_float4(a.y, b.y, c.y, d.y);
    }
}

// Inverse: the real-FFT pre-processing of the band's half-spectrum rows
// (bins above k2max are zero; elements (im0, im1, re0, re1) of the column
// pass), pairs (k, M - k) for 0 <= k <= M/2, written exchanged to their
// digit-reversed positions in shared memory. A thread takes two bins of a
// pair of rows at a time, U times with all their loads (from L2) in flight.
__device__ __forceinline__ c2 spec_bin(float4 r0, float4 r1, int c) {   // bin c of an element of two rows
    return c ? c2{pk(r0.w, r1.w), pk(r0.y, r1.y)} : c2{pk(r0.z, r1.z), pk(r0.x, r1.x)};
}
__device__ __forceinline__ void rows_pre(const PieceDev& P, c2* A, int pitch, int mb, int np, int t, int nt) {
    const int M = P.Prho / 2, half = M / 2, nk = P.k2max + 1;
    const FreqPos pos(P);
    const float inv_np = 1.0f / (float)np;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const int total = (half / 2 + 1) * np;
    constexpr int U = 2;
    for (int i0 = t; i0 < total; i0 += U * nt) {
        float4 a0[U], a1[U], b0[U][2], b1[U][2];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * nt;
            const int kb = (int)(((float)i + 0.5f) * inv_np);   // exact for i < 2^22
            const float4* row = P.spec + mb + 2 * (i - kb * np);
            a0[u] = a1[u] = b0[u][0] = b0[u][1] = b1[u][0] = b1[u][1] = zero;
            if (i >= total) continue;
            if (2 * kb < nk) {
                a0[u] = __ldca(row + (size_t)kb * P.sp);
                a1[u] = __ldca(row + (size_t)kb * P.sp + 1);
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int k2 = M - 2 * kb - c;
                if (k2 >= 0 && k2 < nk) {
                    b0[u][c] = __ldca(row + (size_t)(k2 >> 1) * P.sp);
                    b1[u][c] = __ldca(row + (size_t)(k2 >> 1) * P.sp + 1);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * nt;
            if (i >= total) continue;
            const int kb = (int)(((float)i + 0.5f) * inv_np);
            c2* Z = A + (i - kb * np) * pitch;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int k = 2 * kb + c, k2 = M - k;
                if (k > half) continue;
                c2 a = spec_bin(a0[u], a1[u], c);
                if (k >= nk) a = {0ull, 0ull};
                if (k == 0) {                                   // Z[0] = X0 + i X0, X0 real
                    st2(Z + pos(0), c2{a.re, a.re});
                    continue;
                }
                const c2 b = spec_bin(b0[u][c], b1[u][c], k2 & 1);
                const float2 w = __ldg(reinterpret_cast<const float2*>(P.twP) + k);
                c2 zk, zmk;
                c2r_pre_vals(a, b, c2{pk(w.x, w.x), pk(w.y, w.y)}, zk, zmk);
                st2(Z + pos(k), cswap(zk));
                st2(Z + pos(k2), cswap(zmk));
            }
        }
    }
}

// Real FFT of a band of lattice rows (P.lat, zero-padded to Prho) into the
// half spectrum (first half of Eq. (7)/(16)).
template <class Src>
__global__ void __launch_bounds__(kRowThreadsMax, 2) k_rows_r2c(const __grid_constant__ Src B) {
    int bx;
    const PieceDev& P = piece_of(B, bx);
    chain_next<4>();
    chain_wait<4>();
    if (rows_smem(P) > dyn_smem_bytes()) return;
    const int mb = bx * P.Re, nrows = min(P.Re, P.Ntheta - mb), np = (nrows + 1) / 2;
    const int M = P.Prho / 2, pitch = seq_pitch(M, P.fftM.rad[0]), t = threadIdx.x, nt = blockDim.x;
    const FftPlan& fp = P.fftM;
    const c2* T = reinterpret_cast<const c2*>(P.twM);
    const float* lat = P.lat + (size_t)mb * P.lp;
    c2* A = reinterpret_cast<c2*>(smem_f);
    if (fft_by16(M)) {
        const int ls0 = fp.lst[0];
#define HR_RL(RR) row_first_any<RR>(A, lat, P.lp, P.Nrho, nrows, np, ls0, T, t, nt)
        switch (fp.rad[0]) { HR_RADIX_CASES(HR_RL) }
#undef HR_RL
        __syncthreads();
        row_passes(A, fp, np, T, t, nt);
    } else {
        for (int i = t; i < np * M; i += nt) {
            const int pr = i / M, n = i - pr * M;
            const float* s0 = lat + (size_t)(2 * pr) * P.lp;
            const float* s1 = 2 * pr + 1 < nrows ? s0 + P.lp : s0;
            auto at = [&](const float* s, int j) { return j < P.Nrho ? __ldca(s + j) : 0.f; };
            st2(A + pr * pitch + pad16(n), c2{pk(at(s0, 2 * n), at(s1, 2 * n)), pk(at(s0, 2 * n + 1), at(s1, 2 * n + 1))});
        }
        __syncthreads();
        row_passes_any<false>(A, pitch, fp, np, T, t, nt);
    }
    rows_post(P, A, pitch, mb, np, t, nt);
}

// Inverse real FFT of a band of rows from the half spectrum (bins <= k2max,
// the rest zero) into the real lattice P.lat[Ntheta][lp].
template <class Src>
__global__ void __launch_bounds__(kRowThreadsMax, 2) k_rows_c2r(const __grid_constant__ Src B) {
    int bx;
    const PieceDev& P = piece_of(B, bx);
    chain_next<4>();
    chain_wait<4>();
    if (rows_smem(P) > dyn_smem_bytes()) return;
    const int mb = bx * P.Re, nrows = min(P.Re, P.Ntheta - mb), np = (nrows + 1) / 2;
    const int M = P.Prho / 2, pitch = seq_pitch(M, P.fftM.rad[0]), t = threadIdx.x, nt = blockDim.x;
    const FftPlan& fp = P.fftM;
    const c2* T = reinterpret_cast<const c2*>(P.twM);
    float* lat = P.lat + (size_t)mb * P.lp;
    c2* A = reinterpret_cast<c2*>(smem_f);
    rows_pre(P, A, pitch, mb, np, t, nt);
    __syncthreads();
    if (fft_by16(M)) {
        row_passes_inv(A, fp, np, T, t, nt);
        const int ls0 = fp.lst[0];
#define HR_RW(RR) row_last_any<RR>(A, lat, P.lp, P.Nrho, nrows, np, ls0, T, t, nt)
        switch (fp.rad[0]) { HR_RADIX_CASES(HR_RW) }
#undef HR_RW
    } else {
        row_passes_any<true>(A, pitch, fp, np, T, t, nt);
        for (int i = t; i < np * M; i += nt) {
            const int pr = i / M, n = i - pr * M;
            const c2 z = ld2(A + pr * pitch + pad16(n));
            const float2 re = upk(z.im), im = upk(z.re);
            float* d = lat + (size_t)(2 * pr) * P.lp + 2 * n;
            const bool two = 2 * pr + 1 < nrows;
            if (2 * n < P.Nrho) {
                d[0] = re.x;
                if (two) d[P.lp] = re.y;
            }
            if (2 * n + 1 < P.Nrho) {
                d[1] = im.x;
                if (two) d[P.lp + 1] = im.y;
            }
        }
    }
}

// The theta spread of the adjoint interpolation for NP pairs of rows:
// G'[m][n] = sum_l B(theta_l - theta_m) h_l[n] over the band's columns in
// order, each thread four rho cells of every row, into the rows' packed form
// in shared memory (elements below nz; the rest is zero padding the first pass
// skips). The weights of kBandCols columns at a time sit in shared memory as
// pairs, so a column costs a thread one 16-byte load of its profile, one
// shared load and four packed operations per two rows.
template <int NT, int NP>
__device__ __forceinline__ void band_spread(const PieceDev& P, c2* A, int pitch, int mb, int nz, int2 lr, f2 (*wt)[2 * NP],
                                            int t, int nt) {
    const int hp = P.hpitch, M = P.Prho / 2;
    const int ls0 = fft_by16(M) ? P.fftM.lst[0] : 30;            // 30: pass_any's layout
    const float* h = P.prof;
    const int ncol = max(0, lr.y - lr.x + 1);
    for (int n0 = 0; 2 * n0 < nz; n0 += nt) {
        const int n4 = n0 + t;
        const bool in = 4 * n4 < hp;
        f2 acc[2 * NP][2];
#pragma unroll
        for (int r = 0; r < 2 * NP; ++r) acc[r][0] = acc[r][1] = 0ull;
        for (int l0 = 0; l0 < ncol; l0 += kBandCols) {
            const int nl = min(kBandCols, ncol - l0);
            if (n0 == 0 || ncol > kBandCols) {
                if (n0 > 0 || l0 > 0) __syncthreads();
                for (int i = t; i < nl * 2 * NP; i += nt) {
                    const int c = i / (2 * NP), r = i - c * (2 * NP);
                    const int lc = lr.x + l0 + c - P.l_lo;
                    const int a = mb + r - __ldg(P.colm0 + lc);          // the column's tap of row r
                    float w = 0.f;
                    if (a >= 0 && a < 4) w = __ldg(reinterpret_cast<const float*>(P.colw + lc) + a);
                    else if (NT > 4 && a >= 4 && a < NT) w = __ldg(reinterpret_cast<const float*>(P.colw2 + lc) + a - 4);
                    wt[c][r] = pk(w, w);
                }
                __syncthreads();
            }
            if (in) {
                const float* hl = h + (size_t)(lr.x + l0 - P.l_lo) * hp + 4 * n4;
#pragma unroll 4
                for (int c = 0; c < nl; ++c) {
                    const ulonglong2 v = __ldca(reinterpret_cast<const ulonglong2*>(hl + (size_t)c * hp));
#pragma unroll
                    for (int r = 0; r < 2 * NP; ++r) {
                        acc[r][0] = fma2(wt[c][r], v.x, acc[r][0]);
                        acc[r][1] = fma2(wt[c][r], v.y, acc[r][1]);
                    }
                }
            }
        }
        if (2 * n4 < nz) {
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                c2* Z = A + p * pitch;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 a = upk(acc[2 * p][e]), b = upk(acc[2 * p + 1][e]);
                    if (2 * n4 + e < M) st2(Z + padn(2 * n4 + e, ls0), c2{pk(a.x, b.x), pk(a.y, b.y)});
                }
            }
        }
    }
}

// Pass 0 of the spread rows in shared memory. NZ: the inputs from NZ on are
// zero padding and not read.
template <int R, int NZ>
__device__ __forceinline__ void band_first(c2* A, int np, int ls, const c2* __restrict__ T, int t, int nt) {
    const int S = 1 << ls, SP = first_step(ls);
    for (int i = t; i < np << ls; i += nt) {
        const int m = i & (S - 1);
        c2* Z = A + (i >> ls) * (SP * R) + pad16(m);
        c2 x[R];
#pragma unroll
        for (int r = 0; r < NZ; ++r) x[r] = ld2(Z + r * SP);
        dft_zeros<R, NZ>(x, -1);
#pragma unroll
        for (int k = 1; k < R; ++k) x[k] = cmul(x[k], ldg2(T + (k - 1) * S + m));
#pragma unroll
        for (int r = 0; r < R; ++r) st2(Z + r * SP, x[r]);
    }
}
template <int R>
__device__ __forceinline__ void band_first_any(c2* A, int np, int ls, bool half, const c2* T, int t, int nt) {
    if (half) band_first<R, (R + 1) / 2>(A, np, ls, T, t, nt);
    else band_first<R, R>(A, np, ls, T, t, nt);
}

// One band of lattice rows: G' rows from the profiles of the band's candidate
// columns, then the row FFT into the half spectrum.
template <class Src, int NT>
__global__ void __launch_bounds__(kRowThreadsMax, 2) k_band_rows(const __grid_constant__ Src B) {
    __shared__ f2 wt[kBandCols * kMaxBandRows];
    int band;
    const PieceDev& P = piece_of(B, band);
    chain_next<4>();
    chain_wait<4>();
    if (rows_smem(P) > dyn_smem_bytes()) return;
    const int mb = band * P.Re, npb = P.Re / 2, np = (min(P.Re, P.Ntheta - mb) + 1) / 2;
    const int M = P.Prho / 2, pitch = seq_pitch(M, P.fftM.rad[0]), t = threadIdx.x, nt = blockDim.x;
    const FftPlan& fp = P.fftM;
    const c2* T = reinterpret_cast<const c2*>(P.twM);
    const int2 lr = __ldg(P.lband + band);
    c2* A = reinterpret_cast<c2*>(smem_f);
    const bool by16 = fft_by16(M);
    const int nh = by16 ? ((fp.rad[0] + 1) / 2) << fp.lst[0] : M;   // elements the first pass reads at most half the data
    const bool half = by16 && P.hpitch <= 2 * nh;
    const int nz = half ? nh : M;
    if (npb == 3) band_spread<NT, 3>(P, A, pitch, mb, nz, lr, reinterpret_cast<f2(*)[6]>(wt), t, nt);
    else if (npb == 2) band_spread<NT, 2>(P, A, pitch, mb, nz, lr, reinterpret_cast<f2(*)[4]>(wt), t, nt);
    else band_spread<NT, 1>(P, A, pitch, mb, nz, lr, reinterpret_cast<f2(*)[2]>(wt), t, nt);
    __syncthreads();
    if (by16) {
#define HR_RB(RR) band_first_any<RR>(A, np, fp.lst[0], half, T, t, nt)
        switch (fp.rad[0]) { HR_RADIX_CASES(HR_RB) }
#undef HR_RB
        __syncthreads();
        row_passes(A, fp, np, T, t, nt);
    } else {
        row_passes_any<false>(A, pitch, fp, np, T, t, nt);
    }
    rows_post(P, A, pitch, mb, np, t, nt);
}

// --------------------------------------------------------------------------
// Launchers
// --------------------------------------------------------------------------
size_t rows_smem_bytes(const PieceDev& P) { return rows_smem(P); }

int max_row_pairs(const PieceDev& P, size_t smem_max) {
    const size_t fixed = sizeof(f2) * kBandCols * kMaxBandRows + 1024;   // the band kernel's weights
    return (int)std::min<size_t>(kMaxBandRows / 2, (smem_max - fixed) / (seq_pitch(P.Prho / 2, P.fftM.rad[0]) * sizeof(c2)));
}

// Threads of a row-kernel CTA: a launch that leaves SMs short of CTAs takes
// the most (its time is one CTA's latency, and the passes other than the
// radix-16 ones have work for all). Else the multiple of 32 that keeps most of
// the launch's threads busy over whole rounds of radix-16 butterflies, times
// the share of the SM's 512 threads (at 128 registers) that its CTAs fill
// given their shared memory.
int rows_threads(const PieceDev* P, int n, size_t smem) {
    long blocks = 0;
    for (int k = 0; k < n; ++k) blocks += P[k].nbands;
    if (blocks <= 2 * 152) return kRowThreadsMax;
    int best = 128;
    double best_score = 0;
    for (int tpb = 64; tpb <= kRowThreadsMax; tpb += 32) {
        double work = 0, slots = 0;
        for (int k = 0; k < n; ++k) {
            const double bf = 0.5 * P[k].Re * (P[k].Prho / 32.0);
            work += P[k].nbands * bf;
            slots += P[k].nbands * std::max(1.0, std::ceil(bf / tpb)) * tpb;
        }
        const size_t per_sm = std::min<size_t>(std::min<size_t>(512 / tpb, 32), smem ? (size_t)(227 << 10) / (smem + 4096) : 32);
        const double score = work / slots * std::min(1.0, (double)(per_sm * tpb) / 512);
        if (score > best_score * 1.02) {
            best_score = score;
            best = tpb;
        }
    }
    return best;
}

// One stage over n <= kMaxBatch pieces (descriptors as a parameter) or over
// a device-resident batch (descriptors and block map in device memory).
template <class Src>
static int set_and_launch(void (*kern)(Src), int nb, int tpb, size_t sm, const Src& B, void* stream) {
    if (int e = set_smem((const void*)kern, sm)) return e;
    return nb > 0 ? launch_chain(4, kern, nb, tpb, sm, stream, B) : 0;
}
static size_t rows_smem_max(const PieceDev* P, int n) {
    size_t m = 0;
    for (int k = 0; k < n; ++k) m = std::max(m, rows_smem(P[k]));
    return m;
}

int launch_rows_r2c(const PieceDev* P, int n, int tpb, void* stream) {
    PieceBatch B;
    const int nb = make_batch(P, n, B, [](const PieceDev& q) { return q.nbands; });
    return set_and_launch(k_rows_r2c<PieceBatch>, nb, tpb, rows_smem_max(P, n), B, stream);
}

int launch_band_rows(const PieceDev* P, int n, int tpb, void* stream) {
    PieceBatch B;
    const int nb = make_batch(P, n, B, [](const PieceDev& q) { return q.nbands; });
    const size_t sm = rows_smem_max(P, n);
    if (P[0].ntaps == 6) return set_and_launch(k_band_rows<PieceBatch, 6>, nb, tpb, sm, B, stream);
    if (P[0].ntaps == 4) return set_and_launch(k_band_rows<PieceBatch, 4>, nb, tpb, sm, B, stream);
    return (int)cudaErrorInvalidValue;
}

int launch_rows_c2r(const PieceDev* P, int n, int tpb, void* stream) {
    PieceBatch B;
    const int nb = make_batch(P, n, B, [](const PieceDev& q) { return q.nbands; });
    return set_and_launch(k_rows_c2r<PieceBatch>, nb, tpb, rows_smem_max(P, n), B, stream);
}

int launch_rows_r2c_dev(const DevBatch& S, int nblocks, int tpb, size_t smem, void* stream) {
    return set_and_launch(k_rows_r2c<DevBatch>, nblocks, tpb, smem, S, stream);
}

int launch_band_rows_dev(const DevBatch& S, int nblocks, int ntaps, int tpb, size_t smem, void* stream) {
    if (ntaps == 6) return set_and_launch(k_band_rows<DevBatch, 6>, nblocks, tpb, smem, S, stream);
    if (ntaps == 4) return set_and_launch(k_band_rows<DevBatch, 4>, nblocks, tpb, smem, S, stream);
    return (int)cudaErrorInvalidValue;
}

int launch_rows_c2r_dev(const DevBatch& S, int nblocks, int tpb, size_t smem, void* stream) {
    return set_and_launch(k_rows_c2r<DevBatch>, nblocks, tpb, smem, S, stream);
}

}  // namespace hr
