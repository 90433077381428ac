// Column pass of the transforms: FFT along theta, product with the kernel
// spectrum, inverse FFT (Eq. (7), (16)-(17)); see k_colconv.
#include "device.cuh"
#include "fft2.cuh"

namespace hr {

// --------------------------------------------------------------------------
// Column pass: FFT along theta, product with K (or conj K), inverse FFT
// (Eq. (16)-(17)). The blocked layout [kb][m] stores the two spectrum columns
// of block kb as one 16-byte element (re0, re1, im0, im1) per lattice row, and
// each thread runs a butterfly of both columns with packed arithmetic
// (fft2.cuh). A CTA takes P.C neighbouring column blocks, as many as give its
// threads a radix-16 butterfly each (one at 2560 and 2304, four at 576).
//
//   pass 0        reads the blocks' Ntheta rows straight from global memory
//                 (the zero padding is never loaded) and writes shared memory;
//   (5120 and longer: one more radix-4 pass over the CTA)
//   per warp      its 512 elements through the stride-16 pass, the stride-1
//                 pass with the product and the inverse stride-16 pass: no
//                 CTA barrier. The stride-1 pass runs the forward butterfly,
//                 the product with K at each element's frequency
//                 (digit-reversed order: no reordering) and the inverse
//                 butterfly in registers;
//   last          inverse pass 0 writing only the Ntheta rows back to global
//                 memory.
// The inverse runs on exchanged real and imaginary parts (fft2.cuh): the
// spectrum leaves as (im0, im1, re0, re1) and the inverse row kernel reads it
// so. The slices of K and the middle passes' twiddles are copied to shared
// memory (cp.async) while pass 0 runs.
// --------------------------------------------------------------------------
// Threads of a CTA: 160, the radix-16 butterflies of a 2560-point column (90 %
// busy at 2304; three CTAs per SM), or more, a butterfly each, for the longer
// columns, of which shared memory holds only one or two per SM.
constexpr int kColThreads = 160;
constexpr int kColThreadsMax = 384;
// Bounds a thread to 128 registers, so that the register file holds three CTAs
// of 160 threads, two of 192 to 256, one of more.
constexpr int kColThreadsReg = 480;
// Twiddles of the middle passes (all but the first and the last), kept in
// shared memory.
__host__ __device__ __forceinline__ int col_twiddles(const FftPlan& fp) {
    return fft_by16(fp.n) && fp.nst >= 3 ? fp.ntw - fp.tw[1] : 0;
}
__host__ __device__ __forceinline__ size_t colconv_smem(const PieceDev& P) {
    return ((size_t)P.C * (seq_pitch(P.Ptheta, P.fftT.rad[0]) + P.k1max + 2) + col_twiddles(P.fftT)) * sizeof(float4);
}

// Pass 0: nc column blocks of Nth rows (row pitch sp between blocks) from
// global to shared memory. LS: log2 of the stride where it is compiled in (8,
// the lengths R * 256: immediate offsets, 2 us of 49 at 2048^2), else 0. NZ: the
// rows from NZ << ls on are zero padding (R, or half of it rounded up, which
// holds whenever the padding is as long as the lattice), so the butterfly
// skips them, and the last pass the outputs there.
template <int R, int LS, int NZ>
__device__ __forceinline__ void col_first(c2* A, const c2* col, int sp, int Nth, int nc, int lsr, const c2* T, int t, int nt) {
    const int ls = LS ? LS : lsr, S = 1 << ls, SP = first_step(ls);
    for (int i = t; i < nc << ls; i += nt) {
        const int cp = i >> ls, m = i & (S - 1);
        const c2* src = col + (size_t)cp * sp + m;
        c2 x[R];
#pragma unroll
        for (int r = 0; r < NZ; ++r) {
            ulonglong2 v = make_ulonglong2(0ull, 0ull);
            if (m + r * S < Nth) v = __ldcg(reinterpret_cast<const ulonglong2*>(src + r * S));
            x[r] = {v.x, v.y};
        }
        dft_zeros<R, NZ>(x, -1);
#pragma unroll
        for (int k = 1; k < R; ++k) x[k] = cmul(x[k], ldg2(T + (k - 1) * S + m));
        c2* Z = A + cp * (SP * R) + pad16(m);
#pragma unroll
        for (int r = 0; r < R; ++r) st2(Z + r * SP, x[r]);
    }
}
// Inverse pass 0, shared to global memory.
template <int R, int LS, int NZ>
__device__ __forceinline__ void col_last(const c2* A, c2* col, int sp, int Nth, int nc, int lsr, const c2* T, int t, int nt) {
    const int ls = LS ? LS : lsr, S = 1 << ls, SP = first_step(ls);
    for (int i = t; i < nc << ls; i += nt) {
        const int cp = i >> ls, m = i & (S - 1);
        const c2* Z = A + cp * (SP * R) + pad16(m);
        c2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = ld2(Z + r * SP);
#pragma unroll
        for (int k = 1; k < R; ++k) x[k] = cmul(x[k], ldg2(T + (k - 1) * S + m));
        dft_small<R>(x, -1);
        c2* dst = col + (size_t)cp * sp + m;
#pragma unroll
        for (int r = 0; r < NZ; ++r)
            if (m + r * S < Nth) st2(dst + r * S, x[r]);
    }
}
template <int R>
__device__ __forceinline__ void col_first_any(c2* A, const c2* col, int sp, int Nth, int nc, int ls, const c2* T, int t, int nt) {
    constexpr int H = (R + 1) / 2;
    if (Nth > H << ls) col_first<R, 0, R>(A, col, sp, Nth, nc, ls, T, t, nt);
    else if (R >= 5 && ls == 8) col_first<R, R >= 5 ? 8 : 0, H>(A, col, sp, Nth, nc, ls, T, t, nt);
    else col_first<R, 0, H>(A, col, sp, Nth, nc, ls, T, t, nt);
}
template <int R>
__device__ __forceinline__ void col_last_any(const c2* A, c2* col, int sp, int Nth, int nc, int ls, const c2* T, int t, int nt) {
    constexpr int H = (R + 1) / 2;
    if (Nth > H << ls) col_last<R, 0, R>(A, col, sp, Nth, nc, ls, T, t, nt);
    else if (R >= 5 && ls == 8) col_last<R, R >= 5 ? 8 : 0, H>(A, col, sp, Nth, nc, ls, T, t, nt);
    else col_last<R, 0, H>(A, col, sp, Nth, nc, ls, T, t, nt);
}

// x K or x conj(K), exchanged.
template <bool ADJ>
__device__ __forceinline__ c2 kernel_product(c2 x, c2 k) { return cswap(ADJ ? cmulc(x, k) : cmul(x, k)); }

// First frequency of stride-1 butterfly bb of its column: the digits of the
// other passes (their strides are powers of two).
__device__ __forceinline__ int col_freq(const FftPlan& fp, int bb) {
    int fb = 0, w = 1;
    for (int p = 0; p + 1 < fp.nst; ++p) {
        const int ld = fp.lst[p] - 4;
        const int k = bb >> ld;
        bb -= k << ld;
        fb += k * w;
        w *= fp.rad[p];
    }
    return fb;
}
// Product at the frequencies fb + nb k of stride-1 butterfly b (below n / 2
// for k < 8; K is even, and the entry after the last of its slice is zero).
template <bool ADJ>
__device__ __forceinline__ void kernel_product16(c2 (&x)[16], const FftPlan& fp, const c2* K, int k1n, int b) {
    const int nb = fp.n >> 4;
    const int cp = (int)(((float)b + 0.5f) / (float)nb);       // exact for b < 2^22
    const int fb = col_freq(fp, b - cp * nb);
    const c2* Kc = K + cp * k1n;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int kk = k < 8 ? fb + nb * k : nb * (16 - k) - fb;
        x[k] = kernel_product<ADJ>(x[k], ld2(Kc + min(kk, k1n - 1)));
    }
}
// The stride-1 pass with the product; the butterfly's code is run twice
// (forward, then inverse on the exchanged product).
template <bool ADJ>
__device__ __forceinline__ void col_kernel(c2* A, const FftPlan& fp, const c2* K, int k1n, int b) {
    c2* Z = A + padn(16 * b, fp.lst[0]);
    c2 x[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = ld2(Z + r);
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        dft_small<16>(x, -1);
        if (h == 0) kernel_product16<ADJ>(x, fp, K, k1n, b);
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) st2(Z + r, x[r]);
}

// The same with the stride-16 passes around it when their radix is 16 too
// (the lengths R * 256), with ONE radix-16 butterfly in the code: the inverse
// pass's twiddles W256^(r m) are applied where the stride-1 pass stores its
// outputs (row r = b mod 16, m = k), which by their symmetry are the same
// table entries as the forward pass's (row k, m = b mod 16), so every phase is
// load, butterfly, factors, store. The warps of an SM then run from the
// instruction cache nearest to them: fetching instructions was the top stall
// (2048^2: 53 -> 49 us).
template <bool ADJ>
__device__ __forceinline__ void col_middle16(c2* A, const FftPlan& fp, const c2* K, int k1n, const c2* T1, const Team& w, int b, bool on) {
    const int m = b & 15;
    c2* Z16 = A + padn((b >> 4) * 256, fp.lst[0]) + m;
    c2* Z1 = A + padn(16 * b, fp.lst[0]);
#pragma unroll 1
    for (int ph = 0; ph < 3; ++ph) {
        if (on) {
            c2 x[16];
            if (ph == 1) {
#pragma unroll
                for (int r = 0; r < 16; ++r) x[r] = ld2(Z1 + r);
            } else {
#pragma unroll
                for (int r = 0; r < 16; ++r) x[r] = ld2(Z16 + 17 * r);
            }
#pragma unroll 1
            for (int h = ph == 1 ? 0 : 1; h < 2; ++h) {
                dft_small<16>(x, -1);
                if (h == 0) kernel_product16<ADJ>(x, fp, K, k1n, b);
            }
            if (ph < 2) twiddle2<16>(x, T1 + m, 16);
            if (ph == 1) {
#pragma unroll
                for (int r = 0; r < 16; ++r) st2(Z1 + r, x[r]);
            } else {
#pragma unroll
                for (int r = 0; r < 16; ++r) st2(Z16 + 17 * r, x[r]);
            }
        }
        w.sync();
    }
}

// The last pass of a plan of any length.
template <int R, bool ADJ>
__device__ __forceinline__ void col_kernel_any(c2* A, const FftPlan& fp, const c2* K, int k1n, int nc, int t, int nt) {
    const int n = fp.n, s = fp.nst, nb = n / R, pitch = seq_pitch(n, fp.rad[0]);
    for (int i = t; i < nc * nb; i += nt) {
        const int cp = i / nb, b = i - cp * nb;
        int fb = 0, w = 1, rem = b;
        for (int p = 0; p + 1 < s; ++p) {
            const int d = fp.st[p] / R;
            const int k = rem / d;
            rem -= k * d;
            fb += k * w;
            w *= fp.rad[p];
        }
        c2* Z = A + cp * pitch;
        c2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = ld2(Z + pad16(b * R + r));
        dft_small<R>(x, -1);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int f = fb + nb * k;
            const int kk = f <= n - f ? f : n - f;
            x[k] = kernel_product<ADJ>(x[k], ld2(K + cp * k1n + min(kk, k1n - 1)));
        }
        dft_small<R>(x, -1);
#pragma unroll
        for (int r = 0; r < R; ++r) st2(Z + pad16(b * R + r), x[r]);
    }
}

#define HR_MID248_CASES(CALL)     \
    case 8: CALL(8); break;       \
    case 4: CALL(4); break;       \
    default: CALL(2); break;

template <class Src, bool ADJ>
__global__ void __launch_bounds__(kColThreadsReg, 1) k_colconv(const __grid_constant__ Src B) {
    int bx;
    const PieceDev& P = piece_of(B, bx);
    const int n = P.Ptheta, Nth = P.Ntheta, k1n = P.k1max + 2, sp = P.sp;   // K ends with a zero
    if (colconv_smem(P) > dyn_smem_bytes()) return chain_wait<5>();
    const int kb0 = bx * P.C, nc = min(P.C, P.nkb - kb0);
    const int pitch = seq_pitch(n, P.fftT.rad[0]);
    const FftPlan& fp = P.fftT;
    const int s = fp.nst, ntw = col_twiddles(fp), t = threadIdx.x, nt = blockDim.x;
    c2* A = reinterpret_cast<c2*>(smem_f);
    c2* K = A + P.C * pitch;
    c2* Ts = K + P.C * k1n;
    c2* col = reinterpret_cast<c2*>(P.spec) + (size_t)kb0 * sp;
    const c2* Tg = reinterpret_cast<const c2*>(P.twT);
    {
        const c2* Kg = reinterpret_cast<const c2*>(P.K) + (size_t)kb0 * k1n;
        for (int i = t; i < nc * k1n; i += nt) cp_async16(K + i, Kg + i);
        const c2* Tm = Tg + (ntw ? fp.tw[1] : 0);
        for (int i = t; i < ntw; i += nt) cp_async16(Ts + i, Tm + i);
    }
    chain_next<5>();
    chain_wait<5>();
    if (!fft_by16(n)) {
        for (int i = t; i < nc * Nth; i += nt) {
            const int cp = i / Nth, m = i - cp * Nth;
            const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(col + (size_t)cp * sp + m));
            st2(A + cp * pitch + pad16(m), c2{v.x, v.y});
        }
        for (int i = t; i < nc * (n - Nth); i += nt) {
            const int cp = i / (n - Nth), m = Nth + i - cp * (n - Nth);
            st2(A + cp * pitch + pad16(m), c2{0ull, 0ull});
        }
        cp_async_wait_all();
        __syncthreads();
        for (int p = 0; p + 1 < s; ++p) {
#define HR_CF(RR) pass_any<RR, false>(A, pitch, nc, n / RR, fp.st[p], Tg + fp.tw[p], t, nt)
            switch (fp.rad[p]) { HR_RADIX_CASES(HR_CF) }
            __syncthreads();
        }
#define HR_K(RR) col_kernel_any<RR, ADJ>(A, fp, K, k1n, nc, t, nt)
        switch (fp.rad[s - 1]) { HR_RADIX_CASES(HR_K) }
        __syncthreads();
        for (int p = s - 2; p >= 0; --p) {
#define HR_CI(RR) pass_any<RR, true>(A, pitch, nc, n / RR, fp.st[p], Tg + fp.tw[p], t, nt)
            switch (fp.rad[p]) { HR_RADIX_CASES(HR_CI) }
            __syncthreads();
        }
        for (int i = t; i < nc * Nth; i += nt) {
            const int cp = i / Nth, m = i - cp * Nth;
            st2(col + (size_t)cp * sp + m, ld2(A + cp * pitch + pad16(m)));
        }
        return;
    }
    const int ls0 = fp.lst[0];
#define HR_FIRST(RR) col_first_any<RR>(A, col, sp, Nth, nc, ls0, Tg, t, nt)
    switch (fp.rad[0]) { HR_RADIX_CASES(HR_FIRST) }
    cp_async_wait_all();
    __syncthreads();
    const int nall = nc * n;                       // elements of the CTA's blocks, back to back
    if (s == 4) {
        pass16<4, false>(A, t, nall >> 2, nt, fp.lst[1], ls0, Ts);
        __syncthreads();
    }
    const int r1 = s >= 3 ? fp.rad[s - 2] : 0;
    const c2* T1 = Ts + (s >= 3 ? fp.tw[s - 2] - fp.tw[1] : 0);
    const Team w(nall, t, nt);
    for (int e0 = w.first; e0 < nall; e0 += w.next) {
        const int b = (e0 >> 4) + w.me;
        const bool on = 16 * b < nall;
        if (r1 == 16) {
            col_middle16<ADJ>(A, fp, K, k1n, T1, w, b, on);
            continue;
        }
#define HR_MF(RR) team_mid<RR, false>(A, w, e0, nall, ls0, T1)
#define HR_MI(RR) team_mid<RR, true>(A, w, e0, nall, ls0, T1)
        if (s >= 3) {
            switch (r1) { HR_MID248_CASES(HR_MF) }
            w.sync();
        }
        if (on) col_kernel<ADJ>(A, fp, K, k1n, b);
        if (s >= 3) {
            w.sync();
            switch (r1) { HR_MID248_CASES(HR_MI) }
        }
    }
    __syncthreads();
    if (s == 4) {
        pass16<4, true>(A, t, nall >> 2, nt, fp.lst[1], ls0, Ts);
        __syncthreads();
    }
#define HR_LAST(RR) col_last_any<RR>(A, col, sp, Nth, nc, ls0, Tg, t, nt)
    switch (fp.rad[0]) { HR_RADIX_CASES(HR_LAST) }
}

// --------------------------------------------------------------------------
// Launchers
// --------------------------------------------------------------------------
size_t colconv_smem_bytes(const PieceDev& P) { return colconv_smem(P); }

void set_col_groups(PieceDev* P, int n) {
    long blocks = 0;
    for (int k = 0; k < n; ++k) blocks += P[k].nkb;
    const int most = (int)std::max(1L, blocks / 304);
    for (int k = 0; k < n; ++k) {
        P[k].C = std::max(1, std::min(most, kColThreads / std::max(1, P[k].Ptheta / 16)));
        P[k].nkg = (P[k].nkb + P[k].C - 1) / P[k].C;
    }
}

int col_threads(const PieceDev* P, int n) {
    int t = kColThreads;
    long blocks = 0, most = 0;
    for (int k = 0; k < n; ++k) {
        blocks += P[k].nkg;
        most = std::max<long>(most, P[k].Ptheta / 16 * P[k].C);
        t = std::max(t, std::min(kColThreadsMax, (P[k].Ptheta / 16 * P[k].C + 31) & ~31));
    }
    // short columns that do not fit the chip at once: fewer threads, if that
    // fits them (the launch's time is then one CTA's latency, not two)
    for (int s = kColThreads; s >= 64 && t == kColThreads; s -= 32)
        if (s >= most && blocks > kSMs * (512 / kColThreads) && blocks <= (long)kSMs * (512 / s)) t = s;
    return t;
}

template <class Src, bool ADJ>
static int launch_colconv_as(const Src& B, int nb, int tpb, size_t sm, void* stream) {
    if (int e = set_smem((const void*)k_colconv<Src, ADJ>, sm)) return e;
    return nb > 0 ? launch_chain(5, k_colconv<Src, ADJ>, nb, tpb, sm, stream, B) : 0;
}

int launch_colconv(const PieceDev* P, int n, int adjoint, void* stream) {
    size_t sm = 0;
    for (int k = 0; k < n; ++k) sm = std::max(sm, colconv_smem(P[k]));
    PieceBatch B;
    const int nb = make_batch(P, n, B, [](const PieceDev& q) { return q.nkg; }), tpb = col_threads(P, n);
    return adjoint ? launch_colconv_as<PieceBatch, true>(B, nb, tpb, sm, stream)
                   : launch_colconv_as<PieceBatch, false>(B, nb, tpb, sm, stream);
}

int launch_colconv_dev(const DevBatch& S, int nblocks, int tpb, size_t smem, int adjoint, void* stream) {
    return adjoint ? launch_colconv_as<DevBatch, true>(S, nblocks, tpb, smem, stream)
                   : launch_colconv_as<DevBatch, false>(S, nblocks, tpb, smem, stream);
}

}  // namespace hr
