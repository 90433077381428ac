// sm_103a kernels of the log-polar hyperbolic Radon transform and of the
// direct-summation comparator.
//
// Forward, per sub-problem (Sections 2-4):
//   k_grid_tiles       gridding of the gather samples onto the log-polar
//                      lattice with cubic B-splines (Eq. (14)-(15)), one tile
//                      of lattice cells per CTA in shared memory;
//   k_rows_r2c         real FFT of the lattice rows (first half of Eq. (7)/(16));
//   k_colconv          FFT along theta, product with the kernel spectrum
//                      chi_L zeta_hat / B3_hat^2 (Eq. (16)-(17)), inverse FFT;
//   k_rows_c2r         inverse real FFT of the rows -> B-spline coefficients;
//   k_interp_columns   cubic B-spline interpolation at (phi, eta) = P2 S(tau^2,
//                      q^2) (Eq. (17)), summed over the time pieces.
// Adjoint (Eq. (16), Section 3): the same kernels with the roles exchanged:
//   k_col_profiles_cols -> k_band_rows -> k_colconv (conjugate kernel) -> k_rows_c2r ->
//   k_gather_samples.
//
// Lattice positions do not depend on the data: the plan computes them once in
// FP64 (k_sample_table, k_radon_table) and stores first tap and fractional
// part, so the transforms themselves are FP32 loads, B-spline weights and
// sums. Shared-memory accumulation is fixed point (integer atomics, order
// independent); a lattice tile cut into several gridding work units is
// summed from their partial tiles in a fixed order by the last unit to
// finish. No kernel uses floating-point atomics: the forward and the adjoint
// are bitwise reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "device.cuh"
#include "fft2.cuh"

namespace hr {

// Data another kernel of the stream writes (gathers, images, lattices,
// profiles) are read with ordinary global loads (__ldca): with dependent
// launches the read-only path (__ldg, __restrict__) is for the plan's tables
// alone.
__device__ __forceinline__ float load_in(const float* p) { return __ldca(p); }
__device__ __forceinline__ float load_in(const __nv_bfloat16* p) {
    return __int_as_float((unsigned)__ldca(reinterpret_cast<const unsigned short*>(p)) << 16);
}

// Shared gridding tile: the kTileRows x kTileCols cells plus a halo of
// NT - 1 cells on every side (NT taps per axis: 4 cubic, 6 quintic), so that
// every tap of a sample whose footprint meets the tile lands in it without a
// bounds check (the halo is dropped at the end: the neighbouring tiles'
// units add those cells). The odd pitch puts the rows on different banks.
template <int NT>
struct GridTile {
    static constexpr int halo = NT - 1;
    static constexpr int pitch = kTileCols + 2 * halo + 1;
    static constexpr int rows = kTileRows + 2 * halo;
};

// Fixed-point accumulation in shared memory. Integer adds to shared memory
// are single fire-and-forget instructions, float adds are compare-and-swap
// loops (measured 3.7x apart on conflict-free addresses), and integer sums do
// not depend on the order in which warps arrive. A block accumulating into a
// region whose cells provably stay below vmax * C in magnitude (vmax the
// largest |input| it adds, C a plan-time bound on the total weight any cell
// collects, C < 2^(ec+1)) scales its inputs by 2^sh with
// sh = 28 - ec - ilogb(vmax): every cell stays below 2^30, and every
// contribution is rounded to 2^-31 of at most four times the bound. The
// power of two is applied as two factors so that it spans the whole float
// range. The plan stores 28 - ec.
__device__ __forceinline__ float pow2i(int k) { return __int_as_float((127 + k) << 23); }   // |k| <= 126

struct Pow2Scale {
    float up1, up2, down1, down2;
    __device__ __forceinline__ Pow2Scale(int sh) {
        const int h1 = sh / 2, h2 = sh - h1;
        up1 = pow2i(h1);
        up2 = pow2i(h2);
        down1 = pow2i(-h1);
        down2 = pow2i(-h2);
    }
    __device__ __forceinline__ float up(float v) const { return v * up1 * up2; }
    __device__ __forceinline__ float down(int t) const { return (float)t * down1 * down2; }
};

__device__ __forceinline__ void red_fixed(int* p, float v) { atomicAdd(p, __float2int_rn(v)); }

// Maximum of a non-negative float over the block (all threads get it); NaN
// wins, so a non-finite input shows as a non-finite maximum.
__device__ __forceinline__ float block_max_abs(float v, float* red) {
    v = fabsf(v);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const float o = __shfl_xor_sync(0xffffffffu, v, d);
        v = (o > v || o != o) ? o : v;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float m = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        const float o = red[w];
        m = (o > m || o != o) ? o : m;
    }
    return m;
}

// Forward gridding (Eq. (15)) of the gather f[Nx][Nt] onto the lattice
// P.lat. Every cell is written, a tile without samples has an empty unit (one
// launch less than clearing first: 2 of 40 us at 256 x 64); a batch's lattices
// are cleared before, which is the faster way where the units have no time to
// spare (128 gathers: 2074 against 2109 us).
// The plan lists, per tile of kTileRows x kTileCols
// cells, chunks of at most 8 consecutive samples of one trace whose NT x NT
// footprint meets the tile, and cuts every tile's list into work units of at
// most kUnitChunks chunks (sample density varies by two orders of magnitude
// over the lattice, so units, not tiles, balance the CTAs), each with the
// largest total B-spline weight one of its cells can collect. A CTA takes one
// unit, each thread one chunk: neighbouring threads are 8 samples apart, so
// their footprints rarely meet, and a thread sums its samples in registers
// in an NT x NT register window over the cells of its current footprint. When the
// first tap (m0, n0) moves by one cell along either axis (consecutive samples
// of a trace mostly do), only the row or column that leaves the window goes
// to the fixed-point shared tile and the window slides; a longer jump flushes
// the whole window. The tile's touched cells are then added to P.lat. A
// non-finite sample makes the unit's tile NaN (the FFTs that follow would
// spread it over the whole piece in any case).
// The window acc[NT a + c] holds cells (wm + a, wn + c); t points at
// (wm, wn) in the shared tile.
template <int NT>
__device__ __forceinline__ void flush_window(int* t, const float (&acc)[NT * NT]) {
#pragma unroll
    for (int a = 0; a < NT; ++a)
#pragma unroll
        for (int c = 0; c < NT; ++c) red_fixed(t + a * GridTile<NT>::pitch + c, acc[NT * a + c]);
}
// window one row down (row wm leaves) / up (row wm + NT - 1 leaves)
template <int NT>
__device__ __forceinline__ void slide_rows_down(int* t, float (&acc)[NT * NT]) {
#pragma unroll
    for (int c = 0; c < NT; ++c) {
        red_fixed(t + c, acc[c]);
#pragma unroll
        for (int a = 0; a + 1 < NT; ++a) acc[NT * a + c] = acc[NT * (a + 1) + c];
        acc[NT * (NT - 1) + c] = 0.f;
    }
}
template <int NT>
__device__ __forceinline__ void slide_rows_up(int* t, float (&acc)[NT * NT]) {
#pragma unroll
    for (int c = 0; c < NT; ++c) {
        red_fixed(t + (NT - 1) * GridTile<NT>::pitch + c, acc[NT * (NT - 1) + c]);
#pragma unroll
        for (int a = NT - 1; a > 0; --a) acc[NT * a + c] = acc[NT * (a - 1) + c];
        acc[c] = 0.f;
    }
}
// window one column right (column wn leaves) / left (column wn + NT - 1 leaves)
template <int NT>
__device__ __forceinline__ void slide_cols_right(int* t, float (&acc)[NT * NT]) {
#pragma unroll
    for (int a = 0; a < NT; ++a) {
        red_fixed(t + a * GridTile<NT>::pitch, acc[NT * a]);
#pragma unroll
        for (int c = 0; c + 1 < NT; ++c) acc[NT * a + c] = acc[NT * a + c + 1];
        acc[NT * a + NT - 1] = 0.f;
    }
}
template <int NT>
__device__ __forceinline__ void slide_cols_left(int* t, float (&acc)[NT * NT]) {
#pragma unroll
    for (int a = 0; a < NT; ++a) {
        red_fixed(t + a * GridTile<NT>::pitch + NT - 1, acc[NT * a + NT - 1]);
#pragma unroll
        for (int c = NT - 1; c > 0; --c) acc[NT * a + c] = acc[NT * a + c - 1];
        acc[NT * a] = 0.f;
    }
}

// Split tiles: the unit's partial tile (value(i) of cell i, row-major over
// the kTileRows x kTileCols cells) goes to its slot; the unit that finds it
// is the tile's last to arrive (the others' slots are then complete and
// visible) sums every slot of the tile in slot order into the lattice. The
// result does not depend on which unit runs first; the counter is back at zero
// once every unit has arrived (last_arrival).
// Ordering: the block's slot stores, a barrier, then one thread's fence and
// count (release, cumulative over the block through the barrier); on the
// reading side that thread's fence after the count, a barrier, and L2 loads.
template <class F>
__device__ __forceinline__ void grid_merge_split(const PieceDev& P, int4 us, int m_lo, int n_lo, int nr, int nc,
                                                 F&& value) {
    __shared__ int s_last;
    constexpr int kCells = kTileRows * kTileCols;
    float* slot0 = P.slots + (size_t)us.x * kCells;
    for (int i = threadIdx.x; i < kCells; i += blockDim.x) slot0[(size_t)us.z * kCells + i] = value(i);
    __syncthreads();
    unsigned* counter = reinterpret_cast<unsigned*>(P.lat + (size_t)P.Ntheta * P.lp) + us.w;
    if (threadIdx.x == 0) {
        __threadfence();
        const bool last = last_arrival(us.y, [&](unsigned most) { return atomicInc(counter, most); });
        if (last) __threadfence();
        s_last = last;
    }
    __syncthreads();
    if (!s_last) return;
    // each thread sums two groups of four cells over the slots in slot order,
    // eight slots' loads in flight (the densest tile of the 2048^2 gather has
    // 40 slots, and its merge ends the launch)
    static_assert(kCells == 8 * kUnitChunks, "cells per thread");
    float4 acc[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    const float4* src = reinterpret_cast<const float4*>(slot0) + threadIdx.x;
    for (int u0 = 0; u0 < us.y; u0 += 8) {
        float4 v[8][2];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                v[u][j] = u0 + u < us.y ? __ldcg(src + (size_t)(u0 + u) * (kCells / 4) + j * kUnitChunks)
                                        : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                acc[j].x += v[u][j].x;
                acc[j].y += v[u][j].y;
                acc[j].z += v[u][j].z;
                acc[j].w += v[u][j].w;
            }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = 4 * (threadIdx.x + j * kUnitChunks);
        const int m = i / kTileCols, n = i - m * kTileCols;
        // within the row pitch, a multiple of four like n_lo
        if (m < nr && n < nc) *reinterpret_cast<float4*>(P.lat + (size_t)(m_lo + m) * P.lp + n_lo + n) = acc[j];
    }
}

// Cubic tap weights of both axes at once, packed (w1 and w2 as 2/3 - x^2 +
// x^3 / 2 of x = f and 1 - f): half the instructions of two evaluations.
__constant__ float2 kSplinePairs[5] = {{0.5f, 0.5f}, {-1.f, -1.f}, {1.0f / 6.0f, 1.0f / 6.0f}, {1.f, 1.f}, {2.f / 3.f, 2.f / 3.f}};
__device__ __forceinline__ void both_weights(float ft, float fr, float (&wt)[4], float (&wr)[4]) {
    const f2* k = reinterpret_cast<const f2*>(kSplinePairs);
    const f2 f = pk(ft, fr), g = sub2(k[3], f), ff = mul2(f, f), gg = mul2(g, g);
    const float2 w0 = upk(mul2(gg, mul2(g, k[2]))), w3 = upk(mul2(ff, mul2(f, k[2])));
    const float2 w1 = upk(fma2(ff, fma2(f, k[0], k[1]), k[4])), w2 = upk(fma2(gg, fma2(g, k[0], k[1]), k[4]));
    wt[0] = w0.x, wt[1] = w1.x, wt[2] = w2.x, wt[3] = w3.x;
    wr[0] = w0.y, wr[1] = w1.y, wr[2] = w2.y, wr[3] = w3.y;
}

// Position entries through shared memory: a thread reads its chunk's entries
// 128 bytes from its neighbour's, 32 lines a request. A batch's warps copy them
// with eight neighbouring lanes per chunk instead (four lines a request,
// cp.async, exchanged so that both sides touch different banks); without the
// entries in registers five CTAs share an SM. 128 gathers, bfloat16, forward:
// 2076 -> 1984 us. A single gather's launch gains 1 % at 2048^2 and loses 3 %
// at 1501 x 233 and 1024 x 256, where one CTA's latency counts, and the quintic
// kernel's accumulators leave two CTAs either way: these keep the registers.
template <class Src, int NT>
constexpr bool kGridStaged = NT == 4 && std::is_same<Src, DevBatch>::value;

template <class Src, class T, int NT>
__global__ void __launch_bounds__(kUnitChunks, NT == 6 ? 2 : kGridStaged<Src, NT> ? 5 : 4) k_grid_tiles(const __grid_constant__ Src B,
                                                                             const T* f) {
    using Tile = GridTile<NT>;
    constexpr bool kStaged = kGridStaged<Src, NT>;
    __shared__ int4 s_ent[kStaged ? 8 * kUnitChunks : 1];
    __shared__ int tile[Tile::rows * Tile::pitch];
    __shared__ float red[kUnitChunks / 32];
    int bx;
    const PieceDev& P = piece_of(B, bx);
    const int4 u = __ldg(P.units + bx);           // (tile, first chunk, end chunk, 28 - ec)
    const int ti = u.x / P.ntc, tj = u.x - ti * P.ntc;
    const int m_lo = ti * kTileRows, n_lo = tj * kTileCols;
    const int nr = min(kTileRows, P.Ntheta - m_lo), nc = min(kTileCols, P.Nrho - n_lo);
    chain_next<8>();
    constexpr bool kCleared = std::is_same<Src, DevBatch>::value;   // a batch's lattices are cleared before
    if (kCleared) chain_wait<8>();                // (after the clearing, nothing to start early for)
    if (u.y == u.z) {                             // a tile without samples
        if (kCleared) return;
        chain_wait<8>();
        for (int i = threadIdx.x; i < kTileRows * kTileCols; i += blockDim.x) {
            const int m = i / kTileCols, n = i - m * kTileCols;
            if (m < nr && n < nc) P.lat[(size_t)(m_lo + m) * P.lp + n_lo + n] = 0.f;
        }
        return;
    }
    for (int i = threadIdx.x; i < Tile::rows * Tile::pitch; i += blockDim.x) tile[i] = 0;
    // one chunk per thread: issue every load of the chunk before the first is used
    const int lane = threadIdx.x & 31, c = u.y + threadIdx.x;
    int4* my = s_ent + (kStaged ? 8 * threadIdx.x : 0);
    int4 ent[kStaged ? 1 : 8];
    int4 ch = make_int4(0, 0, 0, 0);                // (trace, first sample, count)
    if (c < u.z) ch = __ldg(P.chunks + c);
    const long long first = (long long)ch.x * P.nj - P.jt_lo + ch.y;
    float v[8];
    float vmax = 0.f;
    const T* fk = f + P.f_off + (size_t)ch.x * P.Nt + ch.y;
    if constexpr (kStaged) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = 4 * j + (lane >> 3), s = lane & 7;
            const long long at = __shfl_sync(0xffffffffu, first, k) + s;
            const bool on = s < __shfl_sync(0xffffffffu, ch.z, k);
            cp_async16_or_zero(s_ent + 8 * ((threadIdx.x & ~31) + k) + (s ^ (k & 7)), P.stab + (on ? at : 0), on);
        }
    } else {
        const int4* st = reinterpret_cast<const int4*>(P.stab) + first;
#pragma unroll
        for (int s = 0; s < 8; ++s) ent[s] = s < ch.z ? __ldg(st + s) : make_int4(0, 0, 0, 0);
    }
    if (!kCleared) chain_wait<8>();
#pragma unroll
    for (int s = 0; s < 8; ++s) v[s] = s < ch.z ? load_in(fk + s) : 0.f;
    if (kStaged) {
        cp_async_wait_all();
        __syncwarp();
    }
    auto entry = [&](int s) -> int4 {
        if constexpr (kStaged) return my[s ^ (lane & 7)];
        else return ent[s];
    };
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const float w = __int_as_float(entry(s).w);
        v[s] = w != 0.f ? v[s] * w : 0.f;   // muted samples add nothing, whatever f holds
        const float a = fabsf(v[s]);
        vmax = (a > vmax || a != a) ? a : vmax;
    }
    vmax = block_max_abs(vmax, red);   // also orders the tile's zeroing before the adds
    const int4 us = __ldg(P.uslot + bx);  // (first slot, units of the tile, index, counter)
    if (!(vmax > 0.f && vmax <= 3.402823466e38f)) {   // all zero (nothing to add) or not finite (NaN tile)
        const float fill = vmax == 0.f ? 0.f : __int_as_float(0x7fc00000);
        if (us.y > 1) {
            grid_merge_split(P, us, m_lo, n_lo, nr, nc, [&](int) { return fill; });
        } else if (fill != 0.f || !kCleared) {
            for (int i = threadIdx.x; i < kTileRows * kTileCols; i += blockDim.x) {
                const int m = i / kTileCols, n = i - m * kTileCols;
                if (m < nr && n < nc) P.lat[(size_t)(m_lo + m) * P.lp + n_lo + n] = fill;
            }
        }
        return;
    }
    const Pow2Scale sc(u.w - ilogbf(vmax));
#pragma unroll
    for (int s = 0; s < 8; ++s) v[s] = sc.up(v[s]);
    float acc[NT * NT];
#pragma unroll
    for (int q = 0; q < NT * NT; ++q) acc[q] = 0.f;
    int* win = nullptr;                                  // shared-tile address of the window's (wm, wn)
    int wm = 0, wn = 0;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        if (v[s] == 0.f) continue;
        const int4 e = entry(s);
        const int m0 = e.x >> 16, n0 = e.x & 0xffff;
        const int dm = m0 - wm, dn = n0 - wn;
        if (win == nullptr || dm < -1 || dm > 1 || dn < -1 || dn > 1) {
            if (win != nullptr) {
                flush_window<NT>(win, acc);
#pragma unroll
                for (int q = 0; q < NT * NT; ++q) acc[q] = 0.f;
            }
        } else {
            if (dm == 1) slide_rows_down<NT>(win, acc);
            else if (dm == -1) slide_rows_up<NT>(win, acc);
            win += dm * Tile::pitch;
            if (dn == 1) slide_cols_right<NT>(win, acc);
            else if (dn == -1) slide_cols_left<NT>(win, acc);
        }
        wm = m0;
        wn = n0;
        win = tile + (m0 - m_lo + Tile::halo) * Tile::pitch + n0 - n_lo + Tile::halo;
        float wt[NT], wr[NT];
        if constexpr (NT == 4) {
            both_weights(__int_as_float(e.y), __int_as_float(e.z), wt, wr);
        } else {
            bspline_weights<NT>(__int_as_float(e.y), wt);
            bspline_weights<NT>(__int_as_float(e.z), wr);
        }
#pragma unroll
        for (int a = 0; a < NT; ++a) {
            const float va = v[s] * wt[a];
#pragma unroll
            for (int q = 0; q < NT; ++q) acc[NT * a + q] = fmaf(va, wr[q], acc[NT * a + q]);
        }
    }
    if (win != nullptr) flush_window<NT>(win, acc);
    __syncthreads();
    if (us.y > 1) {
        grid_merge_split(P, us, m_lo, n_lo, nr, nc,
                         [&](int i) {
                             return sc.down(tile[(i / kTileCols + Tile::halo) * Tile::pitch + i % kTileCols + Tile::halo]);
                         });
        return;
    }
    for (int i = threadIdx.x; i < kTileRows * kTileCols; i += blockDim.x) {   // the tile's only unit
        const int m = i / kTileCols, n = i - m * kTileCols;
        const int t = tile[(m + Tile::halo) * Tile::pitch + n + Tile::halo];
        if ((t != 0 || !kCleared) && m < nr && n < nc) P.lat[(size_t)(m_lo + m) * P.lp + n_lo + n] = sc.down(t);
    }
}

// Adjoint of the output interpolation (transpose of Eq. (17)), separated
// along the two axes. Every output of a slowness column has the same theta
// taps (the column's angle), so the transpose is a 1-D scatter along rho per
// column followed by an NT-tap spread of the column profiles over theta
// (B the cubic or quintic B-spline, NT = 4 or 6 taps):
//   h_l[n]   = s_l sum_i g[l][i] B(rho_il - rho_n)           (k_col_profiles_cols)
//   G'[m][n] = sum_l B(theta_l - theta_m) h_l[n]             (k_band_rows)
// The profiles are summed in fixed point (order-independent), the spread is a
// plain per-thread sum over the band's columns in a fixed order: the adjoint
// interpolation has no floating-point atomics and is deterministic.

// The profiles P.prof[lc][0..Nrho) (pitch hpitch) of every time piece of
// one output column, from the column's outputs g[l][*] scaled by each
// piece's output scale: one CTA per column (cmap[b] = (first piece, number
// of pieces, column l), or, when np_all > 0, column b of pieces[0..np_all)
// with ntau_all outputs), so that the column's outputs are read once for the
// scale and once for all its pieces ([np][nrho_max] in shared memory). Fixed
// point with the bound max|g| of the column times each piece's plan-time
// weight bound for the column; a non-finite g makes the profiles NaN.
template <int NT>
__global__ void __launch_bounds__(256) k_col_profiles_cols(const PieceDev* __restrict__ pieces,
                                                           const int4* __restrict__ cmap, int nrho_max, int ntau_all,
                                                           int np_all, const float* g) {
    chain_next<5>();
    chain_wait<5>();
    const int4 c = np_all > 0 ? make_int4(0, np_all, (int)blockIdx.x, 0) : __ldg(cmap + blockIdx.x);
    const int l = c.z, np = c.y;
    const int Ntau = np_all > 0 ? ntau_all : pieces[c.x].Ntau;
    if (np > kMaxColPieces || (size_t)np * nrho_max * sizeof(int) > dyn_smem_bytes()) return;
    int* prof = reinterpret_cast<int*>(smem_f);
    __shared__ float red[8];
    __shared__ const int2* s_rt[kMaxColPieces];
    __shared__ float* s_hl[kMaxColPieces];
    __shared__ float s_sc[kMaxColPieces];
    __shared__ int s_sh[kMaxColPieces];
    __shared__ int2 s_rg[kMaxColPieces];
    __shared__ int s_nr[kMaxColPieces], s_hp[kMaxColPieces];
    if ((int)threadIdx.x < np) {
        const PieceDev& P = pieces[c.x + threadIdx.x];
        const int lc = l - P.l_lo;
        s_rt[threadIdx.x] = reinterpret_cast<const int2*>(P.rtab + (size_t)lc * Ntau);
        s_hl[threadIdx.x] = P.prof + (size_t)lc * P.hpitch;
        s_sc[threadIdx.x] = __ldg(P.colscale + lc);
        s_sh[threadIdx.x] = __ldg(P.colsh + lc);
        s_rg[threadIdx.x] = __ldg(P.rrange + lc);
        s_nr[threadIdx.x] = P.Nrho;
        s_hp[threadIdx.x] = P.hpitch;
    }
    for (int i = threadIdx.x; i < np * nrho_max; i += blockDim.x) prof[i] = 0;
    const float* gl = g + (np_all > 0 ? 0 : pieces[c.x].g_off) + (size_t)l * Ntau;
    constexpr int Q = 8;                        // outputs per thread
    const int chunk = Q * (int)blockDim.x;
    float mx = 0.f;
    for (int i0 = 0; i0 < Ntau; i0 += chunk) {
        float v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int i = i0 + q * (int)blockDim.x + threadIdx.x;
            v[q] = i < Ntau ? __ldca(gl + i) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float a = fabsf(v[q]);
            mx = (a > mx || a != a) ? a : mx;
        }
    }
    const float vmax = block_max_abs(mx, red);   // also orders the zeroing and the column data before use
    if (!(vmax > 0.f && vmax <= 3.402823466e38f)) {
        const float fill = vmax == 0.f ? 0.f : __int_as_float(0x7fc00000);
        for (int p = 0; p < np; ++p)
            for (int n = threadIdx.x; n < s_hp[p]; n += blockDim.x) s_hl[p][n] = fill;
        return;
    }
    const int ev = ilogbf(vmax);
    int lo = Ntau, hi = -1;                     // outputs valid in some piece
    for (int p = 0; p < np; ++p) {
        lo = min(lo, s_rg[p].x);
        hi = max(hi, s_rg[p].y);
    }
    // every thread takes Q consecutive outputs: their first rho tap is
    // nondecreasing, so each piece's contributions collect in an NT-cell
    // register window that slides one cell as the tap advances (the
    // departing cell goes to the shared profile) and is flushed whole on a
    // longer jump; dozens of outputs that share a cell at small intercept
    // times cost one add
    // (a thread's outputs and table entries are neighbours: 16-byte loads
    // where they are aligned, a quarter and half of the L1 requests, which
    // bound the kernel: 2048^2 47 -> 42.7 us)
    for (int i0 = lo & ~7; i0 <= hi; i0 += chunk) {
        const int ib = i0 + Q * (int)threadIdx.x;
        const bool whole = ib + Q <= Ntau;
        float v[Q];
        if (whole && !(reinterpret_cast<size_t>(gl + ib) & 15)) {
#pragma unroll
            for (int q = 0; q < Q; q += 4) {
                const float4 t = __ldca(reinterpret_cast<const float4*>(gl + ib + q));
                v[q] = t.x, v[q + 1] = t.y, v[q + 2] = t.z, v[q + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] = ib + q < Ntau ? __ldca(gl + ib + q) : 0.f;
        }
        for (int p = 0; p < np; ++p) {
            const int2 rg = s_rg[p];
            const int2* rt = s_rt[p];
            if (ib > rg.y || ib + Q <= rg.x) continue;
            int2 e[Q];
            if (whole && !(reinterpret_cast<size_t>(rt + ib) & 15)) {
#pragma unroll
                for (int q = 0; q < Q; q += 2) {         // entries outside the range hold -1
                    const int4 t = __ldg(reinterpret_cast<const int4*>(rt + ib + q));
                    e[q] = make_int2(t.x, t.y);
                    e[q + 1] = make_int2(t.z, t.w);
                }
            } else {
#pragma unroll
                for (int q = 0; q < Q; ++q) e[q] = ib + q < Ntau ? __ldg(rt + ib + q) : make_int2(-1, 0);
            }
            const Pow2Scale scl(s_sh[p] - ev);
            const float sc = s_sc[p];
            int* pr = prof + p * nrho_max;
            float w[NT];
#pragma unroll
            for (int k = 0; k < NT; ++k) w[k] = 0.f;
            int wn = -1;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int n0 = e[q].x;
                if (n0 < 0) continue;
                if (wn < 0) {
                    wn = n0;
                } else if (n0 != wn) {
                    if (n0 == wn + 1) {
                        red_fixed(pr + wn, w[0]);
#pragma unroll
                        for (int k = 0; k + 1 < NT; ++k) w[k] = w[k + 1];
                        w[NT - 1] = 0.f;
                    } else {
#pragma unroll
                        for (int k = 0; k < NT; ++k) {
                            red_fixed(pr + wn + k, w[k]);
                            w[k] = 0.f;
                        }
                    }
                    wn = n0;
                }
                float wr[NT];
                bspline_weights<NT>(__int_as_float(e[q].y), wr);
                const float x = scl.up(v[q] * sc);
#pragma unroll
                for (int k = 0; k < NT; ++k) w[k] = fmaf(x, wr[k], w[k]);
            }
            if (wn >= 0) {
#pragma unroll
                for (int k = 0; k < NT; ++k) red_fixed(pr + wn + k, w[k]);
            }
        }
    }
    __syncthreads();
    for (int p = 0; p < np; ++p) {
        const Pow2Scale scl(s_sh[p] - ev);
        const int* pr = prof + p * nrho_max;
        const int nr = s_nr[p];
        float* hl = s_hl[p];
        for (int n = threadIdx.x; n < s_hp[p]; n += blockDim.x) hl[n] = n < nr ? scl.down(pr[n]) : 0.f;
    }
}

// --------------------------------------------------------------------------
// Gathers.
// --------------------------------------------------------------------------

// NT x NT taps of the lattice at first tap (m0, n0).
template <int NT>
__device__ __forceinline__ float taps_nt(const float* lat, int Nr, int m0, int n0,
                                         const float (&wt)[NT], const float (&wr)[NT]) {
    float s = 0.f;
#pragma unroll
    for (int a = 0; a < NT; ++a) {
        const float* row = lat + (size_t)(m0 + a) * Nr + n0;
        float r = __ldca(row) * wr[0];
#pragma unroll
        for (int c = 1; c < NT; ++c) r += __ldca(row + c) * wr[c];
        s += wt[a] * r;
    }
    return s;
}

// Forward output interpolation (Eq. (17)): one CTA per output column, summed
// over the time pieces of its slowness piece; cmap[b] = (first piece, number
// of pieces, column l). As in the adjoint, the column's outputs share its
// theta taps, so the NT x NT taps separate: the CTA first spreads the NT
// lattice rows of the column's angle into a rho profile in shared memory,
//   r[n] = sum_a B(theta_l - theta_{m0+a}) H[m0 + a][n],
// for every time piece at once (shared memory: [np][pstride] profiles),
// then every output takes NT taps of each piece's profile and sums the
// pieces in a fixed order. Outputs outside a piece's valid range skip its
// table.
template <int NT>
__global__ void __launch_bounds__(256, NT == 4 ? 8 : 6) k_interp_columns(const PieceDev* __restrict__ pieces,
                                                        const int4* __restrict__ cmap, int pstride,
                                                        int ntau_all, int np_all, float* g) {
    // np_all > 0: one gather with one slowness piece of np_all time pieces and
    // ntau_all outputs per column, column = block (no map load before the work)
    chain_next<8>();
    chain_wait<8>();
    const int4 c = np_all > 0 ? make_int4(0, np_all, (int)blockIdx.x, 0) : __ldg(cmap + blockIdx.x);
    const int l = c.z, np = c.y;
    const int Ntau = np_all > 0 ? ntau_all : pieces[c.x].Ntau;
    if (np > kMaxColPieces || (size_t)np * pstride * sizeof(float) > dyn_smem_bytes()) return;
    // per-piece column data, loaded for all pieces at once (what these arrays
    // take is not left for the profiles, whose length bounds what a plan may
    // hold: 448 bytes with four taps, 512 with six)
    __shared__ float4 s_w4[kMaxColPieces];
    __shared__ float2 s_w2[NT > 4 ? kMaxColPieces : 1];
    __shared__ const float* s_r0[kMaxColPieces];
    __shared__ const int2* s_rt[kMaxColPieces];
    __shared__ float s_sc[kMaxColPieces];
    __shared__ int2 s_rg[kMaxColPieces];
    __shared__ int s_nr[kMaxColPieces];
    if ((int)threadIdx.x < np) {
        const PieceDev& P = pieces[c.x + threadIdx.x];
        const int lc = l - P.l_lo;
        s_w4[threadIdx.x] = __ldg(P.colw + lc);
        if (NT > 4) s_w2[threadIdx.x] = __ldg(P.colw2 + lc);
        s_sc[threadIdx.x] = __ldg(P.colscale + lc);
        s_r0[threadIdx.x] = P.lat + (size_t)__ldg(P.colm0 + lc) * P.lp;
        s_rt[threadIdx.x] = reinterpret_cast<const int2*>(P.rtab + (size_t)lc * Ntau);
        s_rg[threadIdx.x] = __ldg(P.rrange + lc);
        s_nr[threadIdx.x] = P.Nrho;
    }
    __syncthreads();
    // theta taps (the column's NT lattice rows) of every piece: the rho
    // profiles, np * pstride floats; four cells per thread and load (the
    // lattice rows are 16-byte aligned), all pieces' loads in flight together
    for (int p = 0; p < np; ++p) {
        const int lp = lat_pitch(s_nr[p]);
        const float4 w4 = s_w4[p];
        const float2 w2 = NT > 4 ? s_w2[p] : make_float2(0.f, 0.f);
        const float* r0 = s_r0[p];
        float* prof = smem_f + p * pstride;
        for (int n = 4 * threadIdx.x; n < lp; n += 4 * blockDim.x) {
            float4 a[NT];
#pragma unroll
            for (int k = 0; k < NT; ++k) a[k] = __ldca(reinterpret_cast<const float4*>(r0 + (size_t)k * lp + n));
            const float w[6] = {w4.x, w4.y, w4.z, w4.w, w2.x, w2.y};
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                v.x = fmaf(w[k], a[k].x, v.x);
                v.y = fmaf(w[k], a[k].y, v.y);
                v.z = fmaf(w[k], a[k].z, v.z);
                v.w = fmaf(w[k], a[k].w, v.w);
            }
            if (!(pstride & 3)) {
                *reinterpret_cast<float4*>(prof + n) = v;
            } else {                                   // profiles packed to fit shared memory
                const int Nr = s_nr[p];
                prof[n] = v.x;
                if (n + 1 < Nr) prof[n + 1] = v.y;
                if (n + 2 < Nr) prof[n + 2] = v.z;
                if (n + 3 < Nr) prof[n + 3] = v.w;
            }
        }
    }
    __syncthreads();
    // rho taps: every output sums its pieces in piece order
    float* gl = g + (np_all > 0 ? 0 : pieces[c.x].g_off) + (size_t)l * Ntau;
    // each thread takes U outputs at once and loads their table entries of a
    // piece together before using any (the entries come from DRAM and each
    // output's taps wait on its entry: U chains in flight instead of one)
    constexpr int U = 4;
    for (int i0 = threadIdx.x; i0 < Ntau; i0 += U * blockDim.x) {
        float acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = 0.f;
        for (int p = 0; p < np; ++p) {
            const int2 rg = s_rg[p];
            int2 e[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = i0 + u * (int)blockDim.x;
                e[u] = (i >= rg.x && i <= rg.y) ? __ldg(s_rt[p] + i) : make_int2(-1, 0);
            }
            const float scp = s_sc[p];
            const float* rp = smem_f + p * pstride;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (e[u].x < 0) continue;
                float wr[NT];
                bspline_weights<NT>(__int_as_float(e[u].y), wr);
                const float* r = rp + e[u].x;
                float t = wr[0] * r[0];
#pragma unroll
                for (int c = 1; c < NT; ++c) t += wr[c] * r[c];
                acc[u] += scp * t;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * (int)blockDim.x;
            if (i < Ntau) gl[i] = acc[u];
        }
    }
}

// Adjoint of the gridding (transpose of Eq. (15)): every gather sample reads
// the NT x NT taps of each sub-problem that holds it. One CTA per kSampleBlock
// sample slots of one gather, a warp 16 times of two neighbouring traces
// (sample_blocks): smap[b] = (first piece, number of pieces, block within the
// gather). Bound: the L1 request rate. A tap load of a warp
// touches 3 to 4.5 lines at 2048^2 so, against 3.4 to 7 with 32 times of one
// trace (a curve through the lattice crosses rows); 8 x 4 touches as many
// there, but more where traces are sparse.
template <int NT>
__global__ void __launch_bounds__(kSampleBlock, NT == 4 ? 8 : 4) k_gather_samples(const PieceDev* __restrict__ pieces,
                                                                    const int4* __restrict__ smap,
                                                                    float* f, int np_all, int Nt_all,
                                                                    int Nx_all) {
    // np_all > 0: one gather of Nt_all x Nx_all samples in np_all pieces,
    // its blocks in order (no map load before the work)
    chain_next<8>();
    chain_wait<8>();
    const int4 m = np_all > 0 ? make_int4(0, np_all, (int)blockIdx.x, 0) : __ldg(smap + blockIdx.x);
    const int Nt = np_all > 0 ? Nt_all : pieces[m.x].Nt;
    const int Nx = np_all > 0 ? Nx_all : pieces[m.x].Nx;
    const unsigned wp = (unsigned)m.z * (kSampleBlock / 32) + (threadIdx.x >> 5), per = (unsigned)((Nt + 15) >> 4);
    const int kp = (int)(wp / per);
    const int j = (int)(wp - (unsigned)kp * per) * 16 + (threadIdx.x & 15), k = 2 * kp + (threadIdx.x >> 4 & 1);
    if (j >= Nt || k >= Nx) return;
    const long idx = (long)k * Nt + j;
    float acc = 0.f;
    for (int p = m.x; p < m.x + m.y; ++p) {
        const PieceDev& P = pieces[p];
        if (j < P.jt_lo || j > P.jt_hi) continue;
        const int4 e = __ldg(reinterpret_cast<const int4*>(P.stab + (size_t)k * P.nj + (j - P.jt_lo)));
        const float w = __int_as_float(e.w);
        if (w == 0.f) continue;
        float wt[NT], wr[NT];
        bspline_weights<NT>(__int_as_float(e.y), wt);
        bspline_weights<NT>(__int_as_float(e.z), wr);
        acc += w * taps_nt<NT>(P.lat, P.lp, e.x >> 16, e.x & 0xffff, wt, wr);
    }
    f[(np_all > 0 ? 0 : pieces[m.x].f_off) + idx] = acc;
}

// --------------------------------------------------------------------------
// Plan time, FP64: lattice positions of every gather sample and of every
// output (the maps P1 T of Eq. (10)/(14) and P2 S of Eq. (9)/(17)).
// --------------------------------------------------------------------------
__global__ void k_sample_table(TableArgs A, const double* __restrict__ cj, const double* __restrict__ wk,
                               const int* __restrict__ jfirst, SampleEnt* __restrict__ out) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)A.nj * A.Nx) return;
    const int k = (int)(idx / A.nj);
    const int jl = (int)(idx - (long)k * A.nj);
    const int j = A.jt_lo + jl;
    const double tb = j / A.n_t, xb = A.xb[k];
    const double ds = tb * tb - 0.5, dy = xb * xb - 0.5;
    const double u1 = A.a * (A.ca * ds - A.sa * dy) + A.O1;
    const double u2 = A.a * (A.sa * ds + A.ca * dy) + A.O2;
    const double r2 = u1 * u1 + u2 * u2;
    const double xth = (atan2(u2, u1) - A.theta0) / A.dtheta;
    const double xrh = (0.5 * log(r2) - A.rho0) / A.drho;
    const double fm = floor(xth), fn = floor(xrh);
    const int back = A.ntaps / 2 - 1;            // first tap: floor - (order - 1) / 2
    int m0 = (int)fm - back, n0 = (int)fn - back;
    double w = (j >= jfirst[k]) ? cj[jl] * wk[k] / sqrt(r2) : 0.0;
    if (m0 < 0 || m0 + A.ntaps - 1 >= A.Ntheta || n0 < 0 || n0 + A.ntaps - 1 >= A.Nrho) {
        w = 0.0;
        m0 = 0;
        n0 = 0;
    }
    SampleEnt e;
    e.mn = (m0 << 16) | n0;
    e.ft = (float)(xth - fm);
    e.fr = (float)(xrh - fn);
    e.w = (float)w;
    out[idx] = e;
}

__global__ void k_radon_table(TableArgs A, const double* __restrict__ qb2, RadonEnt* __restrict__ out) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)A.ncol * A.Ntau) return;
    const int lc = (int)(idx / A.Ntau);
    const int i = (int)(idx - (long)lc * A.Ntau);
    const double m = qb2[lc];
    const double psi = atan(m);
    const double theta = A.alpha - psi;
    const double tb = (A.tau0 + i * A.dtau) / A.T;
    const double e = A.a * cos(psi) * (tb * tb - 0.5 + 0.5 * m) + A.O1 * cos(theta) + A.O2 * sin(theta);
    RadonEnt r;
    r.n0 = -1;
    r.fr = 0.f;
    if (e >= A.a_r && e <= A.r_max) {
        const double xrh = (log(e) - A.rho0) / A.drho;
        const double fn = floor(xrh);
        const int n0 = (int)fn - (A.ntaps / 2 - 1);
        if (n0 >= 0 && n0 + A.ntaps - 1 < A.Nrho) {
            r.n0 = n0;
            r.fr = (float)(xrh - fn);
        }
    }
    out[idx] = r;
}

// --------------------------------------------------------------------------
// Plan time, FP64: zeta_hat as a quadrature written as a matrix product,
// Z = A B with A[k1][n] = cos(2 pi theta_n w1) and B[n][k2] the complex
// weights (real and imaginary parts as two matrices). 16x16 tiles.
// --------------------------------------------------------------------------
__global__ void k_zeta_gemm(const double* __restrict__ A, const double* __restrict__ Bre,
                            const double* __restrict__ Bim, int n1, int nn, int n2,
                            double* __restrict__ Zre, double* __restrict__ Zim) {
    __shared__ double sA[16][17];
    __shared__ double sR[16][17];
    __shared__ double sI[16][17];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int row = blockIdx.y * 16 + ty;   // k1
    const int col = blockIdx.x * 16 + tx;   // k2
    double accr = 0.0, acci = 0.0;
    for (int t0 = 0; t0 < nn; t0 += 16) {
        const int ta = t0 + tx, tb = t0 + ty;
        sA[ty][tx] = (row < n1 && ta < nn) ? A[(size_t)row * nn + ta] : 0.0;
        sR[ty][tx] = (tb < nn && col < n2) ? Bre[(size_t)tb * n2 + col] : 0.0;
        sI[ty][tx] = (tb < nn && col < n2) ? Bim[(size_t)tb * n2 + col] : 0.0;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            accr = fma(sA[ty][q], sR[q][tx], accr);
            acci = fma(sA[ty][q], sI[q][tx], acci);
        }
        __syncthreads();
    }
    if (row < n1 && col < n2) {
        Zre[(size_t)row * n2 + col] = accr;
        Zim[(size_t)row * n2 + col] = acci;
    }
}

// --------------------------------------------------------------------------
// Direct summation over hyperbolas on the GPU (FP32): the plain O(N^3)
// comparator, Eq. (3) with the same discretisation as the paper's reference
// (Keys cubic in t, trapezoid in x).
// --------------------------------------------------------------------------
__device__ __forceinline__ float keys_w(float s) {
    s = fabsf(s);
    if (s <= 1.f) return (1.5f * s - 2.5f) * s * s + 1.f;
    if (s < 2.f) return ((-0.5f * s + 2.5f) * s - 4.f) * s + 2.f;
    return 0.f;
}

__global__ void __launch_bounds__(256) k_direct_fwd(const float* __restrict__ f, float* __restrict__ g,
                                                    int Nt, int Nx, int Ntau, float tau0_dt,
                                                    float dtau_dt, float qmin_dx_dt, float dq_dx_dt,
                                                    float two_dx) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int l = blockIdx.y;
    if (i >= Ntau) return;
    const float tt = tau0_dt + dtau_dt * (float)i;      // tau / dt
    const float qq = qmin_dx_dt + dq_dx_dt * (float)l;  // q dx / dt
    const float tt2 = tt * tt, qq2 = qq * qq;
    float acc = 0.f;
    for (int k = 0; k < Nx; ++k) {
        const float p = sqrtf(tt2 + qq2 * (float)k * (float)k);  // t / dt
        const float fl = floorf(p);
        const int j0 = (int)fl;
        const float s = p - fl;
        const float* tr = f + (size_t)k * Nt;
        float v = 0.f;
        if (j0 - 1 >= 0 && j0 + 2 < Nt) {
            v = __ldg(tr + j0 - 1) * keys_w(s + 1.f) + __ldg(tr + j0) * keys_w(s) +
                __ldg(tr + j0 + 1) * keys_w(s - 1.f) + __ldg(tr + j0 + 2) * keys_w(s - 2.f);
        } else {
#pragma unroll
            for (int d = -1; d <= 2; ++d) {
                const int jj = j0 + d;
                if (jj >= 0 && jj < Nt) v += __ldg(tr + jj) * keys_w(s - (float)d);
            }
        }
        acc += (k == 0 || k == Nx - 1) ? 0.5f * v : v;
    }
    g[(size_t)l * Ntau + i] = two_dx * acc;
}

__global__ void __launch_bounds__(256) k_direct_adj(const float* __restrict__ g, float* __restrict__ f,
                                                    int Nt, int Nx, int Ntau, int Nq, float tau0_dt,
                                                    float dtau_dt, float qmin_dx_dt, float dq_dx_dt,
                                                    float two_dx) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    if (j >= Nt) return;
    const float kk = (float)k;
    const float lo = fmaxf((float)(j - 2), 0.f), hi = (float)(j + 2);
    float acc = 0.f;
    for (int l = 0; l < Nq; ++l) {
        const float qq = (qmin_dx_dt + dq_dx_dt * (float)l) * kk;   // q x / dt
        const float qq2 = qq * qq;
        const float hi2 = hi * hi - qq2;
        if (hi2 < 0.f) continue;
        const float lo2 = lo * lo - qq2;
        const float tlo = lo2 > 0.f ? sqrtf(lo2) : 0.f;
        const float thi = sqrtf(hi2);
        int i0 = (int)floorf((tlo - tau0_dt) / dtau_dt) - 1;
        int i1 = (int)ceilf((thi - tau0_dt) / dtau_dt) + 1;
        i0 = max(i0, 0);
        i1 = min(i1, Ntau - 1);
        const float* gl = g + (size_t)l * Ntau;
        for (int i = i0; i <= i1; ++i) {
            const float tt = tau0_dt + dtau_dt * (float)i;
            const float p = sqrtf(tt * tt + qq2);
            acc += __ldg(gl + i) * keys_w(p - (float)j);
        }
    }
    f[(size_t)k * Nt + j] = ((k == 0 || k == Nx - 1) ? 0.5f : 1.f) * two_dx * acc;
}

// --------------------------------------------------------------------------
// Launchers
// --------------------------------------------------------------------------
int max_smem_optin() {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}

// Kernels with B-spline taps exist for 4 (cubic) and 6 (quintic) taps per
// axis; every piece of one launch has the same number.
#define HR_TAPS(NTAPS, ...)                                           \
    do {                                                              \
        if ((NTAPS) == 6) {                                           \
            constexpr int NT = 6;                                     \
            __VA_ARGS__;                                              \
        } else if ((NTAPS) == 4) {                                    \
            constexpr int NT = 4;                                     \
            __VA_ARGS__;                                              \
        } else {                                                      \
            return (int)cudaErrorInvalidValue;                        \
        }                                                             \
    } while (0)

template <class Src, class T>
static int launch_grid_as(void (*kern)(Src, const T*), int nb, void* stream, const Src& B, const T* f) {
    return launch_chain(8, kern, nb, kUnitChunks, 0, stream, B, f);
}

int launch_grid_tiles(const PieceDev* P, int n, const float* f, void* stream) {
    PieceBatch B;
    const int nb = make_batch(P, n, B, [](const PieceDev& q) { return q.nunits; });
    if (nb > 0) HR_TAPS(P[0].ntaps, return launch_grid_as(k_grid_tiles<PieceBatch, float, NT>, nb, stream, B, f));
    return 0;
}

int launch_grid_tiles_dev(const DevBatch& S, int nblocks, int ntaps, const void* f, int in_type, void* stream) {
    if (nblocks <= 0) return 0;
    HR_TAPS(ntaps, {
        if (in_type == kInBF16)
            return launch_grid_as(k_grid_tiles<DevBatch, __nv_bfloat16, NT>, nblocks, stream, S, (const __nv_bfloat16*)f);
        return launch_grid_as(k_grid_tiles<DevBatch, float, NT>, nblocks, stream, S, (const float*)f);
    });
    return 0;
}

// Dynamic shared memory the per-column profile kernels (the output
// interpolation and its adjoint's profiles) may take on the current device:
// the opt-in limit less the larger of the two kernels' static shared arrays.
size_t interp_smem_limit(int ntaps) {
    size_t stat = 0;
    const void* fns[2] = {ntaps == 6 ? (const void*)k_interp_columns<6> : (const void*)k_interp_columns<4>,
                          ntaps == 6 ? (const void*)k_col_profiles_cols<6> : (const void*)k_col_profiles_cols<4>};
    for (const void* fn : fns) {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        stat = std::max(stat, (size_t)fa.sharedSizeBytes);
    }
    const size_t lim = (size_t)max_smem_optin();
    return lim > stat ? lim - stat : 0;
}

int launch_col_profiles_cols(const PieceDev* pieces, const int4* cmap, int ncols, int nrho_max, int np_max,
                             int ntau_all, int np_all, int ntaps, const float* g, void* stream) {
    if (np_max > kMaxColPieces) return (int)cudaErrorInvalidValue;
    const size_t sm = (size_t)np_max * nrho_max * sizeof(int);
    HR_TAPS(ntaps, {
        if (int e = set_smem((const void*)k_col_profiles_cols<NT>, sm)) return e;
        if (ncols > 0)
            return launch_chain(5, k_col_profiles_cols<NT>, ncols, 256, sm, stream, pieces, cmap, nrho_max, ntau_all, np_all, g);
    });
    return 0;
}

int launch_interp_columns(const PieceDev* pieces, const int4* cmap, int ncols, int nrho_max, int np_max,
                          int ntau_all, int np_all, int ntaps, size_t limit, float* g, void* stream) {
    if (np_max > kMaxColPieces) return (int)cudaErrorInvalidValue;
    // profiles on 16-byte boundaries where shared memory holds them so
    const int up = (nrho_max + 3) & ~3;
    const int pstride = (size_t)np_max * up * sizeof(float) <= limit ? up : nrho_max;
    const size_t sm = (size_t)np_max * pstride * sizeof(float);
    HR_TAPS(ntaps, {
        if (int e = set_smem((const void*)k_interp_columns<NT>, sm)) return e;
        if (ncols > 0)
            return launch_chain(8, k_interp_columns<NT>, ncols, 256, sm, stream, pieces, cmap, pstride, ntau_all, np_all, g);
    });
    return 0;
}

int launch_gather_samples(const PieceDev* pieces, const int4* smap, int nblocks, float* f, int np_all, int Nt_all,
                          int Nx_all, int ntaps, void* stream) {
    if (nblocks > 0)
        HR_TAPS(ntaps, return launch_chain(8, k_gather_samples<NT>, nblocks, kSampleBlock, 0, stream, pieces, smap, f, np_all,
                                           Nt_all, Nx_all));
    return 0;
}

int launch_sample_table(const TableArgs& A, const double* cj, const double* wk, const int* jfirst,
                        SampleEnt* out) {
    const long total = (long)A.nj * A.Nx;
    k_sample_table<<<(unsigned)((total + 255) / 256), 256>>>(A, cj, wk, jfirst, out);
    return check_launch();
}

int launch_radon_table(const TableArgs& A, const double* qb2, RadonEnt* out) {
    const long total = (long)A.ncol * A.Ntau;
    k_radon_table<<<(unsigned)((total + 255) / 256), 256>>>(A, qb2, out);
    return check_launch();
}

int launch_zeta_gemm(const double* A, const double* Bre, const double* Bim, int n1, int nn, int n2,
                     double* Zre, double* Zim, void* stream) {
    dim3 bs(16, 16);
    dim3 gs((n2 + 15) / 16, (n1 + 15) / 16);
    k_zeta_gemm<<<gs, bs, 0, (cudaStream_t)stream>>>(A, Bre, Bim, n1, nn, n2, Zre, Zim);
    return check_launch();
}

int launch_direct_fwd(const float* f, float* g, int Nt, int Nx, int Ntau, int Nq, double dt,
                      double dx, double tau0, double dtau, double qmin, double dq, void* stream) {
    dim3 bs(256);
    dim3 gs((Ntau + 255) / 256, Nq);
    k_direct_fwd<<<gs, bs, 0, (cudaStream_t)stream>>>(
        f, g, Nt, Nx, Ntau, (float)(tau0 / dt), (float)(dtau / dt), (float)(qmin * dx / dt),
        (float)(dq * dx / dt), (float)(2.0 * dx));
    return check_launch();
}

int launch_direct_adj(const float* g, float* f, int Nt, int Nx, int Ntau, int Nq, double dt,
                      double dx, double tau0, double dtau, double qmin, double dq, void* stream) {
    dim3 bs(256);
    dim3 gs((Nt + 255) / 256, Nx);
    k_direct_adj<<<gs, bs, 0, (cudaStream_t)stream>>>(
        g, f, Nt, Nx, Ntau, Nq, (float)(tau0 / dt), (float)(dtau / dt), (float)(qmin * dx / dt),
        (float)(dq * dx / dt), (float)(2.0 * dx));
    return check_launch();
}

}  // namespace hr
