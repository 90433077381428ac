// Device and launch helpers shared by the kernel files: the piece of a block
// in a batched launch, shared-memory checks and limits.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "internal.h"

namespace hr {

extern __shared__ __align__(16) float smem_f[];

// Piece of this block in a batched launch, and the block's index within it:
// from the descriptors passed as a kernel parameter (up to kMaxBatch pieces)
// or from a device-resident batch (any number of pieces of many gathers).
__device__ __forceinline__ int batch_piece(const PieceBatch& B, int& bx) {
    int pi = 0;
#pragma unroll
    for (int k = 1; k < kMaxBatch; ++k)
        if (k < B.n && (int)blockIdx.x >= B.first[k]) pi = k;
    bx = (int)blockIdx.x - B.first[pi];
    return pi;
}
__device__ __forceinline__ const PieceDev& piece_of(const PieceBatch& B, int& bx) { return B.p[batch_piece(B, bx)]; }
__device__ __forceinline__ const PieceDev& piece_of(const DevBatch& B, int& bx) {
    const int2 m = __ldg(B.map + blockIdx.x);
    bx = m.y;
    return B.p[m.x];
}

// The radices of pass 0 (dif_plan).
#define HR_RADIX_CASES(CALL) \
    case 16: CALL(16); break; \
    case 12: CALL(12); break; \
    case 10: CALL(10); break; \
    case 9: CALL(9); break;   \
    case 8: CALL(8); break;   \
    case 6: CALL(6); break;   \
    case 5: CALL(5); break;   \
    case 4: CALL(4); break;   \
    case 3: CALL(3); break;   \
    default: CALL(2); break;

// Dynamic shared memory of the launch: the row and column kernels check it
// against what their piece needs and leave the block untouched (never write
// past it) if a launch gave too little.
__device__ __forceinline__ unsigned dyn_smem_bytes() {
    unsigned r;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
    return r;
}

// 16-byte asynchronous copies global -> shared (cp.async; the completion
// wait is the hardware's, no spin loop).
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void cp_async16_or_zero(void* smem_dst, const void* gmem_src, bool on) {   // zeros unless on
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gmem_src), "r"(on ? 16 : 0) : "memory");
}

// Programmatic dependent launch: a kernel of a transform may start while its
// predecessor on the stream still runs. Each calls chain_wait() before it
// touches anything another kernel writes (it returns once the predecessor has
// completed, with its writes visible); every CTA waits, so the kernels
// complete in order. A launch that fits the chip at once or nearly so (per_sm
// CTAs per SM) is made so, and calls chain_next() at its start, which lets the next
// kernel's CTAs take the room left and do what depends on the plan alone:
// such transforms are bound by launch and start-up latencies (256 x 64 forward
// 41 -> 33 us, 1024 x 256 FISTA 5.8 -> 4.7 ms). Larger launches are ordinary
// ones: CTAs that start as room appears pile up on the SMs that finish first
// (2048^2 forward 222 -> 231 us, 4096^2 pair 1722 -> 1815 us).
constexpr int kSMs = 152;
template <int PER_SM>
__device__ __forceinline__ void chain_wait() {
    if (gridDim.x <= PER_SM * kSMs) asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <int PER_SM>
__device__ __forceinline__ void chain_next() {
    if (gridDim.x <= PER_SM * kSMs) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... K, class... A>
inline int launch_chain(int per_sm, void (*kern)(K...), int grid, int block, size_t smem, void* stream, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = grid <= per_sm * kSMs ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<K>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return (int)e;
}

inline int check_launch() {
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 0 : (int)e;
}

// Dynamic shared-memory limit of a kernel: raised only when a launch needs
// more than the largest value already set on this device (the attribute call
// costs host time on every launch otherwise).
inline int set_smem(const void* fn, size_t bytes) {
    struct Entry { const void* fn; int dev; size_t bytes; };
    static std::mutex mu;
    static std::vector<Entry> set;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    for (const Entry& e : set)
        if (e.fn == fn && e.dev == dev && e.bytes >= bytes) return 0;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return (int)e;
    for (Entry& en : set)
        if (en.fn == fn && en.dev == dev) {
            en.bytes = bytes;
            return 0;
        }
    set.push_back(Entry{fn, dev, bytes});
    return 0;
}

// Batch descriptor of n pieces with count(piece) blocks each; returns the
// total number of blocks.
template <class F>
inline int make_batch(const PieceDev* P, int n, PieceBatch& B, F&& count) {
    B.n = n;
    int total = 0;
    for (int k = 0; k < kMaxBatch; ++k) {
        B.first[k] = total;
        if (k < n) {
            B.p[k] = P[k];
            total += count(P[k]);
        }
    }
    B.first[kMaxBatch] = total;
    return total;
}

}  // namespace hr
