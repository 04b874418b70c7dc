// What the matrix-vector kernels share: the accumulator word, the ring of record slots and its bounded waits, shared-memory reads.
#pragma once
#include "llvq_cut.h"
#include "llvq_internal.cuh"

namespace llvq {
namespace {

constexpr int kWarps = 16;                 // warps per CTA of the kernels for one and two vectors
constexpr int kThreads = kWarps * 32;
constexpr int kSlots = 2;                  // ring slots per warp
constexpr int kEarlySlots = 1;             // slots filled before the wait for the previous kernel; the rest once x is being prepared

// Vectors in sets of four (batch_in_sets): the bytes of a block's record of x a set, warps per CTA.  Two sets need more registers than
// sixteen warps leave a thread (128): sixteen that spill their sums take twice the time of twelve with 168, which spill 36 bytes.
constexpr int kBatchSetBytes = 480;
constexpr int kBatchSharedWords = sizeof(Cut) / 4 + LLVQ_MAX_BATCH + 1;        // what the CTA of such a launch shares besides: see gemv_batch_kernel
__host__ __device__ constexpr int batch_sets(int batch) { return batch > 4 ? 2 : 1; }
__host__ __device__ constexpr int batch_warps(int sets) { return sets > 1 ? 12 : kWarps; }
// the kernel for one vector, for two and, in pairs, for five and six
__host__ __device__ constexpr int gemv_warps(int vectors) { return vectors > 4 ? 12 : kWarps; }

// fixed-point accumulator word: bits 53..63 count units, bits 0..52 sum the biased unit values
constexpr int kCountShift = 53;
constexpr unsigned long long kSumMask = (1ull << kCountShift) - 1;
constexpr long long kUnitBias = 1ll << 41;     // a unit's value is below 2^40 quanta in magnitude

// running maximum of |fp16| over both halves of a word, kept as two 15-bit patterns; a NaN stays one.  The magnitude goes into the maximum's
// instruction, which an AND of the bits did not: sixteen instructions less in the scan of x, which every launch waits for (us a launch in
// a chain: 1024 x 2560 3.23 -> 3.19, 4096 x 4096 4.89 -> 4.84, 8192 x 8192 9.08 -> 9.01; two vectors on 4096 x 4096 6.37 -> 6.24)
__device__ __forceinline__ uint32_t max_abs_pair(uint32_t m, uint32_t x2) {
    const __half2 r = __hmax2_nan(*reinterpret_cast<const __half2 *>(&m), __habs2(*reinterpret_cast<const __half2 *>(&x2)));
    return *reinterpret_cast<const uint32_t *>(&r);
}

// exact power of two as a float, |e| < 126
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// 2^xexp, xexp the exponent that the largest |x| (FP16 bits) sets the fixed-point scale by: every |x| is below it.  NaN where an entry is infinite or no
// number: such a vector's fixed-point activations mean nothing, and y, which has this factor, must not look like a result.
constexpr uint32_t kInfinity16 = 0x7c00u;
__device__ __forceinline__ int x_exponent(uint32_t most) { return max((int)(most >> 10), 1) - 14; }
__device__ __forceinline__ float x_factor(uint32_t most) { return most < kInfinity16 ? pow2f(x_exponent(most)) : __int_as_float(0x7fffffff); }

// ---- asynchronous copies: global -> shared, completion counted on an mbarrier in shared memory
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Every wait is bounded in time: a poll that fails starts a clock, and once kWaitLimitCycles SM cycles
// (about a second) have passed without the barrier completing, the caller records an error and winds
// down.  The first poll reads no clock, so a wait that is already satisfied costs one instruction.
constexpr long long kWaitLimitCycles = 2000000000ll;
__device__ __forceinline__ bool mbar_wait_for(uint32_t bar, uint32_t parity, long long limit_cycles) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    do {
        if (mbar_try(bar, parity)) return true;
    } while (clock64() - t0 < limit_cycles);
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) { return mbar_wait_for(bar, parity, kWaitLimitCycles); }

// Ring reads through 32-bit shared-memory addresses.  Volatile: they must stay behind the wait on the
// slot's barrier and ahead of the copy that refills the slot.
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
// Returns zero, but only once its operands are available: an address that adds this zero cannot be
// formed before the loads that produced them have completed.
__device__ __forceinline__ uint32_t settled(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t z;
    asm volatile("lop3.b32 %0, %1, %2, %3, 0x00;" : "=r"(z) : "r"(a), "r"(b), "r"(c));
    return z;
}

// Shared-memory reads with a constant byte offset folded into the instruction.  Volatile, so that the
// compiler never moves one out of the branch that guards it: an address formed for a unit this CTA does not
// own may lie outside its shared memory.
template <int OFF>
__device__ __forceinline__ uint32_t lds32_at(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF));
    return v;
}
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}

// (a & b) | c in one instruction
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

__host__ __device__ inline int fast_div(int n, const FastDiv &f, int d) {
#ifdef __CUDA_ARCH__
    (void)d;
    return f.mul ? (int)(__umulhi((uint32_t)n, f.mul) >> f.shift) : n;
#else
    (void)f;
    return n / d;
#endif
}

template <typename K>
int allow_max_smem(K kernel, int optin) {
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess) return -1;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes) != cudaSuccess) return -1;
    // ask for the largest shared-memory carve-out, so that a CTA of the next kernel of the stream can
    // settle beside a running one (programmatic dependent launch) whenever two of them fit
    return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess ? 0 : -1;
}

}  // namespace
int batch_configure(int optin);            // sets the batch kernels' shared-memory attributes
cudaError_t launch_batch(const GemvParams &p, const GemvLaunch &g, bool pdl, cudaStream_t s);
}  // namespace llvq
