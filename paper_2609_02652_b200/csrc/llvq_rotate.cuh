// Device pieces of the exact Walsh-Hadamard rotation: for the rotation kernel integers in units of 2^-24, butterflies on
// 64-bit sums, one rounding to FP16; for the GEMV whose prologue rotates x itself the same sums in f64.
#pragma once
#include <cstdint>

#include <cuda_fp16.h>

namespace llvq {

// Where value i of the array lives in shared memory.  A thread of a pass touches eight values 2^s apart and its
// neighbours the values beside them; with the low four index bits XORed by the next four, every such access of a
// warp (32 values of 8 bytes) spreads evenly over the banks: two wavefronts, the least 256 bytes take.
__device__ __forceinline__ int rot_at(int i) { return i ^ ((i >> 4) & 15); }

// R stages of the in-place butterfly on 2^R values: (a, b) -> (a + b, a - b) over every pair that differs in
// one index bit.  With the values taken at stride 2^s these are stages s .. s + R - 1 of the transform.
template <int R, typename T>
__device__ __forceinline__ void rot_butterflies(T (&a)[8]) {
#pragma unroll
    for (int h = 1; h < (1 << R); h <<= 1) {
#pragma unroll
        for (int i = 0; i < (1 << R); i++) {
            if ((i & h) == 0) {
                const T u = a[i], w = a[i + h];
                a[i] = u + w;
                a[i + h] = u - w;
            }
        }
    }
}

// One pass over `count` values in shared memory (whole blocks): stages S .. S + R - 1.  S and R are compile-time
// so that the eight addresses of a thread come from one computed address and constants.
template <int R, int S>
__device__ __forceinline__ void rot_pass(long long *v, int count, int tid, int nthreads) {
    for (int g = tid; g < (count >> R); g += nthreads) {
        const int base = ((g >> S) << (S + R)) | (g & ((1 << S) - 1));
        long long a[8];
        if (S >= 8) {
            // the stride leaves the eight swizzled index bits alone
            long long *at = v + rot_at(base);
#pragma unroll
            for (int j = 0; j < (1 << R); j++) a[j] = at[j << S];
            rot_butterflies<R>(a);
#pragma unroll
            for (int j = 0; j < (1 << R); j++) at[j << S] = a[j];
        } else {
#pragma unroll
            for (int j = 0; j < (1 << R); j++) a[j] = v[rot_at(base + (j << S))];
            rot_butterflies<R>(a);
#pragma unroll
            for (int j = 0; j < (1 << R); j++) v[rot_at(base + (j << S))] = a[j];
        }
    }
}
template <int S>
__device__ __forceinline__ void rot_pass_from(long long *v, int block_log2, int count, int tid, int nthreads) {
    const int r = block_log2 - S;
    if (r >= 3) rot_pass<3, S>(v, count, tid, nthreads);
    else if (r == 2) rot_pass<2, S>(v, count, tid, nthreads);
    else rot_pass<1, S>(v, count, tid, nthreads);
    __syncthreads();
}
// the passes after the first: stages 3 .. block_log2 - 1 (block_log2 <= 14), three at a time, a barrier after each
__device__ __forceinline__ void rot_later_passes(long long *v, int block_log2, int count, int tid, int nthreads) {
    if (block_log2 > 3) rot_pass_from<3>(v, block_log2, count, tid, nthreads);
    if (block_log2 > 6) rot_pass_from<6>(v, block_log2, count, tid, nthreads);
    if (block_log2 > 9) rot_pass_from<9>(v, block_log2, count, tid, nthreads);
    if (block_log2 > 12) rot_pass_from<12>(v, block_log2, count, tid, nthreads);
}

// stores the eight values first .. first + 7 (first a multiple of eight)
__device__ __forceinline__ void rot_store8(long long *v, int first, const long long (&a)[8]) {
#pragma unroll
    for (int k = 0; k < 8; k++) v[rot_at(first + k)] = a[k];
}

// Eight consecutive FP16 coordinates -> integers in units of 2^-24 (exact: a power-of-two scaling of an 11-bit
// significand), sign flips applied (bit i of `flips` set = coordinate i negated).
__device__ __forceinline__ void rot_load8(const uint4 &raw, uint32_t flips, long long (&a)[8]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
        const long long lo = __float2ll_rn(f.x * 16777216.f), hi = __float2ll_rn(f.y * 16777216.f);
        a[2 * i] = ((flips >> (2 * i)) & 1u) ? -lo : lo;
        a[2 * i + 1] = ((flips >> (2 * i + 1)) & 1u) ? -hi : hi;
    }
}

// The one rounding: eight exact sums -> f64 (exact below 2^53) -> times 2^-24 / sqrt(B) -> FP16, nearest even.
// The sums are values first .. first + 7 of the array v (first a multiple of eight).
__device__ __forceinline__ uint4 rot_round8(const long long *v, int first, double scale) {
    uint32_t out[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const __half lo = __double2half((double)v[rot_at(first + 2 * i)] * scale);
        const __half hi = __double2half((double)v[rot_at(first + 2 * i + 1)] * scale);
        out[i] = (uint32_t)__half_as_ushort(lo) | ((uint32_t)__half_as_ushort(hi) << 16);
    }
    return make_uint4(out[0], out[1], out[2], out[3]);
}

// ---- the rotation of a stretch of x inside the GEMV.  A CTA needs the coordinates [need_lo, need_hi) of the rotated vector, a
// small part of long blocks, so the stages run from the widest stride down: once the stages of strides 2^s and
// more are done, only the pieces of 2^s coordinates that meet the part needed go on (rot_first says which blocks are long).  In f64 the sums are those of the
// integers: every partial sum ahead of a 2^14 block's last stage is a multiple of 2^-24 below 2^29, hence exact, and where
// the last stage's is not, it is rounded as the integer would be on its way to f64.  One instruction an addition where the
// 64-bit integers take two, and no conversion at the end.

// The f64 value of an FP16's bits (in the low half of h), times 2^-1008: its exponent and mantissa, moved up.
__device__ __forceinline__ double rot_widen(uint32_t h) { return __hiloint2double((int)(((uint32_t)(int)(short)h << 10) & 0x81ffffffu), 0); }

// Stages S .. S + R - 1 over the coordinates [lo, hi) (multiples of 2^(S+R)); of the results those in [keep_lo, keep_hi)
// (multiples of 2^S) are stored.  v holds coordinate first + i in place rot_at(i).  RAW: the inputs are FP16, raw[0] = coordinate lo.
template <int R, bool RAW>
__device__ __forceinline__ void rot_narrow(double *v, int first, const __half *raw, int lo, int hi, int keep_lo, int keep_hi, int S, int tid, int nthreads) {
    for (int g = tid; g < ((hi - lo) >> R); g += nthreads) {
        const int base = ((g >> S) << (S + R)) | (g & ((1 << S) - 1));
        double a[8];
#pragma unroll
        for (int j = 0; j < (1 << R); j++) {
            if (RAW) a[j] = rot_widen(reinterpret_cast<const uint16_t *>(raw)[base + (j << S)]);
            else a[j] = v[rot_at(lo - first + base + (j << S))];
        }
        rot_butterflies<R>(a);
#pragma unroll
        for (int j = 0; j < (1 << R); j++) {
            const int c = lo + base + (j << S);
            if (c >= keep_lo && c < keep_hi) v[rot_at(c - first)] = a[j];
        }
    }
}

// Stages 3 .. 2 + R of a piece of 8 * 2^R by 2^R neighbouring lanes: the lane whose eight values begin at place `at` takes its share
// of the sets of values eight apart.  A __syncwarp() belongs between this and rot_finish8.
template <int R>
__device__ __forceinline__ void rot_middle8(double *v, int at) {
    constexpr int kLanes = 1 << R, kSets = 8 >> R;
    const int base = (at & ~(8 * kLanes - 1)) + ((at >> 3) & (kLanes - 1));
    double a[kSets][8];
#pragma unroll
    for (int c = 0; c < kSets; c++) {
#pragma unroll
        for (int j = 0; j < kLanes; j++) a[c][j] = v[rot_at(base + kLanes * c + 8 * j)];
        rot_butterflies<R>(a[c]);
#pragma unroll
        for (int j = 0; j < kLanes; j++) v[rot_at(base + kLanes * c + 8 * j)] = a[c][j];
    }
}

// Eight consecutive FP16 values (two a word) and their three narrowest stages.
__device__ __forceinline__ void rot_widen8(const uint4 &x, double (&a)[8]) {
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int k = 0; k < 8; k++) a[k] = rot_widen(w[k >> 1] >> (16 * (k & 1)));
    rot_butterflies<3>(a);
}

// The same, stored as the values at places at .. at + 7 (at a multiple of eight).
__device__ __forceinline__ void rot_start8(double *v, int at, const uint4 &x) {
    double a[8];
    rot_widen8(x, a);
#pragma unroll
    for (int k = 0; k < 8; k++) v[rot_at(at + k)] = a[k];
}

// The one rounding of eight sums.
__device__ __forceinline__ uint4 rot_to_half8(const double (&a)[8], double scale) {
    uint32_t out[4];
#pragma unroll
    for (int i = 0; i < 4; i++)
        out[i] = (uint32_t)__half_as_ushort(__double2half(a[2 * i] * scale)) | ((uint32_t)__half_as_ushort(__double2half(a[2 * i + 1] * scale)) << 16);
    return make_uint4(out[0], out[1], out[2], out[3]);
}

// The eight values from place `at` on (a multiple of eight), their three narrowest stages if those are still to do, rounded.
__device__ __forceinline__ uint4 rot_finish8(const double *v, int at, bool stages_left, double scale) {
    double a[8];
#pragma unroll
    for (int k = 0; k < 8; k++) a[k] = v[rot_at(at + k)];
    if (stages_left) rot_butterflies<3>(a);
    return rot_to_half8(a, scale);
}

// A whole block of eight.
__device__ __forceinline__ uint4 rot_whole8(const uint4 &x, double scale) {
    double a[8];
    rot_widen8(x, a);
    return rot_to_half8(a, scale);
}

}  // namespace llvq
