// From an index of the ball to the 24 four-bit codes u_i = 8 + floor(x_i / 2) (and magnitudes, signs), with the tables of
// llvq_unrank.h: the first part of `blob` in shared memory, the lists in global memory (5.6 MB, resident in L2).
//
// The index splits as the paper states it (Sec. 2.1: classes first, then arrangements and signs inside a class, as a
// mixed-radix number).  The digit order used here:
//   even type:  ((codeword rank * perm_a + rank_a) * perm_b + rank_b) << sign_bits | signs
//   odd type:   arrangement rank * 4096 + message bits of the codeword
// Arrangement ranks are lexicographic over the distinct orderings, smaller magnitude first; sign bits run over the
// non-zero off-support coordinates first, then the support coordinates but the last, whose sign restores the sum
// condition mod 8.
//
// Coordinates are worked on eight at a time, a nibble each.  With j = (|x| - 1) / 2 (odd type) a positive coordinate's
// code is 8 + j and a negative one's 7 - j, the complement; with h = |x| / 2 (even type) they are 8 + h and 8 - h, the
// two's complement.  So a word of codes is the word of j or h, with bit 3 set, complemented nibble-wise where the
// sign word says so (and, for the even type, one added there).
#pragma once
#include <cstdint>

#include "llvq_unrank.h"

#ifdef __CUDACC__
#define LLVQ_HD __host__ __device__ __forceinline__
#else
#define LLVQ_HD inline
#endif

namespace llvq {

struct UnrankView {
    const uint8_t *blob;         // its first kUnrankSharedBytes are read here
    const uint8_t *far;          // and the others here
    const uint64_t *pairs;
    const uint32_t *tail8;
    const uint32_t *tab_b;
};

// Magnitudes (j or h) and signs (1 = negative) of the 24 coordinates, eight nibbles a word.
struct Point {
    uint32_t mag[3], neg[3];
};

LLVQ_HD int popcount32(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __popc(v);
#else
    return __builtin_popcount(v);
#endif
}
LLVQ_HD uint32_t byte_perm(uint32_t a, uint32_t b, uint32_t select) {
#ifdef __CUDA_ARCH__
    return __byte_perm(a, b, select);
#else
    uint32_t r = 0;
    for (int i = 0; i < 32; i += 8) {
        const uint32_t from = select >> (i / 2) & 7u;
        r |= ((from < 4u ? a >> (8u * from) : b >> (8u * (from - 4u))) & 0xffu) << i;
    }
    return r;
#endif
}
// the low `bits` bits of `low`, and above them the low ones of `high`
LLVQ_HD uint32_t join(uint32_t low, uint32_t high, uint32_t bits) {
#ifdef __CUDA_ARCH__
    return __funnelshift_rc(__funnelshift_lc(0u, low, 32u - bits), high, 32u - bits);
#else
    return (uint32_t)((low & ((1ull << bits) - 1)) | (uint64_t)high << bits);
#endif
}
LLVQ_HD float u64_to_float(uint64_t v) { return (float)v; }
LLVQ_HD uint32_t float_bits(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    union { float f; uint32_t u; } c;
    c.f = f;
    return c.u;
#endif
}
LLVQ_HD float bits_float(uint32_t u) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    union { uint32_t u; float f; } c;
    c.u = u;
    return c.f;
#endif
}
// floor(a * b), a * b below 2^23
LLVQ_HD uint32_t floor_product(float a, float b) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(__fmaf_rd(a, b, 8388608.f)) - 0x4b000000u;       // whole numbers from 2^23 on, rounded down
#else
    return (uint32_t)((double)a * (double)b);
#endif
}
template <typename T>
LLVQ_HD const T &blob_at(const UnrankView &v, int offset, uint32_t i) { return reinterpret_cast<const T *>(v.blob + offset)[i]; }
template <typename T>
LLVQ_HD const T &far_at(const UnrankView &v, int offset, uint32_t i) { return reinterpret_cast<const T *>(v.far + offset)[i]; }

// bits 0..7 of b as the low bits of eight nibbles (the partial products do not overlap)
LLVQ_HD uint32_t spread8(uint32_t b) {
    b = ((b & 0xffu) * 0x1001u) & 0x000f000fu;
    b = (b * 0x41u) & 0x03030303u;
    return (b * 9u) & 0x11111111u;
}
// eight two-bit fields as eight nibbles
LLVQ_HD uint32_t spread_pairs(uint32_t b) {
    b &= 0xffffu;
    b = (b | b << 8) & 0x00ff00ffu;
    b = (b | b << 4) & 0x0f0f0f0fu;
    return (b | b << 2) & 0x33333333u;
}
// the low bits of eight nibbles as bits 0..7
LLVQ_HD uint32_t gather8(uint32_t w) {
    w = (w | w >> 3) & 0x03030303u;
    w = (w | w >> 6) & 0x000f000fu;
    return (w | w >> 12) & 0xffu;
}

// slot of the class guide an index (below 2^48) lies in
LLVQ_HD int guide_slot(uint64_t idx) {
    const int s = (int)(float_bits(u64_to_float(idx)) >> kGuideShift) - kGuideFirst;
    return s < 0 ? 0 : s;
}

// Class of a valid index: the last c with base[c] <= idx, searched between the guide's bounds.
LLVQ_HD int find_class(const UnrankView &v, uint64_t idx) {
    const int s = guide_slot(idx);
    int lo = blob_at<uint16_t>(v, kUnrankGuide, s), hi = blob_at<uint16_t>(v, kUnrankGuide, s + 1) + 1;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (blob_at<uint64_t>(v, kUnrankBase, mid) <= idx) lo = mid; else hi = mid;
    }
    return lo;
}

// Of `left` coordinates that have T orderings, T * copies / left begin with a given value.  The quotient is exact and below
// 2^32: shifted right by left's power of two, the product times the inverse of left's odd part modulo 2^32.
LLVQ_HD uint32_t portion(uint32_t T, uint32_t copies, const UnrankStep &e) { return (uint32_t)(((uint64_t)T * copies) >> e.shift) * e.inverse; }

// The position of rank r among the draws of two from a multiset, given their ratio to its orderings: right, or one too large.
LLVQ_HD uint32_t draw_position(uint32_t r, float ratio, uint32_t draws) {
    const uint32_t at = floor_product((float)r, ratio);
    return at < draws ? at : draws - 1u;
}
// The pair of rank r, from the entry at that position: the first rank of the pair there tells whether it was one too large.  One step back is the
// most there is (a host test runs all the tables), and the most that is taken, whatever a table holds: a loop that looked on until it
// found the rank would not end on a table that does not hold it.  Against that loop, us: 9728 x 2560 34.8 -> 34.6, into the 13-byte layout 35.2 -> 34.7; 17408
// x 5120 into the 10-byte layout 139.5 -> 140.2, 9728 x 2560 48.4 -> 48.2.
LLVQ_HD uint64_t pair_drawn(const uint64_t *entry, uint32_t r) {
    uint64_t pair = *entry;
    if (r < (uint32_t)pair) pair = entry[-1];
    return pair;
}

// Odd type.  Sixteen coordinates come two at a time from the table of draws, the ordering of the last eight is an entry of
// a list.  The position of the draw is a float estimate that is right or one too large, which the first rank of the pair it names
// tells.  Rolled up: eight steps' code would crowd the instruction cache.  The load unit and its latency bound this, so a step
// reads one table only, at random (9728 x 2560: 35.2 us, 17408 x 5120: 106).  With the ratios in a table of their own in shared memory
// it takes 36.2 and 112, with the bounds of a pair worked out from the number of orderings (four multiplications to 64 bits and a
// reciprocal a step) 39 and 125, with the second eight coordinates one at a time from lists in shared memory 46.
LLVQ_HD void unrank_odd(const UnrankView &v, const UnrankDesc &d, uint64_t r47, Point &p) {
    const uint32_t message = (uint32_t)r47 & 4095u;
    const uint32_t cw = blob_at<uint32_t>(v, kUnrankGolayMsg, message & 63u) ^ blob_at<uint32_t>(v, kUnrankGolayMsg, 64 + (message >> 6));
    uint32_t r = (uint32_t)(r47 >> 12), set = (d.flags >> 1) & 255u, word = 0, left = 24, first = 0, high;
    float ratio = blob_at<float>(v, kUnrankRatio, set);
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
    while (true) {
        const uint32_t draws = left * (left - 1u);
        const uint64_t pair = pair_drawn(v.pairs + (first + set * draws + draw_position(r, ratio, draws)), r);
        r -= (uint32_t)pair;
        high = (uint32_t)(pair >> 32);
        word = byte_perm(word, high, 0x5321u);
        left -= 2u;
        if (left == 8u) break;
        first += kOddSets * draws;
        set = high & 255u;
        ratio = bits_float((high >> 4) + kRatioBase);
        if (left == 16u) p.mag[0] = word;
    }
    p.mag[1] = word;
    p.mag[2] = v.tail8[(high >> 16) + r];
    // x_i = 1 + 2 c_i modulo 4: 1 + 2j is of the wrong residue, and so negated, where j's parity differs from c_i
#pragma unroll
    for (int w = 0; w < 3; w++) p.neg[w] = (p.mag[w] & 0x11111111u) ^ spread8(cw >> (8 * w));
}

// The nibbles of `word`: as many as `mask` has bits to the mask's places, in order, the others to the other places.  One selector
// for two byte permutations: masked shifts by 4, 2 and 1 places read 16 bytes for the mask's nibbles and again for the others.
LLVQ_HD uint32_t to_places(const UnrankView &v, uint32_t mask, uint32_t word) {
    const uint32_t select = blob_at<uint32_t>(v, kUnrankMerge, mask);
    const uint32_t even = word & 0x0f0f0f0fu, odd = (word >> 4) & 0x0f0f0f0fu;
    return byte_perm(even, odd, select) | byte_perm(even, odd, select >> 16) << 4;
}

// Deals the low bits of `bits` to the nibbles of `word` that are not zero (two-bit values), in order; drops them from
// `bits`.
LLVQ_HD uint32_t deal_signs(const UnrankView &v, uint32_t word, uint32_t &bits) {
    const uint32_t mask = gather8((word | word >> 1) & 0x11111111u);
    const int n = popcount32(mask);
    const uint32_t dealt = to_places(v, mask, spread8(bits & ((1u << n) - 1u)));
    bits >>= n;
    return dealt;
}

// quotient and remainder of r / d for r < 2^42, quotient < 2^21, d < 2^24, given 1 / d: the float estimate is off by one at
// most, and the remainder settles it
LLVQ_HD uint32_t divide(uint64_t r, uint32_t d, float inv, uint32_t &rem) {
    uint32_t q = (uint32_t)(u64_to_float(r) * inv);
    int m = (int)((uint32_t)r - q * d);
    if (m < 0) { m += (int)d; q--; }
    if (m >= (int)d) { m -= (int)d; q++; }
    rem = (uint32_t)m;
    return q;
}

LLVQ_HD void unrank_even(const UnrankView &v, const UnrankDesc &d, uint64_t r, Point &p) {
    const uint32_t w = (d.flags >> 1) & 31u, sign_bits = (d.flags >> 6) & 31u, nz_b = (d.flags >> 11) & 15u;
    const uint32_t sigma = (uint32_t)r & ((1u << sign_bits) - 1u);
    uint32_t rank_a, rank_b;
    const uint32_t cw = far_at<uint32_t>(v, kUnrankGolayWt, d.golay + divide(divide(r >> sign_bits, d.perm_b, d.inv_b, rank_b), d.perm_a, d.inv_a, rank_a));
    // signs of the support in order: the free ones, then the one that makes sum |x| / 4 + the number of negative support
    // coordinates even (an off-support sign does not matter: it changes the sum by a multiple of 8)
    uint32_t on = sigma >> nz_b, off = sigma & ((1u << nz_b) - 1u);
    on |= w ? (((d.flags >> 15) ^ (uint32_t)popcount32(on)) & 1u) << (w - 1u) : 0u;
    if (w == 0) {
        // all 24 values off the support: the first twelve one by one, the others from the list
        uint32_t T = d.perm_b, n = d.b;
        uint64_t words = 0;
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
        for (int i = 0; i < 12; i++) {
            const UnrankStep e = blob_at<UnrankStep>(v, kUnrankSteps, 24 - i);
            uint32_t sh = 0, s = portion(T, n & 255u, e);
            while (rank_b >= s && sh < 24u) {
                rank_b -= s;
                sh += 8;
                s = portion(T, (n >> sh) & 255u, e);
            }
            n -= 1u << sh;
            T = s;
            words |= (uint64_t)(sh >> 3) << (4 * i);
        }
        const uint32_t rest = v.tab_b[blob_at<uint32_t>(v, kUnrankRest12, ((n >> 8) & 15u) | ((n >> 16) & 3u) << 4 | ((n >> 24) & 1u) << 6) + rank_b];
        const uint32_t k[3] = {(uint32_t)words, (uint32_t)(words >> 32) | spread_pairs(rest) << 16, spread_pairs(rest >> 8)};
#pragma unroll
        for (int j = 0; j < 3; j++) {
            p.mag[j] = 2u * k[j];
            p.neg[j] = deal_signs(v, k[j], off);
        }
        return;
    }
    if (w == 24) {
        const uint64_t a = far_at<uint64_t>(v, kUnrankSupport24, d.a + rank_a);
#pragma unroll
        for (int j = 0; j < 3; j++) {
            p.mag[j] = 2u * spread_pairs((uint32_t)(a >> (16 * j))) + 0x11111111u;
            p.neg[j] = spread8(on >> (8 * j));
        }
        return;
    }
    // the two sequences, a nibble a value: k in bits 0, 1, the sign in bit 2
    uint64_t in, out;
    {
        const uint32_t a = far_at<uint32_t>(v, kUnrankSupport, d.a + rank_a);
        const uint32_t lo = spread_pairs(a) | spread8(on) << 2, hi = spread_pairs(a >> 16) | spread8(on >> 8) << 2;
        in = (uint64_t)hi << 32 | lo;
        const uint32_t b = v.tab_b[d.b + rank_b];
        const uint32_t blo = spread_pairs(b), bhi = spread_pairs(b >> 16);
        const uint32_t slo = deal_signs(v, blo, off), shi = deal_signs(v, bhi, off);
        out = (uint64_t)(bhi | shi << 2) << 32 | (blo | slo << 2);
    }
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const uint32_t mask = (cw >> (8 * j)) & 255u, n = (uint32_t)popcount32(mask);
        const uint32_t m = to_places(v, mask, join((uint32_t)in, (uint32_t)out, 4u * n));
        in >>= 4u * n;
        out >>= 32u - 4u * n;
        p.neg[j] = (m >> 2) & 0x11111111u;
        p.mag[j] = 2u * (m & 0x33333333u) + spread8(mask);
    }
}

// codes u of eight coordinates from their magnitudes and signs
LLVQ_HD uint32_t point_codes(const Point &p, int w, bool odd) {
    return ((p.mag[w] | 0x88888888u) ^ (p.neg[w] * 15u)) + (odd ? 0u : p.neg[w]);
}

}  // namespace llvq
