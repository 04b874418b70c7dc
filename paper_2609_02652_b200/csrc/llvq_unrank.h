// Tables with which an index of the ball becomes coordinates by look-ups and short multiplications instead of
// one 64-bit division a coordinate and candidate (llvq_unrank.cuh reads them).
//
// An ordering of a multiset is ranked lexicographically.  Inside the ball there are few multisets: writing an odd
// magnitude as 1 + 2j, sum x^2 <= 192 leaves sum j(j+1)/2 <= 21 over the 24 coordinates, 225 multisets in all; the
// even type splits into the support (magnitudes 2 + 4k, a few k > 0) and the rest (4k).  So the orderings of what is
// left after the first coordinates can be listed: 64 952 of eight odd magnitudes, 6511 of a support, 291 000 of
// the rest of 8, 12 or 16 coordinates.  Those lists are the tables `tail8`, `tab_a` and `tab_b`; the small tables a
// thread reads at random are one blob that a CTA copies to shared memory.
#pragma once
#include <cstdint>
#include <vector>

#include "llvq_tables.h"

namespace llvq {

// One class, as the un-ranking reads it.  32 bytes.
struct UnrankDesc {
    uint32_t perm_a;      // odd: orderings of the 24 magnitudes; even: orderings of the support
    uint32_t perm_b;      // even: orderings off the support
    uint32_t a;           // even: first entry in tab_a; odd: copies of magnitude 1 | copies of magnitude 3 << 8
    uint32_t b;           // even, w = 8, 12, 16: first entry in tab_b; w = 0: copies of 0, 4, 8, 12 a byte each;
                          // odd: copies of magnitudes 5, 7, 9, 11, 13, a nibble each
    float inv_a, inv_b;   // 1 / perm_a, 1 / perm_b
    uint32_t flags;       // odd | w << 1 | sign_bits << 6 | nz_b << 11 | repair << 15 | shell << 16 | window << 20
    uint32_t golay;       // first entry of weight w in the code sorted by weight
};
static_assert(sizeof(UnrankDesc) == 32, "UnrankDesc layout");

// Division by a number of coordinates left: odd part's inverse modulo 2^32, and the power of two.
struct UnrankStep {
    uint32_t inverse, shift;
};

// flags >> 20: can a block of the class lack a window of the 10-byte layout, whatever its ordering and signs?
enum { kWindowAlways = 0, kWindowDepends = 1, kWindowNever = 2 };

// The shared-memory blob (byte offsets; every part 16-byte aligned).
constexpr int kUnrankClasses = 304;                                   // 301 and room for sentinels
constexpr int kGuideShift = 17;                                       // a class guide slot: exponent and 6 mantissa bits of (float)index
constexpr int kGuideFirst = (127 << (23 - kGuideShift));              // slot of index 1
constexpr int kGuideSlots = 48 * 64;                                  // indices below 2^48
constexpr int kUnrankBase = 0;                                        // uint64[304]: first index of a class, then ~0
constexpr int kUnrankDescs = kUnrankBase + kUnrankClasses * 8;        // UnrankDesc[304]
constexpr int kUnrankMerge = kUnrankDescs + kUnrankClasses * 32;      // uint4[256]: moves that spread nibbles to a byte mask's places
constexpr int kUnrankSteps = kUnrankMerge + 256 * 16;                 // UnrankStep[32], by the number of coordinates left
constexpr int kUnrankGuide = kUnrankSteps + 32 * 8;                   // uint16[kGuideSlots + 8]: first class of a slot
constexpr int kUnrankGolayMsg = kUnrankGuide + (kGuideSlots + 8) * 2; // uint32[4096]: codeword of a message
constexpr int kUnrankGolayWt = kUnrankGolayMsg + 4096 * 4;            // uint32[4096]: codewords by weight, then value
constexpr int kUnrankTailBase = kUnrankGolayWt + 4096 * 4;            // uint16[8192]: first entry in tail8 of the last eight odd magnitudes
constexpr int kUnrankDepositAt = kUnrankTailBase + 8192 * 2;          // uint16[256]: first entry in the deposit table of a byte mask
constexpr int kUnrankDeposit = kUnrankDepositAt + 256 * 2;            // uint32[6561 + 15]: bits dealt to a mask's places, a nibble each
constexpr int kUnrankRest12 = kUnrankDeposit + 6576 * 4;              // uint32[128]: first entry in tab_b of 12 off-support values
constexpr int kUnrankBlobBytes = kUnrankRest12 + 128 * 4;
static_assert(kUnrankDescs % 16 == 0 && kUnrankMerge % 16 == 0 && kUnrankGuide % 16 == 0 && kUnrankGolayMsg % 16 == 0 &&
              kUnrankTailBase % 16 == 0 && kUnrankDeposit % 16 == 0 && kUnrankBlobBytes % 16 == 0, "alignment of the blob's parts");

struct UnrankTables {
    std::vector<uint8_t> blob;       // kUnrankBlobBytes
    std::vector<uint32_t> tail8;     // eight magnitudes' j, a nibble each, first coordinate lowest
    std::vector<uint64_t> tab_a;     // w support values' k, two bits each
    std::vector<uint32_t> tab_b;     // 8, 12 or 16 off-support values' k, two bits each
};

// From the class list and Golay code of build_tables.  Returns false if a class does not fit the tables.
bool build_unrank_tables(const HostTables &t, UnrankTables &u);

}  // namespace llvq
