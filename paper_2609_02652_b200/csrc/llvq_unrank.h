// Tables with which an index of the ball becomes coordinates by look-ups and short multiplications instead of
// one 64-bit division a coordinate and candidate (llvq_unrank.cuh reads them).
//
// An ordering of a multiset is ranked lexicographically.  Inside the ball there are few multisets: writing an odd
// magnitude as 1 + 2j, sum x^2 <= 192 leaves sum j(j+1)/2 <= 21 over the 24 coordinates, 225 multisets in all; the
// even type splits into the support (magnitudes 2 + 4k, a few k > 0) and the rest (4k).  So the orderings of what is
// left after the first coordinates can be listed: 64 952 of eight odd magnitudes, 6511 of a support, 288 000 of
// the rest of 8, 12 or 16 coordinates.  A thread reads its entries at random: what fits is in one
// blob that a CTA copies to shared memory (a gather from there takes three or four wavefronts a warp, one from global
// memory thirty-two).
#pragma once
#include <cstdint>
#include <vector>

#include "llvq_tables.h"

namespace llvq {

// One class, as the un-ranking reads it.  32 bytes.
struct UnrankDesc {
    uint32_t perm_a;      // odd: orderings of the 24 magnitudes (the un-ranking has no use for it); even: orderings of the support
    uint32_t perm_b;      // even: orderings off the support
    uint32_t a;           // even: first entry of the support's orderings; odd: the multiset's number
    uint32_t b;           // even, w = 8, 12, 16: first entry in tab_b; w = 0: copies of 0, 4, 8, 12 a byte each
    float inv_a, inv_b;   // 1 / perm_a, 1 / perm_b
    uint32_t flags;       // odd | w << 1 | sign_bits << 6 | nz_b << 11 | repair << 15 | shell << 16 | window << 20
    uint32_t golay;       // first entry of weight w in the code sorted by weight
};
static_assert(sizeof(UnrankDesc) == 32, "UnrankDesc layout");

// Division by a number of coordinates left: odd part's inverse modulo 2^32, and the power of two.
struct UnrankStep {
    uint32_t inverse, shift;
};

// Two odd magnitudes at a time: with L coordinates left that have T orderings, T n / (L (L - 1)) begin with a given pair of
// values, n the ways to draw the pair.  So the rank times L (L - 1) / T is a position among the L (L - 1) draws in order, and
// the table `pairs` tells for every multiset and position the first rank that begins with the pair drawn there, the pair and the
// multiset left.  The multiset tells T, so the ratio is a table's, too, kept a little larger than it is: the position that comes of it
// in f32 is the one wanted or the next (the product's and the factors' roundings are below 2^-22 of it, and it is below 2^10).
struct PairStep {
    uint32_t first;            // of this L's entries in `pairs`
    uint32_t draws;            // L (L - 1)
};
constexpr double kRatioExcess = 1.0 + 1.0 / (1 << 20);
constexpr int kPairSteps = 8;                                         // L = 24, 22, .. 10
constexpr int kOddSets = 225;                                         // multisets of non-zero j with sum j (j + 1) / 2 <= 21

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
constexpr int kUnrankPairs = kUnrankSteps + 32 * 8;                   // PairStep[8]
constexpr int kUnrankRatios = kUnrankPairs + kPairSteps * 8;          // float[8][256]: draws / orderings of a step and multiset
constexpr int kUnrankWindow = kUnrankRatios + kPairSteps * 256 * 4;   // uint32[kGuideSlots / 32]: bit = a slot with a class that is not kWindowAlways
constexpr int kUnrankGuide = kUnrankWindow + kGuideSlots / 8;         // uint16[kGuideSlots + 8]: first class of a slot
constexpr int kUnrankGolayMsg = kUnrankGuide + (kGuideSlots + 8) * 2; // uint32[128]: codewords of the messages k and, from 64 on, 64 k, k < 64
constexpr int kUnrankTailBase = kUnrankGolayMsg + 128 * 4;            // uint16[256]: first entry in tail8 of a multiset of eight odd magnitudes
constexpr int kUnrankRest12 = kUnrankTailBase + 256 * 2;              // uint32[128]: first entry in tab_b of 12 off-support values
constexpr int kUnrankSharedBytes = kUnrankRest12 + 128 * 4;           // what follows stays in global memory
constexpr int kUnrankSupport = kUnrankSharedBytes;                    // uint32[kSupports]: 8, 12 or 16 support values' k, two bits each
constexpr int kSupports = 4192;
constexpr int kUnrankSupport24 = kUnrankSupport + kSupports * 4;      // uint64[kSupports24]: 24 of them
constexpr int kSupports24 = 2352;
constexpr int kUnrankGolayWt = kUnrankSupport24 + kSupports24 * 8;
constexpr int kUnrankBlobBytes = kUnrankGolayWt + 4096 * 4;
static_assert(kUnrankDescs % 16 == 0 && kUnrankPairs % 16 == 0 && kUnrankRatios % 16 == 0 && kUnrankWindow % 16 == 0 && kUnrankMerge % 16 == 0 && kUnrankGuide % 16 == 0 && kUnrankGolayMsg % 16 == 0 &&
              kUnrankTailBase % 16 == 0 && kUnrankSupport24 % 16 == 0 && kUnrankBlobBytes % 16 == 0, "alignment of the blob's parts");

struct UnrankTables {
    std::vector<uint8_t> blob;       // kUnrankBlobBytes
    std::vector<uint64_t> pairs;     // first rank | pair << 32 (a nibble a value) | multiset left << 40
    std::vector<uint32_t> tail8;     // eight magnitudes' j, a nibble each, first coordinate lowest
    std::vector<uint32_t> tab_b;     // 8, 12 or 16 off-support values' k, two bits each
};

// From the class list and Golay code of build_tables.  Returns false if a class does not fit the tables.
bool build_unrank_tables(const HostTables &t, UnrankTables &u);

}  // namespace llvq
