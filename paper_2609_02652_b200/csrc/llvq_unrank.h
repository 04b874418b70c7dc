// Tables with which an index of the ball becomes coordinates by look-ups and short multiplications instead of
// one 64-bit division a coordinate and candidate (llvq_unrank.cuh reads them).
//
// An ordering of a multiset is ranked lexicographically.  Inside the ball there are few multisets: writing an odd
// magnitude as 1 + 2j, sum x^2 <= 192 leaves sum j(j+1)/2 <= 21 over the 24 coordinates, 225 multisets in all; the
// even type splits into the support (magnitudes 2 + 4k, a few k > 0) and the rest (4k).  So the orderings of what is
// left after the first coordinates can be listed: 64 952 of eight odd magnitudes, 6511 of a support, 288 000 of
// the rest of 8, 12 or 16 coordinates.  A thread reads its entries at random: the small tables are in one
// blob that a CTA copies to shared memory (a gather from there takes three or four wavefronts a warp, one from global
// memory thirty-two).
#pragma once
#include <cstdint>
#include <vector>

#include "llvq_tables.h"

namespace llvq {

// One class, as the un-ranking reads it.  32 bytes.
struct UnrankDesc {
    uint32_t flags;       // even: w << 1 | sign_bits << 6 | nz_b << 11 | repair << 15 | shell << 16 | window << 20; odd: 1 | the multiset's number << 1 | shell, window
    // even type only
    uint32_t perm_a;      // orderings of the support
    uint32_t perm_b;      // orderings off the support
    float inv_a, inv_b;   // 1 / perm_a, 1 / perm_b
    uint32_t a;           // first entry of the support's orderings
    uint32_t b;           // w = 8, 12, 16: first entry in tab_b; w = 0: copies of 0, 4, 8, 12 a byte each
    uint32_t golay;       // first entry of weight w in the code sorted by weight
};
static_assert(sizeof(UnrankDesc) == 32, "UnrankDesc layout");

// The same for the expander, in shared memory, a table a part: 32-byte records would have every lane's word in one of four banks,
// and its 16 bytes in one of four places.
struct alignas(16) UnrankPerms {
    uint32_t perm_a, perm_b;
    float inv_a, inv_b;
};
struct alignas(8) UnrankFirsts {
    uint32_t a_golay, b;  // a | golay << 16
};

// Division by a number of coordinates left: odd part's inverse modulo 2^32, and the power of two.
struct UnrankStep {
    uint32_t inverse, shift;
};

// Two odd magnitudes at a time: with L coordinates left that have T orderings, T n / (L (L - 1)) begin with a given pair of
// values, n the ways to draw the pair.  So the rank times L (L - 1) / T is a position among the L (L - 1) draws in order, and
// the table `pairs` tells for every multiset and position, in its low word, the first rank that begins with the pair drawn there; in
// its high word the multiset left (8 bits), the pair (8) and, as 5 bits of exponent and 11 of mantissa, the ratio for the multiset
// left (the last step: where its orderings begin in tail8).  The ratio is read with the other fields below its mantissa and is the
// least such number that is not below the ratio times kRatioExcess: the position that comes of it in f32 is the one wanted or the
// next (the roundings of product and factors are below 2^-22 of it, the excess below 2^-10, and the position below 2^9).
constexpr double kRatioExcess = 1.0 + 1.0 / (1 << 20);
constexpr uint32_t kRatioBase = 104u << 23;                            // of the least exponent: ratios from 2^-23 to 2^9
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
constexpr int kUnrankFlags = kUnrankBase + kUnrankClasses * 8;        // uint32[304]: UnrankDesc::flags
constexpr int kUnrankPerms = kUnrankFlags + kUnrankClasses * 4;       // UnrankPerms[304]
constexpr int kUnrankFirsts = kUnrankPerms + kUnrankClasses * 16;     // UnrankFirsts[304]
constexpr int kUnrankMerge = kUnrankFirsts + kUnrankClasses * 8;      // uint32[256]: byte selectors that take nibbles to the places of a byte mask and the others
constexpr int kUnrankSteps = kUnrankMerge + 256 * 4;                  // UnrankStep[32], by the number of coordinates left
constexpr int kUnrankRatio = kUnrankSteps + 32 * 8;                   // float[256]: 24 * 23 / orderings of a multiset
constexpr int kUnrankWindow = kUnrankRatio + 256 * 4;                 // uint32[kGuideSlots / 32]: bit = a slot with a class that is not kWindowAlways
constexpr int kUnrankGuide = kUnrankWindow + kGuideSlots / 8;         // uint16[kGuideSlots + 8]: first class of a slot
constexpr int kUnrankGolayMsg = kUnrankGuide + (kGuideSlots + 8) * 2; // uint32[128]: codewords of the messages k and, from 64 on, 64 k, k < 64
constexpr int kUnrankRest12 = kUnrankGolayMsg + 128 * 4;              // uint32[128]: first entry in tab_b of 12 off-support values
constexpr int kUnrankSharedBytes = kUnrankRest12 + 128 * 4;           // what follows stays in global memory
constexpr int kUnrankSupport = kUnrankSharedBytes;                    // uint32[kSupports]: 8, 12 or 16 support values' k, two bits each
constexpr int kSupports = 4192;
constexpr int kUnrankSupport24 = kUnrankSupport + kSupports * 4;      // uint64[kSupports24]: 24 of them
constexpr int kSupports24 = 2352;
constexpr int kUnrankGolayWt = kUnrankSupport24 + kSupports24 * 8;
constexpr int kUnrankDescs = kUnrankGolayWt + 4096 * 4;               // UnrankDesc[304]
constexpr int kUnrankBlobBytes = kUnrankDescs + kUnrankClasses * 32;
static_assert(kUnrankFlags % 16 == 0 && kUnrankPerms % 16 == 0 && kUnrankFirsts % 16 == 0 && kUnrankMerge % 16 == 0 && kUnrankSteps % 16 == 0 && kUnrankRatio % 16 == 0 &&
              kUnrankWindow % 16 == 0 && kUnrankGuide % 16 == 0 && kUnrankGolayMsg % 16 == 0 && kUnrankRest12 % 16 == 0 && kUnrankSharedBytes % 16 == 0 && kUnrankSupport24 % 16 == 0 &&
              kUnrankGolayWt % 16 == 0 && kUnrankDescs % 16 == 0 && kUnrankBlobBytes % 16 == 0, "alignment of the blob's parts");

struct UnrankTables {
    std::vector<uint8_t> blob;       // kUnrankBlobBytes
    std::vector<uint64_t> pairs;     // first rank | multiset left << 32 | pair << 40 (a nibble a value) | ratio or first entry in tail8 << 48
    std::vector<uint32_t> tail8;     // eight magnitudes' j, a nibble each, first coordinate lowest
    std::vector<uint32_t> tab_b;     // 8, 12 or 16 off-support values' k, two bits each
};

// From the class list and Golay code of build_tables.  Returns false if a class does not fit the tables.
bool build_unrank_tables(const HostTables &t, UnrankTables &u);

}  // namespace llvq
