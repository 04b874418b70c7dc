#include "llvq_unrank.h"

#include <array>
#include <cstring>
#include <map>

namespace llvq {
namespace {

// Appends every ordering of the `left` values of the multiset `cnt` (values 0..N-1), lexicographically, BITS bits a value.
template <int N, int BITS, typename T>
__attribute__((noinline)) void list_orderings(int *cnt, int left, int at, uint64_t word, std::vector<T> &out) {
    if (cnt[0] == left) { out.push_back((T)word); return; }         // zeros to the end
    for (int v = 0; v < N; v++) {
        if (cnt[v] == 0) continue;
        const uint64_t with = word | (uint64_t)v << (BITS * at);
        if (left == 1) { out.push_back((T)with); return; }
        cnt[v]--;
        list_orderings<N, BITS>(cnt, left - 1, at + 1, with, out);
        cnt[v]++;
    }
}

// Window of the 10-byte layout (codes u = 8 + floor(x / 2)): a block lacks one if two codes are more than seven apart,
// or a code is below 3 or above 13.
int window_of(const ClassDesc &d) {
    int lo[24], hi[24], n = 0;                           // codes of the negative and of the positive coordinate
    for (int v = 0; v < (d.odd ? 7 : 8); v++)
        for (int j = 0; j < d.cnt[v]; j++) {
            const int a = d.odd ? 1 + 2 * v : (v < 4 ? 2 + 4 * v : 4 * (v - 4));
            lo[n] = d.odd ? 7 - v : 8 - a / 2;
            hi[n] = 8 + a / 2;
            n++;
        }
    bool can = false, must = false;
    for (int i = 0; i < n; i++) {
        const bool bad_hi = hi[i] > 13, bad_lo = lo[i] < 3;
        can |= bad_hi || bad_lo;
        must |= bad_hi && bad_lo;
        for (int j = 0; j < n; j++) can |= i != j && hi[i] - lo[j] > 7;
    }
    return must ? kWindowNever : (can ? kWindowDepends : kWindowAlways);
}

template <typename T>
T *part(std::vector<uint8_t> &blob, int offset) { return reinterpret_cast<T *>(blob.data() + offset); }

}  // namespace

bool build_unrank_tables(const HostTables &t, UnrankTables &u) {
    u.blob.assign(kUnrankBlobBytes, 0);
    u.pairs.clear(); u.tail8.clear(); u.tab_b.clear();
    u.tail8.reserve(1 << 16); u.tab_b.reserve(300000);
    if (t.num_classes > kUnrankClasses - 2) return false;

    UnrankStep *steps = part<UnrankStep>(u.blob, kUnrankSteps);
    for (uint32_t n = 1; n < 32; n++) {
        steps[n].shift = (uint32_t)__builtin_ctz(n);
        const uint32_t odd = n >> steps[n].shift;
        uint32_t x = odd;                                // correct to 3 bits, doubled by each Newton step
        for (int i = 0; i < 4; i++) x *= 2u - odd * x;
        steps[n].inverse = x;
    }

    // ---- the multisets of odd magnitudes 1 + 2j, by their copies of j = 1..6 (sum j (j + 1) / 2 <= 21, at most 24 of them)
    std::map<std::array<int, 7>, int> set_of;            // key: copies of j = 1..6, [0] unused
    std::vector<std::array<int, 7>> sets;
    {
        static const int cost[7] = {0, 1, 3, 6, 10, 15, 21};
        std::array<int, 7> c{};
        for (c[6] = 0; c[6] <= 1; c[6]++)
        for (c[5] = 0; c[5] <= 1; c[5]++)
        for (c[4] = 0; c[4] <= 2; c[4]++)
        for (c[3] = 0; c[3] <= 3; c[3]++)
        for (c[2] = 0; c[2] <= 7; c[2]++)
        for (c[1] = 0; c[1] <= 21; c[1]++) {
            int sum = 0;
            for (int v = 1; v < 7; v++) sum += c[v] * cost[v];
            if (sum > 21) continue;
            set_of[c] = (int)sets.size();
            sets.push_back(c);
        }
        if ((int)sets.size() != kOddSets) return false;
    }
    auto copies_in = [](const std::array<int, 7> &c) { int n = 0; for (int v = 1; v < 7; v++) n += c[v]; return n; };
    // the multiset with one copy of v less (itself for v = 0: the copies of 0 are what is left)
    std::vector<std::array<int, 7>> less(sets.size());
    for (int k = 0; k < kOddSets; k++)
        for (int v = 0; v < 7; v++) {
            std::array<int, 7> c = sets[k];
            less[k][v] = v == 0 ? k : (c[v] ? (c[v]--, set_of[c]) : -1);
        }
    // every ordering of eight
    std::vector<uint32_t> tail_first(sets.size(), 0);
    for (int k = 0; k < kOddSets; k++) {
        const int n = copies_in(sets[k]);
        if (n > 8) continue;
        int c[7];
        for (int v = 1; v < 7; v++) c[v] = sets[k][v];
        c[0] = 8 - n;
        if (u.tail8.size() > 0xffff) return false;
        tail_first[k] = (uint32_t)u.tail8.size();
        list_orderings<7, 4>(c, 8, 0, 0, u.tail8);
    }
    // the draws of two from L
    // L! / (the copies' factorials): L over the copies of each value in turn, whole numbers all along
    auto orderings_of = [&](int k, int L) {
        uint64_t n = 1;
        for (int v = 1, left = L; v < 7; v++)
            for (int j = 1; j <= sets[k][v]; j++) n = n * (uint64_t)left-- / (uint64_t)j;
        return n;
    };
    auto ratio_bits = [&](int k, int L) {                // as a float's bits
        const float f = (float)(L * (L - 1) / (double)orderings_of(k, L) * kRatioExcess);
        uint32_t bits;
        std::memcpy(&bits, &f, 4);
        return bits;
    };
    uint32_t *first_ratio = part<uint32_t>(u.blob, kUnrankRatio);
    size_t entries = 0;
    for (int i = 0; i < kPairSteps; i++) entries += (size_t)kOddSets * (24 - 2 * i) * (23 - 2 * i);
    u.pairs.reserve(entries);
    for (int i = 0; i < kPairSteps; i++) {
        const int L = 24 - 2 * i, draws = L * (L - 1);
        const size_t first = u.pairs.size();
        u.pairs.resize(first + (size_t)kOddSets * draws, 0);
        for (int k = 0; k < kOddSets; k++) {
            const std::array<int, 7> &c = sets[k];
            const int n = copies_in(c);
            if (n > L) continue;
            uint64_t *entry = u.pairs.data() + first + (size_t)k * draws;
            const uint64_t orderings = orderings_of(k, L);
            if (orderings >= 0x80000000ull) return false;
            if (i == 0) first_ratio[k] = ratio_bits(k, L);
            int at = 0;
            for (int va = 0; va < 7; va++)
                for (int vb = 0; vb < 7; vb++) {
                    const int na = va ? c[va] : L - n, nb = (vb ? c[vb] : L - n) - (va == vb);
                    if (na < 1 || nb < 1) continue;
                    const int left = less[less[k][va]][vb];
                    uint32_t high = (uint32_t)left | (uint32_t)(va | vb << 4) << 8;
                    if (i == kPairSteps - 1) {
                        high |= tail_first[left] << 16;
                    } else {
                        const uint32_t wanted = ratio_bits(left, L - 2), below = high >> 4;
                        uint32_t bits = (wanted & ~0xfffu) | below;
                        if (bits < wanted) bits += 0x1000u;
                        if (bits - kRatioBase >= 1u << 28) return false;
                        high |= (bits - kRatioBase - below) << 4;
                    }
                    const uint64_t e = orderings * (uint64_t)at / (uint64_t)draws | (uint64_t)high << 32;
                    for (int j = 0; j < na * nb; j++) entry[at + j] = e;
                    at += na * nb;
                }
            if (at != draws) return false;
        }
    }

    // ---- supports of 8, 12, 16, 24 coordinates: (w - n1 - n2, n1, n2) copies of k = 0, 1, 2 with 8 n1 + 24 n2 <= 48 - w
    std::map<int, uint32_t> first_a, first_b;
    static const int weights[4] = {8, 12, 16, 24};
    std::vector<uint32_t> support;
    std::vector<uint64_t> support24;
    for (int w : weights)
        for (int n2 = 0; 24 * n2 <= 48 - w; n2++)
            for (int n1 = 0; 8 * n1 + 24 * n2 <= 48 - w; n1++) {
                int c[3] = {w - n1 - n2, n1, n2};
                first_a[w << 16 | n1 << 8 | n2] = (uint32_t)(w < 24 ? support.size() : support24.size());
                if (w < 24) list_orderings<3, 2>(c, w, 0, 0, support); else list_orderings<3, 2>(c, w, 0, 0, support24);
            }
    if (support.size() > kSupports || support24.size() > kSupports24) return false;
    std::memcpy(u.blob.data() + kUnrankSupport, support.data(), support.size() * 4);
    std::memcpy(u.blob.data() + kUnrankSupport24, support24.data(), support24.size() * 8);
    // ---- off-support values of 8, 12, 16 coordinates: n1, n2, n3 copies of k = 1, 2, 3 (and zeros) with
    // n1 + 4 n2 + 9 n3 <= 8 (w = 16), 12 (the last twelve coordinates of w = 0; w = 12 needs 9), 10 (w = 8)
    uint32_t *rest12 = part<uint32_t>(u.blob, kUnrankRest12);
    static const int lengths[3] = {8, 12, 16}, room[3] = {8, 12, 10};
    for (int l = 0; l < 3; l++)
        for (int n3 = 0; n3 <= 1; n3++)
            for (int n2 = 0; n2 <= 3; n2++)
                for (int n1 = 0; n1 <= 12; n1++) {
                    if (n1 + 4 * n2 + 9 * n3 > room[l] || n1 + n2 + n3 > lengths[l]) continue;
                    int c[4] = {lengths[l] - n1 - n2 - n3, n1, n2, n3};
                    first_b[lengths[l] << 16 | n1 << 8 | n2 << 4 | n3] = (uint32_t)u.tab_b.size();
                    if (lengths[l] == 12) rest12[n1 | n2 << 4 | n3 << 6] = (uint32_t)u.tab_b.size();
                    list_orderings<4, 2>(c, lengths[l], 0, 0, u.tab_b);
                }

    // ---- classes
    uint64_t *base = part<uint64_t>(u.blob, kUnrankBase);
    UnrankDesc *desc = part<UnrankDesc>(u.blob, kUnrankDescs);
    for (int c = 0; c < kUnrankClasses; c++) base[c] = c <= t.num_classes ? t.base[(size_t)c] : ~0ull;
    for (int c = 0; c < t.num_classes; c++) {
        const ClassDesc &d = t.desc[(size_t)c];
        UnrankDesc &e = desc[c];
        if (d.perm_a >= 0x80000000ull || d.perm_b > 0x1000000ull) return false;
        e.flags = (uint32_t)d.shell << 16 | (uint32_t)window_of(d) << 20;
        if (d.odd) {
            std::array<int, 7> c{};
            for (int v = 1; v < 7; v++) c[v] = d.cnt[v];
            const auto k = set_of.find(c);
            if (k == set_of.end()) return false;
            e.flags |= 1u | (uint32_t)k->second << 1;
            continue;
        }
        e.flags |= (uint32_t)d.w << 1 | (uint32_t)d.sign_bits << 6 | (uint32_t)d.nz_b << 11;
        e.perm_a = (uint32_t)d.perm_a;
        e.perm_b = (uint32_t)d.perm_b;
        e.inv_a = 1.0f / (float)d.perm_a;
        e.inv_b = 1.0f / (float)d.perm_b;
        e.golay = (uint32_t)t.weight_offset[d.w];
        int half_sum = 0;                                // sum |x| / 2
        for (int k = 0; k < 4; k++) half_sum += d.cnt[k] * (1 + 2 * k) + d.cnt[4 + k] * 2 * k;
        if (d.w > 0) {
            if (half_sum & 1) return false;
            e.flags |= (uint32_t)((half_sum >> 1) & 1) << 15;
            const auto a = first_a.find(d.w << 16 | d.cnt[1] << 8 | d.cnt[2]);
            if (a == first_a.end() || d.cnt[3]) return false;
            e.a = a->second;
        }
        if (d.w == 0) {
            e.b = (uint32_t)d.cnt[4] | (uint32_t)d.cnt[5] << 8 | (uint32_t)d.cnt[6] << 16 | (uint32_t)d.cnt[7] << 24;
        } else if (d.w < 24) {
            const auto b = first_b.find((24 - d.w) << 16 | d.cnt[5] << 8 | d.cnt[6] << 4 | d.cnt[7]);
            if (b == first_b.end()) return false;
            e.b = b->second;
        }
    }
    uint32_t *flags = part<uint32_t>(u.blob, kUnrankFlags);
    UnrankPerms *perms = part<UnrankPerms>(u.blob, kUnrankPerms);
    UnrankFirsts *firsts = part<UnrankFirsts>(u.blob, kUnrankFirsts);
    for (int c = 0; c < t.num_classes; c++) {
        const UnrankDesc &e = desc[c];
        if (e.a >= 0x10000u || e.golay >= 0x10000u) return false;
        flags[c] = e.flags;
        perms[c] = {e.perm_a, e.perm_b, e.inv_a, e.inv_b};
        firsts[c] = {e.a | e.golay << 16, e.b};
    }
    // ---- guide: class of the smallest index of every slot (a slot's indices share exponent and leading mantissa bits
    // of their value rounded to float; rounding is monotonic, so slots are ranges of indices)
    {
        uint16_t *guide = part<uint16_t>(u.blob, kUnrankGuide);
        auto slot_of = [](uint64_t idx) {
            const float f = (float)idx;
            uint32_t bits;
            std::memcpy(&bits, &f, 4);
            const int s = (int)(bits >> kGuideShift) - kGuideFirst;
            return s < 0 ? 0 : s;
        };
        // guide[s] = last class c whose first index lies in a slot before s, or is the slot's first index: the largest c with
        // slot_of(base[c]) < s is a lower bound that holds for every index of slot s
        for (int s = 0, c = 0; s < kGuideSlots + 8; s++) {
            while (c + 1 < t.num_classes && slot_of(t.base[(size_t)c + 1]) < s) c++;
            guide[s] = (uint16_t)c;
        }
        uint32_t *window = part<uint32_t>(u.blob, kUnrankWindow);
        for (int s = 0; s < kGuideSlots; s++)
            for (int c = guide[s]; c <= guide[s + 1]; c++)
                if (desc[c].flags >> 20 != kWindowAlways) window[s >> 5] |= 1u << (s & 31);
    }
    uint32_t *message = part<uint32_t>(u.blob, kUnrankGolayMsg);
    for (int k = 0; k < 64; k++) { message[k] = t.golay_by_message[k]; message[64 + k] = t.golay_by_message[64 * k]; }
    std::memcpy(u.blob.data() + kUnrankGolayWt, t.golay_by_weight.data(), 4096 * 4);

    // ---- eight nibbles, as many as a byte mask has bits for its places in order and then the others for the others: where
    // the bytes of the even places come from, and those of the odd places (nibble r is byte r / 2 of the even or the odd nibbles)
    uint32_t *merge = part<uint32_t>(u.blob, kUnrankMerge);
    for (int mask = 0; mask < 256; mask++) {
        uint32_t in = 0, out = (uint32_t)__builtin_popcount((unsigned)mask);
        for (int i = 0; i < 8; i++) {
            const uint32_t r = (mask >> i & 1) ? in++ : out++;
            merge[mask] |= ((r >> 1) | (r & 1u) << 2) << (4 * (i >> 1) + 16 * (i & 1));
        }
    }
    return true;
}

}  // namespace llvq
