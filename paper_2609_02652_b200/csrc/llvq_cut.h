// How the warps of a CTA divide its share of a launch where they add their sums up before the hand-over (llvq_batch.cu).  Apart from
// the kernel so that the host can run it too.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define LLVQ_CUT_HD __host__ __device__ __forceinline__
#else
#define LLVQ_CUT_HD inline
#endif

namespace llvq {

// a / b for 0 <= a < 2^20 and 0 < b < 2^20: the half keeps the estimate off whole numbers by more than it is wrong
LLVQ_CUT_HD int cut_ratio(int a, int b) {
#ifdef __CUDA_ARCH__
    return (int)__fdividef((float)a + 0.5f, (float)b);
#else
    return (int)(((float)a + 0.5f) / (float)b);
#endif
}

// A share of units in ranges, a warp a range, none of which crosses a row group (`width` units): `groups` row groups from `first_group` on, of the first
// of which the share has `head` units, and `rest` of the last, if that is another and not whole (else 0).
struct alignas(16) Cut {
    int first_group, groups, head, rest;
    int in_head, in_row, in_rest, width;               // ranges of the first row group, of a whole one and of the last; a row group's units
};
// The warps whose sums are those of a row group of a cut share.
struct CutWarps {
    int first, end;
};

// Cuts a share that has `head` units in its first row group, then `rows` whole ones, then `rest` units, into ranges of `most` units.
// False if that takes more ranges than there are warps.
LLVQ_CUT_HD bool cut_share(int first_group, int head, int rows, int rest, int width, int most, int warps, Cut &c) {
#ifdef __CUDA_ARCH__
    const float inverse = __fdividef(1.f, (float)most);
#else
    const float inverse = 1.f / (float)most;
#endif
    auto ranges = [&](int n) { return (int)(((float)(n + most) - 0.5f) * inverse); };       // ranges of `most` units that n units make
    const int in_head = ranges(head), in_row = ranges(width), in_rest = ranges(rest);
    if (in_head + rows * in_row + in_rest > warps) return false;
    c = {first_group, 1 + rows + (rest > 0 ? 1 : 0), head, rest, in_head, in_row, in_rest, width};
    return true;
}
// the units [at, at + k) of the share of `n` that are `warp`'s; returns k
LLVQ_CUT_HD int cut_range(const Cut &c, int n, int most, int warp, int &at) {
    auto least = [](int a, int b) { return a < b ? a : b; };
    int begin, end;
    if (warp < c.in_head) {
        begin = warp * most;
        end = least(begin + most, c.head);
    } else {
        const int row = cut_ratio(warp - c.in_head, c.in_row), row_begin = c.head + row * c.width;
        begin = row_begin + (warp - c.in_head - row * c.in_row) * most;
        end = least(least(begin + most, row_begin + c.width), n);
    }
    at = least(begin, n);
    return end > begin ? end - begin : 0;
}
LLVQ_CUT_HD bool cut_ends_in(const Cut &c, int s) { return s == c.groups - 1 && c.rest > 0; }
// of the share's row group number `s`: the warps that hold its sums, and its units
LLVQ_CUT_HD CutWarps cut_warps(const Cut &c, int s) {
    const int first = s == 0 ? 0 : c.in_head + (s - 1) * c.in_row;
    return {first, first + (s == 0 ? c.in_head : (cut_ends_in(c, s) ? c.in_rest : c.in_row))};
}
LLVQ_CUT_HD int cut_units(const Cut &c, int s) { return s == 0 ? c.head : (cut_ends_in(c, s) ? c.rest : c.width); }
// The sums a CTA hands over: one a row of its row groups and vector, but none if a warp's wait ran out (`lost`).  Such a warp left no
// sums, and what lies in their place is a record.
LLVQ_CUT_HD int cut_outputs(const Cut &c, int batch, bool lost) { return lost ? 0 : c.groups * 32 * batch; }

}  // namespace llvq
