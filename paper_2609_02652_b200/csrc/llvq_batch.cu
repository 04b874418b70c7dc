// The matvec for three, four, seven or eight activation vectors at once (llvq_gemv_batch): one pass over the 14-byte records, the decode of a
// tile and its block constants shared by the vectors.  Order of work, ring and accumulators are those of the kernel for one
// vector (llvq_gemv.cu), and so is the value of every row, bit for bit; the contraction is another.
//
// Arithmetic.  2 X_i (X the fixed-point activation, |X_i| < 2^29) is split in two, 2 X_i = L_i + 65536 H_i with
// -32896 <= L_i < 32640.  An FP16 activation has eleven significant bits, so X_i has, and both halves are FP16
// numbers exactly: a vector needs two columns of the contraction where 8-bit limbs need four, mma.sync m16n8k16
// f16 x f16 -> f32 serves four vectors, and an accumulator is the integer that limbs are recombined to - nothing is recombined or
// converted.  A code is taken as u 2^-18: its four bits moved to bits 6..9 of an FP16 word are that number, a subnormal one, which the
// instruction takes exactly.  So
//     2^-18 e = sum x_i L_i / 2^19 = sum (u_i 2^-18) L_i + (parity - 16) / 2^19 sum L_i,
// and one multiply-add a half and block adds the offset, one more applies the scale.  All of it is exact up to there: in units of
// 2^-18 the partial sums are whole numbers below 2^24 (|L_i| <= 32896, |H_i| <= 2^14), and e is a whole number below 2^23.
// One octave breaks the rule on L: 2 X = 32656, 32688, 32720 or 32752 (eleven bits and the sign) leave L = 2 X - 65536, which has
// twelve.  Such an activation is kept as L' = 2 X, H' = 0 - no other L is that large - and a CTA that meets one takes tiles
// through a second build of their code, which counts L' back: the contraction of the marks [L' >= 32640] takes 65536 times itself from L
// and adds itself to H.
//
// Bound: instruction issue (four vectors on 8192 x 8192: 466 warp instructions a tile with the launch's start, issue slots 59 % busy; eight: 649
// and 50 %, three warps a scheduler), and on small launches the preparation of x (4096 x 4096: issue slots 48 and 37 % busy, barriers and reads of
// global memory the longest stalls).  Against the 8-bit limbs two vectors at a time that this replaces, us a launch in a chain: see
// launch_gemv (llvq_gemv.cu).
#include <type_traits>

#include "llvq_gemv.cuh"

namespace llvq {
namespace {

// x in shared memory, a record a block and set of four vectors.  Column 2v + h of the contraction is half h (L, H) of vector v.
// Chunk c (0..5) of a column holds coordinates 4c, 4c+2, 4c+1, 4c+3, the order in which a payload byte pair is split; chunk 6 zeros.
// Chunk c of column n lies at 224 (n >> 2) + 32 c + 8 (n & 3): a half-warp's 64-bit reads are 128 consecutive bytes.  At 448,
// each vector's sum of 2 X in two parts (convert_third).
constexpr float kCodeUnit = 1.f / (1 << 18);      // what a code's bits count as FP16
constexpr int kSetBytes = kBatchSetBytes, kHalfBytes = 224, kSumsAt = 448;

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(0.f));
}
__device__ __forceinline__ void mma_f16_add(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}
// two floats in a register pair: L in the low half, H in the high
__device__ __forceinline__ uint64_t pair(float lo, float hi) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float2 halves(uint64_t v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint2 lds64_at(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(a), "n"(OFF));
    return v;
}

// What the decode needs in registers.  Left shifts are multiplications (by factors the compiler cannot see, or they would become shifts
// again): the logic unit takes two cycles an instruction, as the multiplier does, and has more to do.
struct Factors { uint32_t by4, by8, by16, by64; };
__device__ __forceinline__ Factors factors() {
    Factors f;
    asm volatile("mov.u32 %0, 4;\n\tmov.u32 %1, 16;\n\tmov.u32 %2, 64;\n\tmov.u32 %3, 8;" : "=r"(f.by4), "=r"(f.by16), "=r"(f.by64), "=r"(f.by8));
    return f;
}
// The A operand of a half-step (16 rows x two block slots).  Positions 0..15, 16..31, 32..47 of the half-step are an
// operand each; of the middle one the first two lanes of a quad hold slot 0's last eight coordinates and the other two slot 1's
// first eight.  k[s][e] = {2^18 gain / (4 sqrt m), (parity - 16) / 2^19} of slot s, row g + 8e.
struct Half {
    uint32_t first[4], middle[4], last[4];
    float2 k[2][2];
};
__device__ __forceinline__ Half decode_half16(uint32_t wa, uint32_t wb, uint32_t wc, uint32_t hw0, uint32_t hw1, uint32_t tab, const Factors &f) {
    auto code = [](uint32_t w) { return w & 0x03c003c0u; };
    Half h;
    // low nibbles of bytes 0 and 2, of bytes 1 and 3, then the high nibbles
    const uint32_t sa = wa >> 6, sb = wb >> 6, sc = wc >> 6;
    h.first[0] = code(wa * f.by64); h.first[1] = code(wb * f.by64); h.first[2] = code(sa * f.by16); h.first[3] = code(sb * f.by16);
    h.middle[0] = code(wa * f.by4); h.middle[1] = code(wb * f.by4); h.middle[2] = code(sa); h.middle[3] = code(sb);
    h.last[0] = code(wc * f.by64); h.last[1] = code(wc * f.by4); h.last[2] = code(sc * f.by16); h.last[3] = code(sc);
    // the headers of rows g (low half) and g + 8 (high half), eight bytes an entry; `tab` is 8 KiB-aligned
    h.k[0][0] = lds_f2(and_or(hw0 * f.by8, 0x1ff8u, tab));
    h.k[0][1] = lds_f2(and_or(hw0 >> 13, 0x1ff8u, tab));
    h.k[1][0] = lds_f2(and_or(hw1 * f.by8, 0x1ff8u, tab));
    h.k[1][1] = lds_f2(and_or(hw1 >> 13, 0x1ff8u, tab));
    return h;
}
// This lane's addresses in the x records of a block: its chunk t (and, 64 bytes on, chunk 2 + t, slot 1's last); the middle
// operand's chunk for slot 0 (chunk 4 + t, or zeros) and for slot 1 (zeros, or chunk t - 2); its vector's sums.
struct XAddr { uint32_t chunk, middle0, middle1, sums; };
__device__ __forceinline__ XAddr x_addr(int lane, uint32_t rec) {
    const int g = lane >> 2, t = lane & 3;
    const uint32_t column = rec + kHalfBytes * (g >> 2) + 8 * (g & 3);
    XAddr a;
    a.chunk = column + 32 * t;
    a.middle0 = column + 32 * (t < 2 ? 4 + t : 6);
    a.middle1 = column + 32 * (t < 2 ? 6 : t - 2);
    a.sums = rec + kSumsAt + 8 * t;
    return a;
}
// The B operand of a step (two block slots) for one set of vectors, and the slots' sums of this lane's vector
struct StepB {
    uint2 first, middle0, middle1, last;
    float2 sum0, sum1;
};
// OFF0, OFF1: slot 0's and slot 1's block
template <int OFF0, int OFF1>
__device__ __forceinline__ StepB load_b(const XAddr &a) {
    StepB b;
    b.first = lds64_at<OFF0>(a.chunk);
    b.middle0 = lds64_at<OFF0>(a.middle0);
    b.middle1 = lds64_at<OFF1>(a.middle1);
    b.last = lds64_at<OFF1 + 64>(a.chunk);
    const uint2 s0 = lds64_at<OFF0>(a.sums), s1 = lds64_at<OFF1>(a.sums);
    b.sum0 = make_float2(__uint_as_float(s0.x), __uint_as_float(s0.y));
    b.sum1 = make_float2(__uint_as_float(s1.x), __uint_as_float(s1.y));
    return b;
}
// WIDE: some L may be kept as L' (marks: 1 where it is).
__device__ __forceinline__ uint2 marks(uint2 b) {
    auto of = [](uint32_t w) {
        const __half2 m = __hge2(*reinterpret_cast<const __half2 *>(&w), __half2half2(__ushort_as_half(0x77f8)));      // 32640
        return *reinterpret_cast<const uint32_t *>(&m);
    };
    return make_uint2(of(b.x), of(b.y));
}
__device__ __forceinline__ void count_back(float (&d)[4], const float (&m)[4]) {
    d[0] = fmaf(m[0], -65536.f, d[0]); d[1] += m[0];
    d[2] = fmaf(m[2], -65536.f, d[2]); d[3] += m[2];
}
// One half-step of one set: adds to s0 (slot 0) and s1 (slot 1) the scaled sums {L, H} of rows g and g + 8 and this lane's vector, each
// rounded where the kernel for one vector rounds it.  FIRST: they are written, not added to.
template <bool FIRST, bool WIDE>
__device__ __forceinline__ void contract(const Half &h, const StepB &b, float2 (&s0)[2], float2 (&s1)[2]) {
    float d[4], f[4];
    mma_f16(d, h.first, b.first);
    mma_f16(f, h.last, b.last);
    mma_f16_add(d, h.middle, b.middle0);
    mma_f16_add(f, h.middle, b.middle1);
    if (WIDE) {
        float m[4];
        mma_f16(m, h.first, marks(b.first));
        mma_f16_add(m, h.middle, marks(b.middle0));
        count_back(d, m);
        mma_f16(m, h.last, marks(b.last));
        mma_f16_add(m, h.middle, marks(b.middle1));
        count_back(f, m);
    }
#pragma unroll
    for (int e = 0; e < 2; e++) {
        const float2 &k0 = h.k[0][e], &k1 = h.k[1][e];
        const float l0 = fmaf(k0.y, b.sum0.x, d[2 * e]), h0 = fmaf(k0.y, b.sum0.y, d[2 * e + 1]);
        const float l1 = fmaf(k1.y, b.sum1.x, f[2 * e]), h1 = fmaf(k1.y, b.sum1.y, f[2 * e + 1]);
        // FIRST: rounded products, which no sum below may take into a multiply-add
        s0[e] = FIRST ? make_float2(__fmul_rn(l0, k0.x), __fmul_rn(h0, k0.x)) : make_float2(fmaf(l0, k0.x, s0[e].x), fmaf(h0, k0.x, s0[e].y));
        s1[e] = FIRST ? make_float2(__fmul_rn(l1, k1.x), __fmul_rn(h1, k1.x)) : make_float2(fmaf(l1, k1.x, s1[e].x), fmaf(h1, k1.x, s1[e].y));
    }
}
// the unit's sum of a row from its two slots' shares, as quad_sum of llvq_gemv.cu adds them
__device__ __forceinline__ float row_sum(float2 s0, float2 s1) { return fmaf(s0.y + s1.y, 65536.f, s0.x + s1.x); }

// x (FP16, eight coordinates: a third of a block) -> its two chunks of the record, the first of them at `at`.  Returns the third's share of the block's
// activation sum, {sum L, sum H} but for a unit between the two.  2 rint(x scale) and the nearest multiple of 65536 come from additions of
// 1.5 * 2^23: x scale is a whole number of eleven significant bits, which such an addition leaves as it is, or below 2^11.  H is
// floor((z + 32896) / 65536) of the even z = 2 X, the nearest whole number to (z + 129) / 65536, which is never halfway between two.
// `wide` is set if an L had to be kept as L'.
__device__ __forceinline__ float2 convert_third(uint4 v, uint32_t at, float scale, bool finite, uint32_t *wide) {
    constexpr float kRound = 12582912.f;
    if (!finite) v = make_uint4(0u, 0u, 0u, 0u);
    const uint32_t hv[4] = {v.x, v.y, v.z, v.w};
    float x[8];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&hv[i]));
        x[2 * i] = f.x; x[2 * i + 1] = f.y;
    }
    uint32_t lo[4], hi[4];                                         // coordinates 0, 2 and 1, 3 of either chunk
    uint64_t exact[4], sum_lo = 0, sum_hi = 0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int c = 4 * (i >> 1) + (i & 1);
        const uint64_t z = fma2(fma2(pair(x[c], x[c + 2]), pair(scale, scale), pair(kRound, kRound)), pair(2.f, 2.f), pair(-2.f * kRound, -2.f * kRound));
        const uint64_t y = fma2(z, pair(1.f / 65536.f, 1.f / 65536.f), pair(129.f / 65536.f, 129.f / 65536.f));
        const uint64_t h = add2(add2(y, pair(kRound, kRound)), pair(-kRound, -kRound)), l = fma2(h, pair(-65536.f, -65536.f), z);
        sum_lo = i ? add2(sum_lo, l) : l;
        sum_hi = i ? add2(sum_hi, h) : h;
        exact[i] = l;
        const float2 fl = halves(l), fh = halves(h);
        const __half2 l2 = __floats2half2_rn(fl.x, fl.y), h2 = __floats2half2_rn(fh.x, fh.y);
        lo[i] = *reinterpret_cast<const uint32_t *>(&l2);
        hi[i] = *reinterpret_cast<const uint32_t *>(&h2);
    }
    auto as_half2 = [](uint32_t w) { return *reinterpret_cast<const __half2 *>(&w); };
    const __half2 least = __hmin2(__hmin2(as_half2(lo[0]), as_half2(lo[1])), __hmin2(as_half2(lo[2]), as_half2(lo[3])));
    if (__hle(__hmin(__low2half(least), __high2half(least)), __ushort_as_half(0xf800))) {          // an L of -32768 or less, seldom
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float2 l = halves(exact[i]), r = __half22float2(as_half2(lo[i]));
            const uint32_t keep = (r.x != l.x ? 0u : 0xffffu) | (r.y != l.y ? 0u : 0xffff0000u);
            const __half2 kept = __floats2half2_rn(l.x + 65536.f, l.y + 65536.f);
            lo[i] = (lo[i] & keep) | (*reinterpret_cast<const uint32_t *>(&kept) & ~keep);
            hi[i] &= keep;                                         // H is 1 there, H' 0
            if (~keep) *wide = 1u;
        }
    }
#pragma unroll
    for (int c = 0; c < 2; c++)
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at + 32 * c), "r"(lo[2 * c]), "r"(lo[2 * c + 1]), "r"(hi[2 * c]), "r"(hi[2 * c + 1]) : "memory");
    const float2 sl = halves(sum_lo), sh = halves(sum_hi);
    // an odd sum of H passes a unit on to the sum of L, as in the kernels for pairs and for one vector, whose records hold the halves of both
    // as whole numbers
    float sum_l = sl.x + sl.y, sum_h = sh.x + sh.y;
    if (__float_as_uint(sum_h + kRound) & 1u) {
        sum_l += 65536.f;
        sum_h -= 1.f;
    }
    return make_float2(sum_l, sum_h);
}

// SETS = 1: three or four vectors; 2: seven or eight.  The launch is one matrix (p.prob[0]).
template <int SETS>
__global__ void __launch_bounds__(32 * batch_warps(SETS), 1) gemv_batch_kernel(const __grid_constant__ GemvParams p) {
    constexpr int kWarps = batch_warps(SETS), kThreads = 32 * kWarps, kXBlock = SETS * kSetBytes;
    extern __shared__ __align__(128) unsigned char smem[];
    // shared memory: ring | block constants (1024, from an 8 KiB boundary of the shared window) | x records | barriers |
    // the row groups the CTA's share is cut at | maxima
    const uint32_t ring = smem_addr(smem), tab_pad = (0u - (ring + kWarps * kSlots * kTileBytes)) & 8191u, tab = ring + kWarps * kSlots * kTileBytes + tab_pad;
    float2 *tab_at = reinterpret_cast<float2 *>(smem + kWarps * kSlots * kTileBytes + tab_pad);
    const uint32_t xrec = tab + 8192, bars = xrec + (p.xblocks * kXBlock + 127) / 128 * 128;
    Cut *cut_at = reinterpret_cast<Cut *>(smem + (bars - ring) + kWarps * kSlots * 8);
    uint32_t *most_at = reinterpret_cast<uint32_t *>(cut_at + 1);  // largest |x| of every vector, as FP16 bits; then whether an L is kept as L'
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t my_ring = ring + warp * kSlots * kTileBytes, my_bar = bars + 8 * warp * kSlots;
    const GemvProblemDev &pr = p.prob[0];

    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < kSlots; s++) mbar_init(my_bar + 8 * s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid <= LLVQ_MAX_BATCH) most_at[tid] = 0u;
    __syncwarp();

    // This warp's units [u0, u0 + n_units) of the CTA's share, and the first one's place.  A run - a warp's units of one row group - ends
    // with a hand-over to the row accumulators.  Where the units are few, the warps' ranges do not cross row groups if there are warps
    // enough for that with as many units each, or one more: every warp then has one run at most, and the CTA adds up the runs of a row group
    // before it hands them over (`cut`), with an atomic a row and vector instead of one for every warp.  (Eight vectors on 4096 x 4096:
    // 450 000 atomics took 3000 cycles at the end of a launch.)
    const CtaShare me = p.cta[blockIdx.x];
    const int cta_n = p.cta[blockIdx.x + 1].first - me.first, blk_lo = me.blk_lo, blk_hi = me.blk_hi;
    int panel = fast_div(blk_lo / kTileCells, p.div_panel, p.panel), first = panel * p.panel, width = min(p.panel, p.units - first);
    const int panel_u0 = panel * (p.total_groups * p.panel);
    int u0 = me.first + (warp * cta_n + kWarps - 1) / kWarps, n_units = me.first + ((warp + 1) * cta_n + kWarps - 1) / kWarps - u0;
    bool cut = false;
    const int fewest = (cta_n + kWarps - 1) / kWarps;
    if (fewest <= width && cta_n > 0 && me.first + cta_n - panel_u0 <= p.total_groups * width) {
        const FastDiv by_width = panel == p.npanels - 1 ? p.div_last : p.div_panel;
        const int in_panel = me.first - panel_u0, group0 = fast_div(in_panel, by_width, width);
        const int head = min(width - (in_panel - width * group0), cta_n), rows = fast_div(cta_n - head, by_width, width), rest = cta_n - head - rows * width;
#pragma unroll 1
        for (int most = fewest; most <= fewest + 1 && !cut; most++) {
            Cut c;
            if (!cut_share(group0, head, rows, rest, width, most, kWarps, c)) continue;
            cut = true;
            int at;
            n_units = cut_range(c, cta_n, most, warp, at);
            u0 = me.first + at;
            if (tid == 0) *cut_at = c;
        }
    }
    int r = u0 - panel_u0;
    while (r >= p.total_groups * width && panel < p.npanels - 1) {
        r -= p.total_groups * width;
        panel++;
        first += p.panel;
        width = min(p.panel, p.units - first);
    }
    int group = panel == p.npanels - 1 ? fast_div(r, p.div_last, width) : fast_div(r, p.div_panel, width);
    int col = first + (r - group * width);

    // the issue side: next unit's first byte and size, units left in its stretch (a row group's columns of the panel), its row group and panel
    const uint32_t tail_bytes = (uint32_t)p.tail_cells * kCellBytes;
    const uint8_t *next = pr.layout + (size_t)(uint32_t)group * p.group_bytes + (size_t)col * kTileBytes;
    int issued = 0, i_left = first + width - col, i_group = group, i_first = first, i_width = width;
    int i_turn = (p.tail_cells != 0 && first + width == p.units) ? 1 : 0;      // 1 while the stretch ends with the leftover blocks (a unit of another size)
    uint32_t i_bytes = i_turn && i_left == 1 ? tail_bytes : (uint32_t)kTileBytes;
    const int my_issues = lane == 0 ? n_units : 0;
    auto issue = [&](uint32_t bar, uint32_t dst) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.lt.s32 p, %0, %1;\n\t"
            "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%2], %3;\n\t"
            "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%4], [%5], %3, [%2];\n\t}"
            ::"r"(issued), "r"(my_issues), "r"(bar), "r"(i_bytes), "r"(dst), "l"(next));
        issued++;
        next += kTileBytes;
        if (--i_left <= i_turn) {                      // once a stretch (twice where it ends with the leftover unit)
            if (i_left == 0) {
                if (++i_group == p.total_groups) {     // the panel is done: the next one's first stretch
                    i_group = 0;
                    i_first += p.panel;
                    i_width = min(p.panel, p.units - i_first);
                    i_turn = (p.tail_cells != 0 && i_first + i_width == p.units) ? 1 : 0;
                    next = pr.layout + (size_t)i_first * kTileBytes;
                } else {                               // the same columns of the next row group
                    next += (long long)p.group_bytes - (long long)i_width * kTileBytes;
                }
                i_left = i_width;
            }
            i_bytes = i_turn && i_left == 1 ? tail_bytes : (uint32_t)kTileBytes;
        }
        // no "memory" clobber: the slot's last reads feed `dst` through settled(), its next ones follow the next wait on `bar`
    };

    // the caller's constants and the library's tables: their loads go out now and are used after the wait
    constexpr int kClasses = (kClassSlots + kThreads - 1) / kThreads;
    float2 my_class[kClasses];
#pragma unroll
    for (int i = 0; i < kClasses; i++) {
        my_class[i] = make_float2(0.f, 0.f);
        if (kClassSlots % kThreads == 0 || tid + i * kThreads < kClassSlots)
            asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(my_class[i].x), "=f"(my_class[i].y) : "l"(p.cls_block + tid + i * kThreads));
    }
    if (n_units > 0 && lane == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(pr.row_scale + group * kRowsPerGroup));
    const int nx = p.nb * 3;
#pragma unroll
    for (int s = 0; s < kEarlySlots; s++) issue(my_bar + 8 * s, my_ring + s * kTileBytes);
    // (class | gain << 9) -> the block's constants
    auto build_table = [&]() {
#pragma unroll
        for (int i = 0; i < kClasses; i++) {
            const int c = tid + i * kThreads;
            if (kClassSlots % kThreads != 0 && c >= kClassSlots) break;
            const float offset = (float)__float_as_int(my_class[i].y) * (0.5f * kCodeUnit);
            tab_at[c] = make_float2(my_class[i].x * (pr.gain0 / kCodeUnit), offset);
            tab_at[512 + c] = make_float2(my_class[i].x * (pr.gain1 / kCodeUnit), offset);
        }
    };
    // The preparation of x: a vector is shared by `each` warps, ten blocks a warp at a time, three lanes a block.  More vectors than
    // half the warps go in two rounds.  Its code is met once by a launch and fetched as it goes: short loops beat unrolled ones (two blocks a lane
    // side by side and both rounds' loads together: 4096 x 4096, four vectors 8.2 -> 9.2 us).
    const int each = (p.batch > kWarps / 2 ? 2 * kWarps : kWarps) / (unsigned)p.batch, work = each * p.batch;
    const int blocks = blk_hi - blk_lo, my_block = lane / 3, third = lane - 3 * my_block;
    const uint32_t xs0 = xrec - (uint32_t)blk_lo * kXBlock;                   // address of block 0's record, were it there
    // in the shadow of the previous kernel: between the loads of x and their use, its wait for the class constants is a wait for x as well
    // (us, eight vectors: 1024 x 2560 8.83 -> 8.68, 34816 x 5120 54.0 -> 53.6)
    build_table();
    __syncthreads();                                   // the maxima are zero
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // a thread's pieces (eight coordinates): third `third` of blocks 10 (part + i each) + lane / 3 of the CTA's, two of them on their way at a time
    struct Share { int vector, part; const uint4 *x; };
    auto share_of = [&](int w) {
        Share q = {0, w, nullptr};
        while (q.part >= each) { q.part -= each; q.vector++; }
        q.x = reinterpret_cast<const uint4 *>(p.x) + (size_t)q.vector * nx;
        return q;
    };
    auto load_piece = [&](const Share &q, int block) { return lane < 30 && block < blocks ? __ldcg(q.x + 3 * (blk_lo + block) + third) : make_uint4(0u, 0u, 0u, 0u); };
    const Share first_share = share_of(warp);
    uint4 own0 = make_uint4(0u, 0u, 0u, 0u), own1 = own0;
    if (warp < work) {
        own0 = load_piece(first_share, 10 * first_share.part + my_block);
        own1 = load_piece(first_share, 10 * (first_share.part + each) + my_block);
    }
    // every vector's largest |x|
#pragma unroll 1
    for (int w = warp; w < work; w += kWarps) {
        const Share q = w == warp ? first_share : share_of(w);
        constexpr int kInFlight = 8;
        const int step = 32 * each;
        uint32_t m = 0;
        int e = 32 * q.part + lane;
        uint4 v[kInFlight];
        auto load = [&]() {
#pragma unroll
            for (int i = 0; i < kInFlight; i++) v[i] = e + i * step < nx ? __ldcg(q.x + e + i * step) : make_uint4(0u, 0u, 0u, 0u);
            e += kInFlight * step;
        };
        load();
        for (;;) {
#pragma unroll
            for (int i = 0; i < kInFlight; i++) m = max_abs_pair(max_abs_pair(max_abs_pair(max_abs_pair(m, v[i].x), v[i].y), v[i].z), v[i].w);
            if (e - lane >= nx) break;
            load();
        }
        const uint32_t most = __reduce_max_sync(0xffffffffu, max(m & 0xffffu, m >> 16));
        if (lane == 0) atomicMax(most_at + q.vector, most);
    }
    __syncthreads();                                   // publishes the maxima and the block constants
#pragma unroll
    for (int s = kEarlySlots; s < kSlots; s++) issue(my_bar + 8 * s, my_ring + s * kTileBytes);
#pragma unroll 1
    for (int w = warp; w < work; w += kWarps) {
        const Share q = w == warp ? first_share : share_of(w);
        const uint32_t most = most_at[q.vector];
        const float scale = pow2f(29 - x_exponent(most));
        int b = 10 * q.part + my_block;
        const uint32_t rec = xrec + (uint32_t)b * kXBlock + (SETS > 1 ? (q.vector >> 2) * kSetBytes : 0);
        uint32_t at = rec + ((q.vector >> 1) & 1) * kHalfBytes + (q.vector & 1) * 16 + 64 * third, sums = rec + kSumsAt + 8 * (q.vector & 3);
        if (w != warp) {
            own0 = load_piece(q, b);
            own1 = load_piece(q, b + 10 * each);
        }
#pragma unroll 1
        for (int b0 = 10 * q.part; b0 < blocks; b0 += 10 * each, b += 10 * each) {
            const bool here = lane < 30 && b < blocks;
            const uint4 now = own0;
            own0 = own1;
            own1 = load_piece(q, b + 20 * each);
            float2 s = make_float2(0.f, 0.f);
            if (here) s = convert_third(now, at, scale, most < kInfinity16, most_at + LLVQ_MAX_BATCH);
            const float lo1 = __shfl_down_sync(0xffffffffu, s.x, 1), lo2 = __shfl_down_sync(0xffffffffu, s.x, 2);
            const float hi1 = __shfl_down_sync(0xffffffffu, s.y, 1), hi2 = __shfl_down_sync(0xffffffffu, s.y, 2);
            if (here && third == 0) {
                asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(at + 192), "r"(0) : "memory");
                asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(sums), "f"(s.x + lo1 + lo2), "f"(s.y + hi1 + hi2) : "memory");
            }
            at += 10 * each * kXBlock;
            sums += 10 * each * kXBlock;
        }
    }
    __syncthreads();                                   // publishes the x records

    const Factors by = factors();
    const bool wide = most_at[LLVQ_MAX_BATCH] != 0u;
    // the last arrival of a row: `word` is the whole accumulator
    auto finish = [&](int v, int row, unsigned long long word, __half scale) {
        const float quantum = x_factor(most_at[v]) * pow2f(pr.qexp_base);
        pr.y[(size_t)v * p.y_stride + row] = (float)((long long)(word & kSumMask) - (long long)p.units * kUnitBias) * (quantum * __half2float(scale));
        p.accum[(size_t)v * ((size_t)p.total_groups * 32) + row] = 0ull;           // ready for the next launch on this context
    };
    constexpr int kCutStride = 40;                     // rows of a vector in a warp's sums: two vectors sixteen banks apart
    int n = 0;
    bool failed = false;
    uint32_t parity = 0, bar = my_bar, sbuf = my_ring;
    const uint32_t sbuf_end = my_ring + kSlots * kTileBytes;
    const float inv_q = pow2f(-29 - pr.qexp_base);
    const uint32_t lane16 = 16 * lane, lane4 = 4 * lane, head = 32 * (lane >> 2);
    auto next_slot = [&]() {
        bar += 8;
        sbuf += kTileBytes;
        const bool wrap = sbuf == sbuf_end;            // every slot completes once a round
        sbuf = wrap ? my_ring : sbuf;
        bar = wrap ? my_bar : bar;
        parity ^= wrap ? 1u : 0u;
    };
    // A run: this warp's units of one row group, summed in registers and handed over together.  sum[set][i] = row 8i + g of vector 4 set + t
    while (n < n_units) {
        const int run = min(first + width - col, n_units - n), run_tiles = max(0, min(run, p.tiles - col));
        // the row scales are needed by the arrival that finishes a row: on their way into L2
        if (n != 0 && lane == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(pr.row_scale + group * kRowsPerGroup));
        XAddr xa = x_addr(lane, xs0 + (uint32_t)col * (4 * kXBlock));
        long long sum[SETS][4];
#pragma unroll
        for (int j = 0; j < SETS; j++) sum[j][0] = sum[j][1] = sum[j][2] = sum[j][3] = 0;
        auto add_unit = [&](const float2 (&s0)[SETS][2][2], const float2 (&s1)[SETS][2][2]) {
#pragma unroll
            for (int j = 0; j < SETS; j++)
#pragma unroll
                for (int i = 0; i < 4; i++) sum[j][i] += __float2ll_rn(row_sum(s0[j][i >> 1][i & 1], s1[j][i >> 1][i & 1]) * inv_q);
        };
        auto tiles = [&](auto is_wide) {
            constexpr bool kWide = decltype(is_wide)::value;
#pragma unroll 1
            for (int u = 0; u < run_tiles; u++) {
                if (!mbar_try(bar, parity)) {
                    if (!mbar_wait(bar, parity)) { failed = true; break; }
                }
                const uint4 a0 = lds128(sbuf + lane16), a1 = lds128(sbuf + lane16 + 512), a2 = lds128(sbuf + lane16 + 1024);
                const uint4 h0 = lds128(sbuf + head + 1536), h1 = lds128(sbuf + head + 1552);      // slot 0's headers, slot 1's
                issue(bar, sbuf + (settled(a0.w, a1.w, a2.w) | settled(h0.w, h1.w, a0.x)));
                float2 s0[SETS][2][2], s1[SETS][2][2];                // slot 0 and slot 1: [set][m][e]
                {
                    StepB b[SETS];
                    b[0] = load_b<0, kXBlock>(xa);
                    if constexpr (SETS > 1) b[1] = load_b<kSetBytes, kXBlock + kSetBytes>(xa);
#pragma unroll
                    for (int m = 0; m < 2; m++) {
                        const Half h = m == 0 ? decode_half16(a0.x, a0.y, a0.z, h0.x, h1.x, tab, by) : decode_half16(a0.w, a1.x, a1.y, h0.y, h1.y, tab, by);
#pragma unroll
                        for (int j = 0; j < SETS; j++) contract<true, kWide>(h, b[j], s0[j][m], s1[j][m]);
                    }
                }
                {
                    StepB b[SETS];
                    b[0] = load_b<2 * kXBlock, 3 * kXBlock>(xa);
                    if constexpr (SETS > 1) b[1] = load_b<2 * kXBlock + kSetBytes, 3 * kXBlock + kSetBytes>(xa);
#pragma unroll
                    for (int m = 0; m < 2; m++) {
                        const Half h = m == 0 ? decode_half16(a1.z, a1.w, a2.x, h0.z, h1.z, tab, by) : decode_half16(a2.y, a2.z, a2.w, h0.w, h1.w, tab, by);
#pragma unroll
                        for (int j = 0; j < SETS; j++) contract<false, kWide>(h, b[j], s0[j][m], s1[j][m]);
                    }
                }
                add_unit(s0, s1);
                xa.chunk += 4 * kXBlock; xa.middle0 += 4 * kXBlock; xa.middle1 += 4 * kXBlock; xa.sums += 4 * kXBlock;
                next_slot();
            }
        };
        if (wide) tiles(std::true_type{}); else tiles(std::false_type{});
        if (failed) break;
        if (run_tiles < run) {
            // the run ends with the nb mod 4 last block columns of the row group: a pair, a single, or both
            if (!mbar_wait(bar, parity)) { failed = true; break; }
            const bool two = p.tail_cells >= 2, one = p.tail_cells & 1;
            uint32_t piece = sbuf, w[6] = {0, 0, 0, 0, 0, 0}, l[3] = {0, 0, 0};
            uint4 hp = make_uint4(0u, 0u, 0u, 0u);                 // slot 0's headers of m = 0, 1, then slot 1's
            uint2 hl = make_uint2(0u, 0u);                         // the headers of the two halves of the row group
            if (two) {
#pragma unroll
                for (int k = 0; k < 6; k++) w[k] = lds32(piece + 128 * k + lane4);
                hp = lds128(piece + 768 + 16 * (lane >> 2));
                piece += 2 * kCellBytes;
            }
            if (one) {
#pragma unroll
                for (int k = 0; k < 3; k++) l[k] = lds32(piece + 128 * k + lane4);
                hl = lds64(piece + 384 + 8 * (lane >> 2));
            }
            issue(bar, sbuf + (settled(w[0], w[1], w[2]) | settled(w[3], w[4], w[5]) | settled(hp.x, hp.w, l[0]) | settled(l[1], l[2], hl.y)));
            const XAddr xt = x_addr(lane, xs0 + (uint32_t)p.tiles * (4 * kXBlock)), xl = x_addr(lane, xs0 + (uint32_t)(p.nb - 1) * kXBlock);
            auto block = [&](const Half &h, const StepB &b, float2 (&s0)[2], float2 (&s1)[2]) {
                if (wide) contract<true, true>(h, b, s0, s1); else contract<true, false>(h, b, s0, s1);
            };
            float2 s0[SETS][2][2], s1[SETS][2][2];
#pragma unroll
            for (int j = 0; j < SETS; j++)
#pragma unroll
                for (int i = 0; i < 4; i++) s0[j][i >> 1][i & 1] = s1[j][i >> 1][i & 1] = make_float2(0.f, 0.f);
            if (two) {
                const Half h = decode_half16(w[0], w[1], w[2], hp.x, hp.z, tab, by), k = decode_half16(w[3], w[4], w[5], hp.y, hp.w, tab, by);
                StepB b = load_b<0, kXBlock>(xt);
                block(h, b, s0[0][0], s1[0][0]);
                block(k, b, s0[0][1], s1[0][1]);
                if constexpr (SETS > 1) {
                    b = load_b<kSetBytes, kXBlock + kSetBytes>(xt);
                    block(h, b, s0[1][0], s1[1][0]);
                    block(k, b, s0[1][1], s1[1][1]);
                }
            }
            if (one) {
                // the slots are the two halves of the row group, with the same block of x
                const Half h = decode_half16(l[0], l[1], l[2], hl.x, hl.y, tab, by);
                auto add_single = [&](const StepB &b, float2 (&a0)[2][2], float2 (&a1)[2][2]) {
                    float2 c0[2], c1[2];
                    block(h, b, c0, c1);
#pragma unroll
                    for (int e = 0; e < 2; e++) {
                        a0[0][e] = make_float2(a0[0][e].x + c0[e].x, a0[0][e].y + c0[e].y);
                        a1[1][e] = make_float2(a1[1][e].x + c1[e].x, a1[1][e].y + c1[e].y);
                    }
                };
                add_single(load_b<0, 0>(xl), s0[0], s1[0]);
                if constexpr (SETS > 1) add_single(load_b<kSetBytes, kSetBytes>(xl), s0[1], s1[1]);
            }
            add_unit(s0, s1);
            next_slot();
        }
        n += run;
        const int row0 = group * kRowsPerGroup + (lane >> 2), t = lane & 3;
        const unsigned long long counted = (unsigned long long)((long long)run * kUnitBias) + ((unsigned long long)run << kCountShift);
        if (cut) {
            // this warp's one run: its sums wait, in the place of its ring, for the CTA's sum of the row group (below)
            unsigned long long *mine = reinterpret_cast<unsigned long long *>(smem + warp * kSlots * kTileBytes);
            static_assert(4 * SETS * kCutStride * 8 <= kSlots * kTileBytes, "a warp's sums fit its ring");
#pragma unroll
            for (int j = 0; j < SETS; j++)
#pragma unroll
                for (int i = 0; i < 4; i++) mine[kCutStride * (4 * j + t) + 8 * i + (lane >> 2)] = (unsigned long long)sum[j][i] + counted;
        } else {
            // hand over: all the atomics are on their way before the first answer is looked at
            const size_t stride = (size_t)p.total_groups * 32;
            unsigned long long *slot = p.accum + row0;
            unsigned long long old[SETS][4];
            __half scale[4];
#pragma unroll
            for (int i = 0; i < 4; i++) scale[i] = row0 + 8 * i < pr.rows ? pr.row_scale[row0 + 8 * i] : __half();
#pragma unroll
            for (int j = 0; j < SETS; j++)
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (4 * j + t < p.batch && row0 + 8 * i < pr.rows) old[j][i] = atomicAdd(slot + (4 * j + t) * stride + 8 * i, (unsigned long long)sum[j][i] + counted);
#pragma unroll
            for (int j = 0; j < SETS; j++)
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (4 * j + t < p.batch && row0 + 8 * i < pr.rows && (int)(old[j][i] >> kCountShift) + run == p.units)
                        finish(4 * j + t, row0 + 8 * i, old[j][i] + ((unsigned long long)sum[j][i] + counted), scale[i]);
        }
        col += run;
        if (col == first + width) {
            if (++group == p.total_groups) {
                group = 0;
                first += p.panel;
                width = min(p.panel, p.units - first);
            }
            col = first;
        }
    }
    if (cut) {
        const bool lost = __syncthreads_or(failed);    // the warps' sums, and whether one has none
        // a thread a row, vector and row group at a time; all the atomics are on their way before the first answer is looked at
        constexpr int kMost = 4 * SETS;                // kWarps row groups at most, of 32 rows and 4 SETS vectors
        const Cut c = *cut_at;
        const int outputs = cut_outputs(c, p.batch, lost);
        unsigned long long old[kMost], word[kMost];
        __half scale[kMost];
        int units[kMost], row[kMost], v[kMost];
#pragma unroll
        for (int i = 0; i < kMost; i++) {
            const int o = tid + i * kThreads;
            row[i] = -1;
            if (o >= outputs) continue;
            const int k = o >> 5, s = cut_ratio(k, p.batch);
            v[i] = k - s * p.batch;
            const int r0 = (c.first_group + s) * kRowsPerGroup + (o & 31);
            const CutWarps of = cut_warps(c, s);
            units[i] = cut_units(c, s);
            if (r0 >= pr.rows) continue;
            row[i] = r0;
            scale[i] = pr.row_scale[r0];
            word[i] = 0ull;
            for (int w = of.first; w < of.end; w++) word[i] += *reinterpret_cast<const unsigned long long *>(smem + w * kSlots * kTileBytes + 8 * (kCutStride * v[i] + (o & 31)));
            old[i] = atomicAdd(p.accum + (size_t)v[i] * ((size_t)p.total_groups * 32) + r0, word[i]);
        }
#pragma unroll
        for (int i = 0; i < kMost; i++)
            if (row[i] >= 0 && (int)(old[i] >> kCountShift) + units[i] == p.units) finish(v[i], row[i], old[i] + word[i], scale[i]);
    }
    if (failed) {
        // a wait ran out: report it, then give the copies still in flight a bounded chance to land
        if (lane == 0) atomicExch(p.error, 1);
        for (int s = 0; s < kSlots && s < min(issued, n_units); s++) mbar_wait(my_bar + 8 * s, parity);
    }
}

}  // namespace

int batch_configure(int optin) {
    return allow_max_smem(gemv_batch_kernel<1>, optin) || allow_max_smem(gemv_batch_kernel<2>, optin) ? -1 : 0;
}

cudaError_t launch_batch(const GemvParams &p, const GemvLaunch &g, bool pdl, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.grid);
    cfg.blockDim = dim3(32 * batch_warps(batch_sets(p.batch)));
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, batch_sets(p.batch) == 1 ? gemv_batch_kernel<1> : gemv_batch_kernel<2>, p);
}

}  // namespace llvq
